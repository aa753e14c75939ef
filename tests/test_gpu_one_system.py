"""Plans of one system (GPU): whatever the size of the system's table, a sweep pops its parents in the
commit of the sweep before it and has no kernel for that; results equal those of a plan of two."""

import dataclasses

import numpy as np
import pytest

from paper_1802_00330_gb300 import synth

pytestmark = pytest.mark.gpu


def _system(n):
    if n <= 8:
        return synth.config_batched(1, seed=n * 1000 + 5, n_range=(n, n))[0]
    s = synth.served_systems(1, seed=102, n_range=(n, n))[0]
    half = {9: 0.125, 11: 0.0625, 12: 0.03125, 14: 0.25}[n]
    root = np.array([float(v) for v in s.roots[0]]) + half / 8
    return dataclasses.replace(s, box_lo=root - half, box_hi=root + half)


@pytest.mark.parametrize("n, options", [(2, {}), (6, {}), (9, {}), (11, {"centred_form": True}), (12, {"max_depth": 3}),
                                        (14, {"max_depth": 1}), (11, {"split_mode": 1, "max_depth": 24})])
def test_pop_shares_the_commit(n, options):
    from paper_1802_00330_gb300 import _binding as B

    s = _system(n)
    opts = dict(options, max_results=1 << 18)
    one, two = B.Plan([s], opts=opts), B.Plan([s, synth.config_n2()], opts=opts)
    try:
        one.run()
        two.run()
        a, b = one.result(0), two.result(0)
        for key in ("lo", "hi", "flags", "depth"):
            assert np.array_equal(a[key], b[key]), key
        assert a["status"] == b["status"]
        for key in ("boxes", "hs_applied", "hs_empty", "hs_contracted", "accepted", "split", "depth_boxes"):
            assert np.array_equal(a["stats"][key], b["stats"][key]), key
        # a sweep: evaluation in FP32 and FP64, screen (from four variables on), two contractions, commit;
        # before the sweeps: initial boxes, first pop
        st = one.stats()
        assert st["launches"] == 2 + st["waves"] * (6 if n >= 4 else 5)
    finally:
        one.close()
        two.close()
