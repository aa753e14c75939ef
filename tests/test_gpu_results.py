"""Results of a run on their way to the host (GPU): packed in one copy up to 16 MB, system by system above; both
return the same rows."""

import dataclasses

import numpy as np
import pytest

from paper_1802_00330_gb300 import synth

pytestmark = pytest.mark.gpu


def _wide(max_depth):
    s = synth.config_batched(1, seed=4000, n_range=(4, 4))[0]
    return dataclasses.replace(s, coef_lo=s.coef_lo - 0.25, coef_hi=s.coef_hi + 0.25, tol=0.0), max_depth


# boxes of 4 variables take 72 bytes each: one system's 2.0e5 (depth 7) are packed, two such systems' are not
@pytest.mark.parametrize("max_depth, rows, copies", [(2, 100, 1), (4, 1000, 3), (7, 200_000, 2)])
def test_one_system_and_several(max_depth, rows, copies):
    from paper_1802_00330_gb300 import _binding as B

    s, depth = _wide(max_depth)
    small = synth.config_n2()
    opts = {"max_depth": depth, "max_results": 1 << 18}
    one, many = B.Plan([s], opts=opts), B.Plan([s, small] * copies, opts=opts)
    try:
        one.run()
        a = one.result(0)
        assert len(a["flags"]) >= rows
        for _ in range(2):
            many.run()
            for k in list(range(0, 2 * copies, 2)) + [0]:
                b = many.result(k)
                assert a["status"] == b["status"]
                for key in ("lo", "hi", "flags", "depth"):
                    assert np.array_equal(a[key], b[key]), (k, key)
            assert len(many.result(1)["flags"]) == len(many.result(2 * copies - 1)["flags"])
        again = one.result(0)
        for key in ("lo", "hi", "flags", "depth"):
            assert np.array_equal(a[key], again[key]), key
    finally:
        one.close()
        many.close()
