"""The FP32 screen of the contraction (GPU) in sweeps that are sure to be screened, for each of its kernels' shapes
(4, 8 and 16 lanes per box) with the sweep alone, the centred form before it, and the centred form
alone: boxes, flags, depths and every counter equal the FP64-only path's."""

import dataclasses

import numpy as np
import pytest

from paper_1802_00330_gb300 import synth

from test_gpu_screen_range import FATES, screened

pytestmark = pytest.mark.gpu


def _fat(n, seed, width):
    s = synth.config_batched(1, seed=seed, n_range=(n, n))[0]
    return dataclasses.replace(s, coef_lo=s.coef_lo - width, coef_hi=s.coef_hi + width, tol=0.02)


def _near_root(n, seed, half):
    s = synth.served_systems(1, seed=seed, n_range=(n, n))[0]
    root = np.array([float(v) for v in s.roots[0]]) + half / 8
    return dataclasses.replace(s, box_lo=root - half, box_hi=root + half, tol=1e-3)


SYSTEMS = {
    "n4": (lambda: _fat(4, 4013, 2.0 ** -5), 8),
    "n5": (lambda: _fat(5, 5018, 2.0 ** -5), 8),
    "n6": (lambda: _fat(6, 6017, 0.0), 8),
    "n9": (lambda: _near_root(9, 102, 0.125), 3),
    "n10": (lambda: _near_root(10, 102, 0.078125), 3),
    "n11": (lambda: _near_root(11, 5, 0.0625), 2),
}
OPTIONS = {
    "sweep": {},
    "krawczyk": {"krawczyk": True},
    "centred": {"centred_form": True, "hs_iters": 2},
    "centred_alone": {"centred_form": True, "hs_min_depth": 20},
}


# (too few boxes of n4 stay under the centred form alone for its sweeps to be wide)
CASES = [(n, o) for n in SYSTEMS for o in OPTIONS if (n, o) != ("n4", "centred_alone")]


@pytest.mark.parametrize("name, option", CASES)
def test_wide_sweeps_equal_fp64_only(name, option):
    from paper_1802_00330_gb300 import _binding as B

    make, depth = SYSTEMS[name]
    s = make()
    kw = dict(OPTIONS[option], max_depth=depth)
    a = B.solve(s, **kw)
    b = B.solve(s, prefilter_fp32=False, **kw)
    assert screened(a["stats"])
    assert a["status"] == b["status"]
    for key in ("lo", "hi", "flags", "depth"):
        assert np.array_equal(a[key], b[key]), key
    for key in FATES:
        assert np.array_equal(a["stats"][key], b["stats"][key]), key
