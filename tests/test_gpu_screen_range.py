"""The FP32 screen of the contraction (GPU) where single precision runs out of exponents: a system
scaled by powers of two has the same boxes, scaled, in FP64 (no operation of the sweep changes but
for its exponent), while in float its monomials, coefficients or values underflow.  The screen
may leave more boxes to FP64 there and must not settle one differently."""

import dataclasses

import numpy as np
import pytest

from paper_1802_00330_gb300 import synth

pytestmark = pytest.mark.gpu

FATES = ("boxes", "hs_applied", "hs_empty", "hs_contracted", "hs_singular", "accepted", "unsplittable", "split",
         "max_depth_seen", "excluded_centred", "gap_splits", "depth_boxes", "depth_kept", "depth_hs")
# A sweep is screened from one round of narrow chunks on: 8 boxes a block, blocks of 256 threads, 2048
# threads per SM.  A depth whose children fit one sweep of 2^22 is one sweep.
ROUND = 152 * 8 * 8


def screened(stats):
    """Whether some sweep had more boxes for the contraction than one round: those that entered
    it, or those that it kept (the centred form alone counts none that enter)."""
    most = np.maximum(stats["depth_hs"], stats["depth_kept"])
    return bool(np.any((most > ROUND) & (stats["depth_boxes"] <= 1 << 22)))


def scaled(s, x, f, width=0.0):
    """`s` in the variable 2^x y (its box and tol times 2^x) with its values times 2^f; `width`
    widens the coefficients (relative)."""
    k = s.exps.astype(np.int64).sum(axis=1)
    c = np.ldexp(1.0, f - x * k)
    lo, hi = s.coef_lo - width * np.abs(s.coef_lo), s.coef_hi + width * np.abs(s.coef_hi)
    return dataclasses.replace(s, coef_lo=lo * c, coef_hi=hi * c, box_lo=np.ldexp(s.box_lo, x), box_hi=np.ldexp(s.box_hi, x),
                               tol=float(np.ldexp(s.tol, x)), roots=[])


# (powers of two of the variables, of the values, factor of the exponents): monomials fall to 2^-144 beside
# coefficients of 2^92; the same with exponents of 5, 10, 15; the values themselves fall to 2^-100; coefficients of
# 2^-140 beside variables of 2^40
RANGES = {"small_variables": (-48, -52, 1), "high_powers": (-9, -40, 5), "small_values": (-20, -100, 1),
          "small_coefficients": (40, -20, 1)}
OPTIONS = {"default": {}, "krawczyk": {"krawczyk": True}, "centred": {"centred_form": True},
           "centred_alone": {"centred_form": True, "hs_min_depth": 9}}


@pytest.mark.parametrize("width", [0.0, 2.0 ** -20])
@pytest.mark.parametrize("option", OPTIONS)
@pytest.mark.parametrize("name", RANGES)
def test_scaled_system_has_the_scaled_boxes(name, option, width):
    from paper_1802_00330_gb300 import _binding as B

    x, f, raised = RANGES[name]
    base = dataclasses.replace(synth.config_batched(1, seed=5016, n_range=(5, 5))[0], tol=0.02)
    if raised > 1:
        base = dataclasses.replace(base, exps=base.exps * raised, box_lo=base.box_lo * 0.3125, box_hi=base.box_hi * 0.3125)
    kw = dict(OPTIONS[option], max_depth=8)
    a = B.solve(scaled(base, x, f, width), **kw)
    b = B.solve(scaled(base, 0, 0, width), prefilter_fp32=False, **kw)
    assert screened(a["stats"])
    assert a["status"] == b["status"]
    for key in ("lo", "hi"):
        assert np.array_equal(np.ldexp(a[key], -x), b[key]), key
    for key in ("flags", "depth"):
        assert np.array_equal(a[key], b[key]), key
    for key in FATES:
        assert np.array_equal(a["stats"][key], b["stats"][key]), key
