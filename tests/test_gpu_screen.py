"""The FP32 screen of the contraction (GPU): with it, boxes, flags, depths and every counter of
the fate of a box equal those of the FP64-only path, which has no screen."""

import dataclasses

import numpy as np
import pytest

from paper_1802_00330_gb300 import synth

pytestmark = pytest.mark.gpu

FATES = ("boxes", "hs_applied", "hs_empty", "hs_contracted", "hs_singular", "accepted", "unsplittable", "split",
         "max_depth_seen", "excluded_centred", "gap_splits", "depth_boxes", "depth_kept", "depth_hs")
# a sweep is screened when it has more boxes than one round of narrow chunks takes
NARROW = 152 * 2 * 8


def _batched(n, seed):
    return synth.config_batched(1, seed=seed, n_range=(n, n))[0]


def _near_root(n, seed, half):
    s = synth.served_systems(1, seed=seed, n_range=(n, n))[0]
    root = np.array([float(v) for v in s.roots[0]]) + half / 8
    return dataclasses.replace(s, box_lo=root - half, box_hi=root + half)


def _interval_coefficients(s, width):
    return dataclasses.replace(s, coef_lo=s.coef_lo - width, coef_hi=s.coef_hi + width)


CASES = {
    "n4": (lambda: _batched(4, 4000), {}),
    "n5": (lambda: _batched(5, 5006), {}),
    "n6": (synth.config_n6, {}),
    "n6_krawczyk": (synth.config_n6, {"krawczyk": True}),
    "n6_centred": (synth.config_n6, {"centred_form": True}),
    "n6_centred_alone": (synth.config_n6, {"centred_form": True, "hs_min_depth": 4}),
    "n6_iterated": (synth.config_n6, {"hs_iters": 3, "hs_min_depth": 2}),
    "n6_bisect": (synth.config_n6, {"split_mode": 1}),
    "n6_gap": (synth.config_n6, {"gap_split": True}),
    "n6_coarse": (synth.config_n6, {"tol": 0.3}),
    "n6_interval_coefficients": (lambda: _interval_coefficients(synth.config_n6(), 2.0 ** -12), {"max_depth": 7}),
    "n7": (lambda: _batched(7, 7003), {}),
    "n8": (lambda: _batched(8, 8002), {}),
    "n9": (lambda: _near_root(9, 102, 0.125), {}),
    "n10_centred": (lambda: _near_root(10, 102, 0.078125), {"centred_form": True}),
    "n12": (lambda: _near_root(12, 108, 0.03125), {}),
    "n13_one_level": (lambda: _near_root(13, 3, 0.5), {"max_depth": 1}),
    "n16_one_level": (lambda: _near_root(16, 5, 0.25), {"max_depth": 1}),
}


@pytest.mark.parametrize("name", CASES)
def test_screened_equals_fp64_only(name):
    from paper_1802_00330_gb300 import _binding as B

    make, options = CASES[name]
    s = make()
    a = B.solve(s, **options)
    b = B.solve(s, prefilter_fp32=False, **options)
    assert a["status"] == b["status"]
    assert int(np.max(a["stats"]["depth_hs"])) > NARROW or name in ("n4", "n6_centred_alone", "n10_centred")
    for key in ("lo", "hi", "flags", "depth"):
        assert np.array_equal(a[key], b[key]), key
    for key in FATES:
        assert np.array_equal(a["stats"][key], b["stats"][key]), key
