"""The contraction's own FP64 division (GPU) against the oracle's, through the sweep that uses it:
one- and two-variable systems whose coefficients put quotients in every part of its range
(ordinary, exact, huge and tiny, subnormal operands that go to the library)."""

import numpy as np
import pytest

import oracle
from paper_1802_00330_gb300 import synth

pytestmark = pytest.mark.gpu

SCALES = {"one": 1.0, "third": 1.0 / 3.0, "large": 2.0 ** 400, "tiny": 2.0 ** -400, "subnormal": 2.0 ** -1030}


def _scaled(s, factors):
    """`s` with equation i multiplied by factors[i]."""
    f = np.concatenate([np.full(len(s.terms_of(i)), factors[i]) for i in range(s.n_eqs)])
    lo, hi = s.coef_lo * f, s.coef_hi * f
    return synth.PolySystem(n_vars=s.n_vars, n_eqs=s.n_eqs, eq_offsets=s.eq_offsets, coef_lo=np.minimum(lo, hi),
                            coef_hi=np.maximum(lo, hi), exps=s.exps, box_lo=s.box_lo, box_hi=s.box_hi, tol=s.tol)


@pytest.mark.parametrize("second", SCALES)
@pytest.mark.parametrize("first", SCALES)
def test_sweeps_with_scaled_equations(first, second):
    from paper_1802_00330_gb300 import _binding as B

    rng = np.random.default_rng(len(first) * 16 + len(second))
    for n in (1, 2):
        for k in range(8):
            s = synth.config_batched(1, seed=int(rng.integers(1 << 30)), n_range=(n, n))[0]
            s = _scaled(s, [SCALES[first], -SCALES[second]][:n])
            s.box_lo = s.box_lo - rng.uniform(0, 1, n)
            s.box_hi = s.box_hi + rng.uniform(0, 1, n)
            g, o = B.solve(s, max_depth=24), oracle.solve(s, max_depth=24)
            assert g["status"] == o["status"]
            for key in ("lo", "hi", "flags", "depth"):
                assert np.array_equal(g[key], o[key]), (n, k, key)
            for key in ("boxes", "hs_applied", "hs_empty", "hs_contracted", "hs_singular"):
                assert g["stats"][key] == o["stats"][key], (n, k, key)
