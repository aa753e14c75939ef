"""The evaluation's forms (GPU): with a parent's table per warp, per block, by (equation, child)
pairs, for two children and without a table, in FP32 and in FP64, against the oracle."""

import dataclasses
import functools

import numpy as np
import pytest

import oracle
from paper_1802_00330_gb300 import synth

pytestmark = pytest.mark.gpu


def _batched(n, seed):
    return synth.config_batched(1, seed=seed, n_range=(n, n))[0]


def _near_root(n, seed, half):
    s = synth.served_systems(1, seed=seed, n_range=(n, n))[0]
    root = np.array([float(v) for v in s.roots[0]]) + half / 8
    return dataclasses.replace(s, box_lo=root - half, box_hi=root + half)


def _more_equations(s, extra):
    """`s` with its first equations repeated (over-determined: no contraction)."""
    offs, rows = list(s.eq_offsets), []
    for i in range(extra):
        rows += list(s.terms_of(i % s.n_eqs))
        offs.append(offs[-1] + len(s.terms_of(i % s.n_eqs)))
    take = list(range(s.n_terms)) + rows
    return dataclasses.replace(s, n_eqs=s.n_eqs + extra, eq_offsets=np.array(offs, np.int32), coef_lo=s.coef_lo[take],
                               coef_hi=s.coef_hi[take], exps=s.exps[take])


def _all_variables(n):
    """One equation with a term in nine variables: no table."""
    exps = np.zeros((n + 2, n), np.uint8)
    exps[0, :9] = 1
    for j in range(n):
        exps[j + 1, j] = 2
    coef = np.array([0.25] + [1.0] * n + [-0.5 * n])
    return synth.PolySystem(n_vars=n, n_eqs=1, eq_offsets=np.array([0, n + 2], np.int32), coef_lo=coef.copy(),
                            coef_hi=coef.copy(), exps=exps, box_lo=np.full(n, -1.0), box_hi=np.full(n, 1.5), tol=0.5)


CASES = {
    "n1": (lambda: _batched(1, 7), {}),
    "n2": (synth.config_n2, {}),
    "n3": (lambda: _batched(3, 3000), {}),
    "n4": (lambda: _batched(4, 4000), {}),
    "n5": (lambda: _batched(5, 5001), {}),
    "n5_bisect": (lambda: _batched(5, 5003), {"split_mode": 1}),
    "n7_levels": (lambda: _batched(7, 7007), {"max_depth": 3}),
    "n8_levels": (lambda: _batched(8, 8001), {"max_depth": 2}),
    "n9_levels": (lambda: _near_root(9, 102, 0.5), {"max_depth": 2, "hs_enable": 0}),
    "n11_level": (lambda: _near_root(11, 6, 0.5), {"max_depth": 1}),
    "n5_17_equations": (lambda: _more_equations(_batched(5, 5001), 12), {"hs_enable": 0, "tol": 0.25}),
    "n9_no_table": (lambda: _all_variables(9), {"hs_enable": 0, "max_depth": 1}),
}


@functools.lru_cache(maxsize=1)
def _expected(name):
    make, options = CASES[name]
    return oracle.solve(make(), **options)


@pytest.mark.parametrize("prefilter", [True, False])
@pytest.mark.parametrize("name", CASES)
def test_evaluation_forms(name, prefilter):
    from paper_1802_00330_gb300 import _binding as B

    make, options = CASES[name]
    s = make()
    g = B.solve(s, prefilter_fp32=prefilter, **options)
    o = _expected(name)
    assert g["status"] == o["status"]
    for key in ("lo", "hi", "flags", "depth"):
        assert np.array_equal(g[key], o[key]), key
    st, ot = g["stats"], o["stats"]
    assert st["excluded_prefilter"] + st["excluded_eval"] == ot["excluded_eval"]
    for key in ("boxes", "hs_applied", "hs_empty", "split", "depth_boxes", "depth_kept"):
        assert np.array_equal(st[key], ot[key]), key
