"""What is measured of this solver: its public calls over the range of problems that they serve.

A case names a recipe of this repository (its seeded system generators, or one of the paper's
printed systems), how many variables and systems it has, the call that takes it and the
options.  The seed varies the data and not the problem's kind: every coefficient is scaled by
1 + k / 4096, |k| <= 64, and the constant terms follow, so that the planted root stays exact.
Box counts of the recipes differ by about a factor of ten between two systems of one size.
"""

from __future__ import annotations

import dataclasses
import os

import numpy as np

from paper_1802_00330_gb300 import _binding as B
from paper_1802_00330_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# options by name: what a caller passes beside the system
OPTIONS = {
    "default": {},
    # FP64 alone: the form that the FP32 stage is checked against
    "fp64": {"prefilter_fp32": False},
    # the paper's other contraction and its second exclusion test (Section 2.3)
    "krawczyk": {"krawczyk": True},
    "centred": {"centred_form": True, "hs_iters": 2},
    # split rules: bisection of the widest side, with the two-box split at a gap
    "bisect": {"split_mode": 1, "gap_split": True},
}


def listed():
    return [
        # the smallest call: one textbook system from host arrays to host boxes (latency, launches)
        {"name": "call_n2", "call": "solve", "recipe": "circle_parabola", "n": 2, "system": 0, "count": 1, "options": "default"},
        # a small system by bisection: two children per box, many narrow sweeps
        {"name": "call_n5_bisect", "call": "solve", "recipe": "batched", "n": 5, "system": 5003, "count": 1, "options": "bisect"},
        # the seeded n = 6 system on a plan that the caller keeps
        {"name": "plan_n6", "call": "plan", "recipe": "n6", "n": 6, "system": 0, "count": 1, "options": "default"},
        # the same kind without the FP32 stage
        {"name": "plan_n6_fp64", "call": "plan", "recipe": "batched", "n": 6, "system": 6003, "count": 1, "options": "fp64"},
        # Krawczyk's contraction, n = 7
        {"name": "plan_n7_krawczyk", "call": "plan", "recipe": "batched", "n": 7, "system": 7005, "count": 1, "options": "krawczyk"},
        # an ordinary large single system
        {"name": "plan_n8", "call": "plan", "recipe": "batched", "n": 8, "system": 8005, "count": 1, "options": "default"},
        # one of the paper's printed systems, n = 9 (Section 4, Table 7)
        {"name": "call_n9_kinema", "call": "solve", "recipe": "kinema", "n": 9, "system": 0, "count": 1, "options": "default"},
        # a large system searched in a part of its box, with the centred form and repeated sweeps
        {"name": "part_n11_centred", "call": "plan", "recipe": "part", "n": 11, "system": 6, "count": 1, "options": "centred"},
        # many small systems in one call (host arrays in, host boxes out)
        {"name": "batch_small", "call": "batch", "recipe": "batched", "n": 5, "system": 11, "count": 96, "options": "default"},
        # the batching workload: n = 2..8 in one device run on a kept plan
        {"name": "batch_large", "call": "plan", "recipe": "batched", "n": 8, "system": 12, "count": 64, "options": "default"},
        # requests that arrive together at a server
        {"name": "served_burst", "call": "server", "recipe": "served", "n": 6, "system": 13, "count": 24, "options": "default"},
        # root isolation over a large box set: connected components and dyadic cells
        {"name": "roots_200k", "call": "roots", "recipe": "boxes", "n": 6, "system": 14, "count": 200_000, "options": "default"},
    ]


# seeds of the serving recipe whose part takes at most about half a second: the others' boxes go
# into the billions (the recipe's Jacobian may be nearly singular at the root)
PART_SYSTEMS = {
    9: (2, 3, 4, 5, 101, 102, 103, 104, 105, 106, 107, 108),
    10: (1, 3, 5, 101, 102, 104, 105, 108),
    11: (1, 2, 4, 5, 6, 102, 103, 104, 106, 108),
    12: (1, 2, 3, 4, 101, 103, 105, 106, 107, 108),
}


def draw(rng):
    case = {"system": rng.randrange(1, 1 << 20), "options": "default", "count": 1}
    kind = rng.choice(("solve", "plan", "plan", "part", "batch", "plans", "server", "roots"))
    if kind in ("solve", "plan"):
        option = rng.choice(("default", "default", "default", "fp64", "krawczyk", "centred", "bisect"))
        top = {"default": 8, "krawczyk": 8, "centred": 7, "fp64": 6, "bisect": 5}[option]
        case.update(call=kind, recipe="batched", n=rng.randint(2, top), options=option)
    elif kind == "part":
        n = rng.randint(9, 12)
        case.update(call="plan", recipe="part", n=n, system=rng.choice(PART_SYSTEMS[n]), options=rng.choice(("default", "centred")))
    elif kind == "batch":
        case.update(call="batch", recipe="batched", n=rng.randint(3, 6), count=int(8 * 32 ** rng.random()))
    elif kind == "plans":
        case.update(call="plan", recipe="batched", n=rng.randint(5, 8), count=rng.randint(8, 40))
    elif kind == "server":
        case.update(call="server", recipe="served", n=rng.randint(3, 6), count=rng.randint(5, 24))
    else:
        case.update(call="roots", recipe="boxes", n=rng.randint(2, 9), count=int(2000 * 100 ** rng.random()))
    return case


# ---- inputs --------------------------------------------------------------------------------
def _varied(s, rng):
    """`s` with every coefficient scaled by 1 + k / 4096 and its root kept exactly."""
    scale = 1.0 + rng.integers(-64, 65, size=s.n_terms) / 4096.0
    lo, hi = s.coef_lo * scale, s.coef_hi * scale
    if s.roots:
        point = np.array([float(v) for v in s.roots[0]])
        value = lo * np.prod(point[None, :] ** s.exps.astype(np.float64), axis=1)
        for i in range(s.n_eqs):
            t = [k for k in s.terms_of(i) if s.exps[k].any()]
            c = [k for k in s.terms_of(i) if not s.exps[k].any()]
            lo[c[0]] = hi[c[0]] = -float(np.sum(value[t]))
    return dataclasses.replace(s, coef_lo=lo, coef_hi=hi)


def _part(s, rng):
    """`s` on a part of its box: the neighbourhood that another method named, which holds
    the root off its centre."""
    root = np.array([float(v) for v in s.roots[0]])
    half = {9: 0.125, 10: 0.078125, 11: 0.0625, 12: 0.03125}[s.n_vars]
    centre = root + half * rng.integers(-32, 33, size=s.n_vars) / 64.0
    return dataclasses.replace(s, box_lo=np.maximum(s.box_lo, centre - half), box_hi=np.minimum(s.box_hi, centre + half))


def _systems(case, rng):
    n, count, system, recipe = case["n"], case["count"], case["system"], case["recipe"]
    if recipe == "circle_parabola":
        base = [synth.config_n2()]
    elif recipe == "n6":
        base = [synth.config_n6()]
    elif recipe == "kinema":
        base = [dataclasses.replace(synth.load_fixture(os.path.join(ROOT, "tests", "golden", "kinema.txt")), tol=1e-3)]
    elif recipe == "part":
        return [_part(_varied(s, rng), rng) for s in synth.served_systems(1, seed=system, n_range=(n, n))]
    elif recipe == "served":
        base = synth.served_systems(count, seed=system, n_range=(3, n))
    else:
        base = synth.config_batched(count, seed=system, n_range=(n if count == 1 else 2, n))
    return [_varied(s, rng) for s in base]


def _boxes(case, seed):
    """A box set as a solve to a coarse width leaves it: around each root a cluster of equal
    boxes, every one of which touches an earlier one, far from the other clusters; boxes in
    random order.  Returns (lo, hi, cluster of each box)."""
    rng = np.random.default_rng(seed)
    n, total = case["n"], case["count"]
    roots = max(2, total // 700)
    owner = np.sort(rng.integers(0, roots, size=total))
    start = np.searchsorted(owner, np.arange(roots))
    width = 2.0 ** -10
    # cluster centres on a coarse grid whose cells are wider than any cluster can grow
    cells = 1
    while cells ** min(n, 3) < roots:
        cells += 1
    index = rng.permutation(cells ** min(n, 3))[:roots]
    spot = np.zeros((roots, n))
    for j in range(min(n, 3)):
        spot[:, j] = (index // cells ** j % cells) * (2.0 / cells) - 1.0 + 1.0 / cells
    # box k of a cluster lies one step, along one coordinate, from one a few places before it;
    # clusters wander at most 0.2 of a cell (the walk is folded back)
    step = np.zeros((total, n), dtype=np.int64)
    step[np.arange(total), rng.integers(0, n, size=total)] = rng.choice((-1, 1), size=total)
    walk = np.cumsum(step, axis=0)
    walk -= walk[start[owner]]
    reach = max(2, int(0.2 / cells / width))
    walk = np.abs((walk + reach) % (4 * reach) - 2 * reach) - reach
    centre = spot[owner] + walk * width
    order = rng.permutation(total)
    return (centre - width / 2)[order], (centre + width / 2)[order], owner[order]


def prepare(case, seed):
    rng = np.random.default_rng([seed, 1802])
    options = OPTIONS[case["options"]]
    if case["call"] == "roots":
        lo, hi, _ = _boxes(case, seed)
        return {"call": "roots", "lo": lo, "hi": hi, "box": (np.full(case["n"], -2.0), np.full(case["n"], 2.0)), "level": 10}
    systems = _systems(case, rng)
    # places for the boxes of all results: about 2^n boxes stay around a root on the dyadic grid
    state = {"call": case["call"], "systems": systems, "options": options, "room": case["count"] * 16 << case["n"]}
    if case["call"] == "plan":
        # a plan of one system has the default sweep; the batching workload's has 2^24 children
        state["plan"] = B.Plan(systems, opts=dict(options), wave_children=(1 << 24) if case["count"] > 1 else 0)
    elif case["call"] == "server":
        # room for a request's breadth-first levels, as the serving workload configures it
        state["server"] = B.Server(max_slots=64, workspace_bytes=12 << 30, min_region_entries=1 << 20)
    return state


# ---- one pass --------------------------------------------------------------------------------
COUNTS = ("boxes", "hs_applied", "hs_empty", "hs_contracted", "hs_singular", "accepted", "unsplittable", "split",
          "max_depth_seen", "excluded_centred", "gap_splits")


def _rows(arrays, places):
    """The results' arrays one after the other, in front of zeros."""
    out = np.zeros(places, arrays[0].dtype)
    at = 0
    for a in arrays:
        out[at:at + a.size] = a.reshape(-1)
        at += a.size
    return out


def _outputs(state, results):
    """All boxes of all systems with their flags and depths, and the counts of each system."""
    room, n = state["room"], max(s.n_vars for s in state["systems"])
    counts = [[r["stats"][k] for k in COUNTS] + [r["stats"]["excluded_prefilter"] + r["stats"]["excluded_eval"]] for r in results]
    return {
        "status": np.array([r["status"] for r in results], np.int64),
        "rows": np.array([len(r["flags"]) for r in results], np.int64),
        "lo": _rows([r["lo"] for r in results], room * n),
        "hi": _rows([r["hi"] for r in results], room * n),
        "flags": _rows([r["flags"] for r in results], room),
        "depth": _rows([r["depth"] for r in results], room),
        "counts": np.array(counts, np.int64),
        "per_depth": np.concatenate([r["stats"][k] for r in results for k in ("depth_boxes", "depth_kept", "depth_hs")]),
    }


def run(state):
    call = state["call"]
    if call == "solve":
        return _outputs(state, [B.solve(state["systems"][0], **state["options"])])
    if call == "batch":
        return _outputs(state, B.solve_batch(state["systems"], **state["options"]))
    if call == "plan":
        state["plan"].run()
        return _outputs(state, [state["plan"].result(k) for k in range(len(state["systems"]))])
    if call == "server":
        tickets = [state["server"].submit(s, **state["options"]) for s in state["systems"]]
        return _outputs(state, [state["server"].wait(t) for t in tickets])
    count, labels, hull_lo, hull_hi = B.clusters_gpu(state["lo"], state["hi"])
    cells, groups = B.backtrack_gpu(state["lo"], state["hi"], *state["box"], state["level"], groups=True)
    return {"count": count, "labels": labels, "hull_lo": hull_lo, "hull_hi": hull_hi, "cells": cells, "groups": groups}


# ---- what a pass needs -------------------------------------------------------------------------
# boxes that a system of the recipes takes through the whole path, about (geometric means)
BATCHED_BOXES = {2: 2.5e2, 3: 1.2e3, 4: 1.0e4, 5: 1.3e5, 6: 1.8e6, 7: 1.3e7, 8: 7e7}
SERVED_BOXES = {3: 4e3, 4: 4e4, 5: 7e5, 6: 3.5e7}
OTHER_BOXES = {"circle_parabola": 85.0, "n6": 1.19e6, "kinema": 8.2e8, "part": 2e7}


def work(case):
    """Bytes: the inputs read and the boxes written once.  Operations: per box the natural
    form of as many equations as decide it (two on average), and for the one box in thirty
    that stays a Hansen-Sengupta sweep."""
    n, count, recipe = case["n"], case["count"], case["recipe"]
    if recipe == "boxes":
        # each box read for both results, a label and (per coordinate) one comparison and one
        # cell index written or made
        return {"bytes": float(count * (2 * 16 * n + 8)), "flops": float(count * 6 * n)}
    if recipe in OTHER_BOXES:
        boxes = {n: OTHER_BOXES[recipe]}
    else:
        table = SERVED_BOXES if recipe == "served" else BATCHED_BOXES
        low = n if count == 1 else min(table)
        boxes = {k: table[k] * count / (n - low + 1) for k in range(low, n + 1)}
    terms, flops, rows = 7, 0.0, 0.0
    for k, b in boxes.items():
        flops += b * 2 * terms * 6 + b / 30 * (6 * k ** 3 + 40 * k * k)
    rows = 30.0 * count
    return {"bytes": float(count * n * terms * (16 + n) + rows * (16 * n + 8)), "flops": flops}


def exact(case, seed):
    """Box ends come from directed roundings in one fixed order and have no value of their own
    beside the solver's; the clusters' hulls have one."""
    if case["call"] != "roots":
        return None
    lo, hi, owner = _boxes(case, seed)
    # clusters are numbered in the order of their first box
    _, first, inverse = np.unique(owner, return_index=True, return_inverse=True)
    rank = np.empty(len(first), np.int64)
    rank[np.argsort(first)] = np.arange(len(first))
    labels = rank[inverse]
    hull_lo, hull_hi = np.full((len(first), case["n"]), np.inf), np.full((len(first), case["n"]), -np.inf)
    np.minimum.at(hull_lo, labels, lo)
    np.maximum.at(hull_hi, labels, hi)
    return {"count": len(first), "labels": labels, "hull_lo": hull_lo, "hull_hi": hull_hi, "cells": None, "groups": None}
