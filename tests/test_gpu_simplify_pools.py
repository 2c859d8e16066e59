"""Simplification whose row pool runs full, from the first round on and in different rounds of a batch: its rows
are gathered into the other pool in the middle of the round, which then goes on.  MSC_FAULT=rows@n starts the
pools with room for n entries beyond the complex, so that they fill whatever headroom they are given otherwise."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from synth import fields
from tests.gpu_util import dims_of, gpu_field, msc, to_np

pytestmark = pytest.mark.gpu


def _simplify(f, threshold):
    m = msc()
    plan = m.Plan(dims_of(f))
    d = gpu_field(f)
    m.msc_compute(plan, d)
    m.msc_complex_graph_size(plan)
    before = m.msc_get_stats(plan)["n_launches"]
    r = m.msc_simplify(plan, d, threshold)
    launches = m.msc_get_stats(plan)["n_launches"] - before
    nodeptr, adj, mult = (to_np(r[k]) for k in ("nodeptr", "adj", "mult"))
    u = np.repeat(np.arange(len(nodeptr) - 1), np.diff(nodeptr))
    keep = u < adj
    return dict(r, alive=to_np(r["alive"]).astype(bool), log=to_np(r["log"]), longest=int(np.diff(nodeptr).max()),
                arcs=sorted(zip(u[keep].tolist(), adj[keep].tolist(), mult[keep].tolist()))), launches


# the first leaves rows longer than a warp
@pytest.mark.parametrize("shape,alpha,quantile,row", [((36, 44, 40), 2.0, 0.97, 33), ((33, 20, 65), 3.5, 0.9, 2)])
def test_full_pools(shape, alpha, quantile, row, monkeypatch):
    f = fields.grf(shape, alpha, seed=77)
    sk = oracle.skeleton(f)
    th = float(np.quantile(np.abs(sk["value"][sk["arc_u"]] - sk["value"][sk["arc_v"]]), quantile))
    want = oracle.simplify(sk, th, rounds=True)
    log = np.stack([want["upper"], want["lower"], want["round"]], 1)
    arcs = sorted(zip(want["arc_u"].tolist(), want["arc_v"].tolist(), want["arc_mult"].tolist()))
    # the last room cannot fill
    runs = {}
    for rows in (0, 500, 4000, 20000, 60000, 10 ** 8):
        monkeypatch.setenv("MSC_FAULT", f"rows@{rows}")
        g, runs[rows] = _simplify(f, th)
        assert g["n_rounds"] == want["n_rounds"] > 8
        assert np.array_equal(g["alive"], want["alive"]) and np.array_equal(g["log"], log) and g["arcs"] == arcs
    assert runs[0] > runs[10 ** 8] and len(set(runs.values())) > 2  # gathers, in different rounds
    assert g["longest"] >= row
