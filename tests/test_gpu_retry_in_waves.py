"""A replayed pass whose field fits every count that the pass was captured for but needs more room for the
rows of J: the pool runs out in the middle of a wave, with blocks of that wave still to start, and the pass
is run again."""
from __future__ import annotations

import numpy as np
import pytest

from synth import fields
from tests.gpu_util import dims_of, gpu_field, msc, to_np

pytestmark = pytest.mark.gpu


def _noise_in_a_slab(n=88, width=20):
    """Many short rows: rough noise in a slab, and a ramp behind it."""
    f = fields.grf((n, n, n), 2.0, seed=52)
    ramp = np.maximum(np.arange(n, dtype=np.float32) - width, 0)[None, None, :] * 10
    return (ramp + np.where(np.arange(n)[None, None, :] < width, f, 0)).astype(np.float32)


def test_pool_runs_out_in_a_wave():
    m = msc()
    short, long = _noise_in_a_slab(), fields.gaussian_blobs(n=88, n_blobs=8, sigma_range=(8, 20), seed=5)
    alone = m.Plan(dims_of(long), path_count_method=2)
    m.msc_compute(alone, gpu_field(long))
    want, need = [to_np(t) for t in m.msc_saddle_arcs(alone)], m.msc_get_stats(alone)
    plan = m.Plan(dims_of(short), path_count_method=2)
    field = gpu_field(short)
    for _ in range(2):
        m.msc_compute(plan, field)
    had = m.msc_get_stats(plan)
    room = lambda n: n + n // 4 + 1024  # noqa: E731  (what a captured pass leaves for a count)
    assert all(need["counts"][k] <= room(had["counts"][k]) for k in range(4))
    assert need["n_junctions"] <= room(had["n_junctions"])
    assert need["n_frontier_entries"] > room(had["n_frontier_entries"])
    field.copy_(gpu_field(long))
    for _ in range(3):  # run again, captured again, replayed
        m.msc_compute(plan, field)
        assert all(np.array_equal(to_np(g), w) for g, w in zip(m.msc_saddle_arcs(plan), want))
