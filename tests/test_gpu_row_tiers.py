"""The row-wise path count's first tiers -- a lane per row, and eight lanes per row for the rows that
outgrow it or for small fields -- against the junction waves, which share no code with them: D* entry by
entry, on fields to both sides of the line between the two, with rows that fill each tier's tables and
counts beyond its widths."""
from __future__ import annotations

import numpy as np
import pytest

from synth import fields
from tests.cubical import random_field
from tests.gpu_util import dims_of, gpu_field, msc, to_np

pytestmark = pytest.mark.gpu

CASES = {
    "two-rows": lambda: random_field((3, 3, 4), 5, "normal"),
    "lattice": lambda: fields.cosine_lattice(),
    "ties": lambda: random_field((21, 30, 33), 6, "ties"),
    # counts beyond 8 bits, D* rows beyond the lane tier's 16 slots and the group tier's 112
    "blobs": lambda: fields.gaussian_blobs(n=56, n_blobs=3, sigma_range=(10, 20), seed=2),
    "grf-small": lambda: fields.grf((40, 51, 64), 3.0, seed=31),    # 21 thousand 1-saddles
    "grf-large": lambda: fields.grf((108, 96, 100), 3.0, seed=32),  # 168 thousand: lanes first
}


@pytest.mark.parametrize("tier", [0, -1])
@pytest.mark.parametrize("name", list(CASES))
def test_first_tiers_agree_with_the_waves(name, tier):
    m = msc()
    f = CASES[name]()
    d = gpu_field(f)
    waves = m.Plan(dims_of(f), path_count_method=2)
    m.msc_compute(waves, d)
    want = [to_np(t) for t in m.msc_saddle_arcs(waves)]
    ws = m.msc_get_stats(waves)
    plan = m.Plan(dims_of(f), path_count_tier=tier, path_count_method=1)
    for _ in range(3):  # synchronised, then replayed
        m.msc_compute(plan, d)
        for g, w in zip(m.msc_saddle_arcs(plan), want):
            assert np.array_equal(to_np(g), w)
        s = m.msc_get_stats(plan)
        assert all(s[k] == ws[k] for k in ("n_iter", "max_path_count", "nnz_Dstar"))
