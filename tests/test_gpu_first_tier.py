"""The row-wise path count's first tier is chosen by the number of 1-saddles, also in a captured pass, whose
capacity for them lies a quarter and 1024 higher."""
from __future__ import annotations

import numpy as np
import pytest

from synth import fields
from tests.gpu_util import dims_of, gpu_field, msc, to_np

pytestmark = pytest.mark.gpu


# 1-saddles of the field: below the line by more than the headroom, by less, and above it
@pytest.mark.parametrize("n,group_first", [(64, True), (89, True), (96, False)])
def test_first_tier_of_a_replay(n, group_first):
    m = msc()
    f = fields.grf((n, n, n), 3.0, seed=52)
    d = gpu_field(f)
    launches, arcs = {}, {}
    for tier in (0, -1):  # -1: a lane per row first, then eight lanes for what it defers
        plan = m.Plan(dims_of(f), path_count_tier=tier, path_count_method=1)
        for _ in range(3):
            m.msc_compute(plan, d)
        launches[tier] = m.msc_get_stats(plan)["n_launches"]
        arcs[tier] = [to_np(t) for t in m.msc_saddle_arcs(plan)]
        n1 = m.msc_get_stats(plan)["counts"][1]
    assert (n1 <= 128 * 1024) == group_first and (n != 89 or n1 + n1 // 4 + 1024 > 128 * 1024)
    assert launches[0] == launches[-1] - group_first
    assert all(np.array_equal(a, b) for a, b in zip(arcs[0], arcs[-1]))
