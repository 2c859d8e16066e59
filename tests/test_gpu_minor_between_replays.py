"""The minor's matrices asked for between replayed passes: the replays' own buffers stay where the captured
graph has them, so the passes after it give what the passes before it gave."""
from __future__ import annotations

import numpy as np
import pytest

from synth import fields
from tests.gpu_util import dims_of, gpu_field, msc, to_np

pytestmark = pytest.mark.gpu


def test_minor_between_replays():
    m = msc()
    f = fields.grf((60, 64, 70), 3.0, seed=51)
    d = gpu_field(f)
    plan = m.Plan(dims_of(f))
    for _ in range(3):
        m.msc_compute(plan, d)
    want = [to_np(t) for t in m.msc_saddle_arcs(plan)]
    minor = [[to_np(t) for t in m.msc_minor(plan, w)] for w in range(4)]
    for _ in range(2):
        m.msc_compute(plan, d)
        assert all(np.array_equal(to_np(g), w) for g, w in zip(m.msc_saddle_arcs(plan), want))
    again = [[to_np(t) for t in m.msc_minor(plan, w)] for w in range(4)]
    assert all(np.array_equal(a, b) for x, y in zip(minor, again) for a, b in zip(x, y))


def test_larger_field_by_stages_between_replays():
    """A field with more cells run stage by stage on a plan with a captured pass: its lists grow, and the
    next pass is captured again."""
    m = msc()
    smooth, rough = (gpu_field(fields.grf((40, 48, 52), a, seed=52)) for a in (5.0, 2.0))
    plan = m.Plan((52, 48, 40))
    for _ in range(3):
        m.msc_compute(plan, smooth)
    want = [to_np(t) for t in m.msc_saddle_arcs(plan)]
    m.msc_gradient(plan, rough)
    got = [to_np(t) for t in m.msc_saddle_arcs(plan)]
    alone = m.Plan((52, 48, 40))
    m.msc_compute(alone, rough)
    assert all(np.array_equal(g, to_np(w)) for g, w in zip(got, m.msc_saddle_arcs(alone)))
    for _ in range(2):
        m.msc_compute(plan, smooth)
        assert all(np.array_equal(to_np(g), w) for g, w in zip(m.msc_saddle_arcs(plan), want))
