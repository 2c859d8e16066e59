"""What is asked for after a pass may grow its own buffers between replays without costing the plan its
captured pass: with MSC_FAULT=capture@2 a second capture would fail."""
from __future__ import annotations

import numpy as np
import pytest

from tests.cubical import random_field
from tests.gpu_util import dims_of, gpu_field, msc, to_np

pytestmark = pytest.mark.gpu

SHAPE = (8, 9, 10)  # 720 vertices: every count stays within the headroom of an empty complex


def _asked_for(m, plan, field):
    """Every output on request."""
    out = [to_np(t) for t in m.msc_saddle_arcs_csc(plan)]
    for w in range(4):
        out += [to_np(t) for t in m.msc_minor(plan, w)]
    out += [to_np(t) for t in m.msc_arc_geometry(plan)]
    out += [to_np(t) for t in m.msc_saddle_arc_geometry(plan)]
    r = m.msc_simplify(plan, field, 0.5)
    return out + [to_np(r[k]) for k in ("alive", "nodeptr", "adj", "mult", "log")]


def test_growing_requests_keep_the_captured_pass(monkeypatch):
    m = msc()
    z, y, x = np.mgrid[:SHAPE[0], :SHAPE[1], :SHAPE[2]].astype(np.float32)
    ramp, noise = gpu_field(x + 20 * y + 400 * z), gpu_field(random_field(SHAPE, 7, "normal"))
    alone = m.Plan(dims_of(noise))
    m.msc_compute(alone, noise)
    want = _asked_for(m, alone, noise)
    monkeypatch.setenv("MSC_FAULT", "capture@2")
    plan = m.Plan(dims_of(noise), path_count_method=1)  # so that the first pass leaves its staging room too
    field = ramp.clone()
    for _ in range(3):  # synchronised, captured, replayed
        m.msc_compute(plan, field)
        _asked_for(m, plan, field)
    field.copy_(noise)  # a complex a few hundred times larger, within the headroom of the captured pass
    for _ in range(3):
        m.msc_compute(plan, field)
        assert all(np.array_equal(g, w) for g, w in zip(_asked_for(m, plan, field), want))


def test_a_failed_capture_is_reported(monkeypatch):
    m = msc()
    f = gpu_field(random_field(SHAPE, 8, "normal"))
    monkeypatch.setenv("MSC_FAULT", "capture@1")
    plan = m.Plan(dims_of(f))
    m.msc_compute(plan, f)
    with pytest.raises(m.MscError, match="injected capture failure"):
        m.msc_compute(plan, f)
    m.msc_compute(plan, f)  # the next capture succeeds
    alone = m.Plan(dims_of(f))
    m.msc_compute(alone, f)
    assert m.msc_critical(plan)[0] == m.msc_critical(alone)[0]
