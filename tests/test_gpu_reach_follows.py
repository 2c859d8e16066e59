"""A captured pass follows its fields: one that was captured with too few sweeps of the reachability for a
field (whose dense levels it then pushes cell by cell) is captured again with as many as a plan of that field's
own takes, and one with more than its fields need gives them up after many passes."""
from __future__ import annotations

import numpy as np
import pytest

from synth import fields
from tests.gpu_util import gpu_field, msc, to_np

pytestmark = pytest.mark.gpu


def _part_noise(n):
    """Two sweep iterations: white noise in a tenth of the grid, a ramp elsewhere."""
    f = np.random.default_rng(1).standard_normal((n, n, n)).astype(np.float32)
    z = np.arange(n, dtype=np.float32)[:, None, None]
    return np.where(z < 0.1 * n, f, 10 * z).astype(np.float32)


# the levels after the sweeps pushed by the whole device, and in one cluster
@pytest.mark.parametrize("n", [152, 140])
@pytest.mark.parametrize("other,passes", [(_part_noise, 2), (lambda n: fields.gaussian_blobs(n=152, n_blobs=53, seed=4), 70)],
                         ids=["too-few", "too-many"])
def test_sweeps_follow_the_field(n, other, passes):
    m = msc()
    f = gpu_field(fields.grf((n, n, n), 3.0, seed=3))  # three iterations
    own = m.Plan((n, n, n), path_count_method=2)
    for _ in range(3):
        m.msc_compute(own, f)
    want, launches = [to_np(t) for t in m.msc_saddle_arcs(own)], m.msc_get_stats(own)["n_launches"]
    plan = m.Plan((n, n, n), path_count_method=2)
    m.msc_compute(plan, f)
    g = other(n)
    m.msc_gradient(plan, gpu_field(g[:n, :n, :n]))  # the last synchronised stage is another field's
    m.msc_reachability(plan)
    m.msc_compute(plan, f)
    assert m.msc_get_stats(plan)["n_launches"] != launches
    for _ in range(passes):
        m.msc_compute(plan, f)
    assert m.msc_get_stats(plan)["n_launches"] == launches
    assert all(np.array_equal(to_np(a), w) for a, w in zip(m.msc_saddle_arcs(plan), want))
