"""Reachability whose queue runs full -- where the pushed levels start, in a level pushed by the whole device,
and in the cluster's levels -- gives the reached set and the levels all the same, synchronised and replayed,
and the plan pushes again on a field that fits."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from synth import fields
from tests.gpu_util import dims_of, gpu_field, msc
from tests.test_gpu_reach_levels import CASES, _reference, _unpacked

pytestmark = pytest.mark.gpu


def _plates(nz=330, ny=330, nx=8):
    """A flat grid of 108900 row words, so that levels are pushed by the whole device too; 56 levels of 49,
    134, 219, 299, 379, 459, 539, 619, ... 650 cells."""
    rng = np.random.default_rng(1)
    z, y, x = np.mgrid[:nz, :ny, :nx].astype(np.float32)
    return (np.cos(x / 11) * np.cos(y / 13) + np.sin(z / 12) + 1e-6 * rng.standard_normal((nz, ny, nx))).astype(np.float32)


FIELDS = dict(CASES, plates=_plates)
# field, room in each queue, and the level that it is too small for
ROOMS = [
    ("lattice", 10),      # every level in the cluster: 12 cells to start from
    ("lattice", 100),     # 147 at level 3, which the first block keeps to itself
    ("rows-2048", 20000),  # 30099 at level 1, all blocks
    ("ridges", 200),      # 249 handed over by the sweeps
    ("ridges", 1050),     # 1087 at level 13, as the first block passes on
    ("ridges", 1100),     # 1169 at level 14, all blocks
    ("plates", 150),      # 219 handed over
    ("plates", 300),      # 379 at level 4, the whole device
    ("plates", 560),      # 619 at level 7, which the first block keeps to itself
]


@pytest.mark.parametrize("name,room", ROOMS)
def test_full_queue(name, room, monkeypatch):
    m = msc()
    f = FIELDS[name]()
    nz, ny, nx = f.shape
    d = gpu_field(f)
    monkeypatch.setenv("MSC_FAULT", f"queue@{room}")
    plan = m.Plan(dims_of(f))
    m.msc_gradient(plan, d)
    want, new = _reference(m.msc_gradient_words(plan).view(torch.int32))
    assert max(new) > room
    for step in range(4):  # stage by stage, a synchronised pass, a captured one, a replayed one
        if step:
            m.msc_compute(plan, d)
        visited, levels = m.msc_reachability(plan)
        assert levels == len(new)
        assert all(torch.equal(g, w) for g, w in zip(_unpacked(visited, nz, ny, nx), want))
        assert m.msc_get_stats(plan)["n_reachable"] == sum(new) or step == 0


def _launches(m, plan, field):
    """Kernels of the reachability stage."""
    m.msc_gradient(plan, field)
    m.msc_critical(plan)
    before = m.msc_get_stats(plan)["n_launches"]
    levels = m.msc_reachability(plan)[1]
    return m.msc_get_stats(plan)["n_launches"] - before, levels


def test_sweeps_alone_only_while_the_queue_is_too_small(monkeypatch):
    m = msc()
    deep = gpu_field(fields.cosine_lattice())
    monkeypatch.setenv("MSC_FAULT", "queue@10")  # the lattice starts from 12 cells
    plan = m.Plan((32, 32, 32))
    few = torch.zeros_like(deep) + torch.arange(deep.numel(), device="cuda").view_as(deep) * 1e-3
    few[9:12, 9:12, 9:12] = deep[9:12, 9:12, 9:12]
    want, levels = _launches(m, m.Plan((32, 32, 32)), few)
    assert _launches(m, plan, few) == (want, levels)
    assert _launches(m, plan, deep)[0] > want + 20  # overflowed: ten iterations of sweeps after it
    assert _launches(m, plan, few) == (want, levels)
