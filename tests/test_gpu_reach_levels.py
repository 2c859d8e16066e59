"""Saddle-saddle reachability against the level rule written with torch operators on the decoded
gradient: the reached set, the number of levels and where the iteration cap trips, on grids to both
sides of each line between sweeps, pushed levels and the one-cluster levels, and after a replayed pass."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from synth import fields
from tests.cubical import random_field
from tests.gpu_util import dims_of, gpu_field, msc

pytestmark = pytest.mark.gpu


def _waves(nz, ny, nx, seed):
    """Long ridges under faint noise: long paths and many levels."""
    rng = np.random.Generator(np.random.PCG64(seed))
    z, y, x = (np.arange(n, dtype=np.float32) for n in (nz, ny, nx))
    f = np.cos(x / 9)[None, None, :] * np.cos(y / 23)[None, :, None] + 0.7 * np.sin(z / 17)[:, None, None] * np.cos(y / 31)[None, :, None]
    return (f + 1e-3 * rng.standard_normal((nz, ny, nx), dtype=np.float32)).astype(np.float32)


CASES = {
    "tiny": lambda: random_field((2, 3, 4), 1, "normal"),
    "lattice": lambda: fields.cosine_lattice(),
    "rows-2048": lambda: fields.grf((32, 32, 64), 3.0, seed=3),   # the largest grid of one cluster
    "rows-2112": lambda: fields.grf((33, 32, 64), 3.0, seed=4),   # sweeps, then one cluster
    "ridges-small": lambda: _waves(40, 90, 70, 5),
    "ridges": lambda: _waves(96, 100, 130, 6),
    "rows-405000": lambda: _waves(450, 450, 33, 7),                 # sweeps, pushes, then one cluster
}


def _shift(R, d):
    """R at v + d (offsets z, y, x), False outside."""
    out = torch.zeros_like(R)
    dst, src = [], []
    for n, o in zip(R.shape, d):
        dst.append(slice(max(0, -o), n - max(0, o)))
        src.append(slice(max(0, o), n - max(0, -o)))
    out[tuple(dst)] = R[tuple(src)]
    return out


def _reference(words):
    """The reached 1-cells by axis, and the new cells of every level, by the definition: a cell paired
    with a quad is reached one level after another facet of that quad."""
    unit = lambda a, s=1: [s if 2 - i == a else 0 for i in range(3)]  # noqa: E731
    plus = lambda *d: [sum(c) for c in zip(*d)]  # noqa: E731
    code = [(words >> (3 << a)) & 7 for a in range(3)]  # slot 1 << a, 3 bits each
    R = [c == 0 for c in code]
    new = [sum(int(r.sum()) for r in R)]
    while new[-1]:
        add = []
        for a in range(3):
            acc = torch.zeros_like(R[a])
            for b in range(3):
                if b == a:
                    continue
                for s in (-1, 1):
                    paired = code[a] == 1 + 2 * b + (s > 0)
                    back = unit(b, -1) if s < 0 else [0, 0, 0]
                    acc |= paired & (_shift(R[a], unit(b, s)) | _shift(R[b], plus(unit(a), back)) | _shift(R[b], back))
            add.append(acc & ~R[a])
        new.append(sum(int(x.sum()) for x in add))
        R = [r | x for r, x in zip(R, add)]
    return R, new[:-1]


def _unpacked(visited, nz, ny, nx):
    W = (nx + 31) // 32
    w = visited.view(torch.int32).view(nz, 2, ny, 2, W)
    bits = lambda v: ((v[..., None] >> torch.arange(32, device=v.device)) & 1).reshape(nz, ny, 32 * W)[..., :nx] == 1  # noqa: E731
    return [bits(w[:, 0, :, 0]), bits(w[:, 0, :, 1]), bits(w[:, 1, :, 0])]


@pytest.mark.parametrize("name", list(CASES))
def test_levels_and_reached_set(name):
    m = msc()
    f = CASES[name]()
    nz, ny, nx = f.shape
    d = gpu_field(f)
    plan = m.Plan(dims_of(f))
    m.msc_gradient(plan, d)
    want, new = _reference(m.msc_gradient_words(plan).view(torch.int32))
    for step in range(3):  # stage by stage, a synchronised pass, a replayed one
        if step:
            m.msc_compute(plan, d)
        visited, levels = m.msc_reachability(plan)
        assert levels == len(new)
        assert all(torch.equal(g, w) for g, w in zip(_unpacked(visited, nz, ny, nx), want))
    assert m.msc_get_stats(plan)["n_reachable"] == sum(new)
    # the cap is looked at after every second level, while that level adds cells
    L = len(new)
    last = (L - 1) // 2 * 2
    for cap in {1, 2, max(1, L - 2), max(1, L - 1), L, L + 1}:
        capped = m.Plan(dims_of(f), max_iterations=cap)
        m.msc_gradient(capped, d)
        if last >= 2 and last + 1 >= cap:
            with pytest.raises(m.MscError, match="ITER_LIMIT"):
                m.msc_reachability(capped)
        else:
            assert m.msc_reachability(capped)[1] == L
