"""The lower-star core on the CPU against the oracle on fields whose large stars are full of ties and near
ties: whole keys equal, keys equal but for their lowest bits in and out of index order, and both mixed.
The ranked path keeps the first two and must hand the third to the pairwise comparisons."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from synth import fields
from tests.test_kernel_core_host import host_lib  # noqa: F401  (fixture)


def _low_bits(base, bits):
    """base with its keys' lowest five bits replaced (base > 0, so the order of keys is that of the bits)."""
    return ((base.astype(np.float32).view(np.uint32) & ~np.uint32(31)) | bits.astype(np.uint32)).view(np.float32)


def _cases():
    rng = np.random.default_rng(9)
    g = fields.grf((20, 24, 28), 3.0, seed=11)
    levels = np.round((g - g.min()) / (g.max() - g.min()) * 15).astype(np.float32) + 1
    index = np.arange(g.size).reshape(g.shape)
    return {
        "8-bit": np.round((g - g.min()) / (g.max() - g.min()) * 255).astype(np.float32),
        "16-levels": levels,
        "constant": np.full((6, 7, 9), 2.5, np.float32),
        "low-bits-in-order": _low_bits(levels, index * 32 // index.size),
        "low-bits-reversed": _low_bits(levels, 31 - index * 32 // index.size),
        "low-bits-random": _low_bits(levels, rng.integers(0, 32, g.shape)),
        "low-bits-sparse": _low_bits(levels, np.where(rng.random(g.shape) < 0.1, rng.integers(0, 32, g.shape), 7)),
    }


@pytest.mark.parametrize("name", list(_cases()))
def test_ties_match_oracle(host_lib, name):  # noqa: F811
    f = np.ascontiguousarray(_cases()[name])
    nz, ny, nx = f.shape
    d = np.array([nx, ny, nz], dtype=np.int64)
    words = np.empty(f.shape, dtype=np.uint32)
    assert host_lib.host_words(d.ctypes.data, f.ctypes.data, words.ctypes.data) == 0
    assert np.array_equal(words, oracle.pack(d, oracle.gradient(f)))
