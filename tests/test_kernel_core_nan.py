"""The lower-star core on the CPU, built with the compiler's address and bounds checks, on fields with
regions of NaN: such a field is rejected, but only after the kernel has run on it, so the core has to stay
within its arrays whatever the NaNs' bits are (0x7FFFFFFF is what the GPU's own arithmetic gives).
Fields without a NaN, infinities among them, keep the words of the oracle."""
from __future__ import annotations

import os
import subprocess

import numpy as np
import pytest

import oracle
from synth import fields

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def words_of(tmp_path_factory):
    d = tmp_path_factory.mktemp("nan")
    exe = str(d / "core")
    subprocess.check_call(["g++", "-O1", "-g", "-std=c++17", "-fsanitize=address,undefined", "-fno-sanitize-recover=all",
                           "-o", exe, os.path.join(HERE, "host_harness", "nan_fields_host.cpp")])

    def run(f):
        nz, ny, nx = f.shape
        (d / "in").write_bytes(np.array([nx, ny, nz], np.int64).tobytes() + np.ascontiguousarray(f).tobytes())
        r = subprocess.run([exe, str(d / "in"), str(d / "out")], capture_output=True, text=True)
        assert r.returncode == 0, (r.returncode, r.stderr[:2000])
        return np.frombuffer((d / "out").read_bytes(), np.uint32).reshape(f.shape)

    return run


def _masks(n=14):
    z, y, x = np.mgrid[:n, :n, :n]
    rng = np.random.default_rng(3)
    return {
        "box-inside": (abs(z - 6) < 4) & (abs(y - 7) < 4) & (abs(x - 6) < 4),
        "box-on-faces": (z < 4) | (y >= n - 3) | (x < 2),
        "ball": (z - 6) ** 2 + (y - 6) ** 2 + (x - 7) ** 2 < 25,
        "scattered": rng.random((n, n, n)) < 0.2,
        "pair-on-a-face": (y == 0) & (z == 5) & (abs(x - 5.5) < 1),
        "all": np.ones((n, n, n), bool),
    }


# positive payloads beside and away from the padding words, the usual quiet NaNs, signalling and negative ones
BITS = [0x7FFFFFFF, 0x7FFFFFE0, 0x7FFFFE40, 0x7FFFFCC0, 0x7FC00000, 0x7F800001, 0xFFFFFFFF, 0xFFC00000]


@pytest.mark.parametrize("mask", list(_masks()))
def test_nan_fields_stay_in_bounds(words_of, mask):
    where = _masks()[mask]
    base = np.random.default_rng(4).standard_normal(where.shape).astype(np.float32).view(np.uint32)
    for bits in BITS:
        words_of(np.where(where, np.uint32(bits), base))
    some = np.random.default_rng(5).choice(np.array(BITS[:6], np.uint32), where.shape)
    words_of(np.where(where, some, base))


def test_fields_without_nan_keep_their_words(words_of):
    f = fields.grf((14, 15, 17), 2.5, seed=8)
    for lo, hi in [(-np.inf, np.inf), (-3.4e38, 3.4e38)]:
        g = np.where(f > 1, np.float32(hi), np.where(f < -1, np.float32(lo), f)).astype(np.float32)
        d = np.array(g.shape[::-1], dtype=np.int64)
        assert np.array_equal(words_of(g.view(np.uint32)), oracle.pack(d, oracle.gradient(g)))
