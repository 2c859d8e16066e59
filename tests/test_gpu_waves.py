"""Junction waves (path_count_method 2) against the oracle's D*: a field whose longest row is merged by a
block (317 entries), others by warps, and fields with hardly a junction; synchronised and replayed."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from synth import fields
from tests.cubical import random_field
from tests.gpu_util import csr_to_coo, dims_of, gpu_field, msc, to_np

pytestmark = pytest.mark.gpu

CASES = {
    "tiny": lambda: random_field((2, 3, 4), 1, "normal"),
    "lattice": lambda: fields.cosine_lattice(),
    "ties": lambda: random_field((20, 21, 33), 8, "ties"),
    "long-rows": lambda: fields.gaussian_blobs(n=88, n_blobs=8, sigma_range=(8, 20), seed=5),
}


@pytest.mark.parametrize("name", list(CASES))
def test_waves_match_oracle(name):
    m = msc()
    f = CASES[name]()
    er, ec, en = oracle.compute_all(f, with_minor=False, with_dstar=True)["dstar"]
    plan = m.Plan(dims_of(f), path_count_method=2)
    for _ in range(3):
        m.msc_compute(plan, gpu_field(f))
        rows, cols, cnt = csr_to_coo(*(to_np(x) for x in m.msc_saddle_arcs(plan)))
        assert np.array_equal(rows, er) and np.array_equal(cols, ec) and np.array_equal(cnt, en)
