"""Fields with regions of NaN, the bits that the GPU's own arithmetic gives (0x7FFFFFFF) among them: every
entry point that computes a gradient answers MSC_ERR_NAN, synchronised and replayed, and the plan goes on."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from tests.gpu_util import dims_of, gpu_field, msc, to_np
from tests.test_kernel_core_nan import _masks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [0x7FFFFFFF, 0x7FFFFE40, 0x7FC00000, 0xFFFFFFFF])
@pytest.mark.parametrize("mask", list(_masks(19)))
def test_nan_regions_are_rejected(mask, bits):
    m = msc()
    where = _masks(19)[mask]
    clean = np.random.default_rng(6).standard_normal(where.shape).astype(np.float32)
    bad = gpu_field(np.where(where, np.uint32(bits), clean.view(np.uint32)).view(np.float32))
    assert torch.isnan(bad).any()
    field = gpu_field(clean)
    plan = m.Plan(dims_of(clean))
    for run in range(4):  # the NaN field synchronised first, then in a captured pass
        if run != 1:
            held = field.clone()
            field.copy_(bad)
            with pytest.raises(m.MscError) as e:
                m.msc_compute(plan, field)
            assert e.value.status == 2
            field.copy_(held)
        m.msc_compute(plan, field)
    alone = m.Plan(dims_of(clean))
    m.msc_compute(alone, field)
    assert all(np.array_equal(to_np(a), to_np(b)) for a, b in zip(m.msc_saddle_arcs(plan), m.msc_saddle_arcs(alone)))
    m.msc_static_prepare(torch.cuda.current_device())
    n = field.numel()
    words = torch.zeros(field.shape, dtype=torch.int32, device="cuda").view(torch.uint32)
    cells = [torch.zeros(n, dtype=torch.int32, device="cuda").view(torch.uint32) for _ in range(4)]
    with pytest.raises(m.MscError) as e:
        m.msc_gradient_critical_static(bad, words, cells, [n] * 4)
    assert e.value.status == 2
    assert m.msc_gradient_critical_static(field, words, cells, [n] * 4) == m.msc_critical(alone)[0]


def test_numbers_of_every_size_keep_their_words():
    """Both zeros, denormals, the largest numbers and infinities, many of them equal, against the oracle."""
    m = msc()
    rng = np.random.default_rng(12)
    bits = np.array([0, 1, 2, 0x7FFFFF, 0x800000, 0x3F800000, 0x7F7FFFFF, 0x7F800000], np.uint32)
    f = (rng.choice(bits, (13, 21, 35)) | (rng.integers(0, 2, (13, 21, 35), dtype=np.uint32) << 31)).view(np.float32)
    plan = m.Plan(dims_of(f))
    m.msc_gradient(plan, gpu_field(f))
    m.msc_critical(plan)
    assert np.array_equal(to_np(m.msc_gradient_words(plan)), oracle.pack(dims_of(f), oracle.gradient(f)))
