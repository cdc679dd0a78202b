"""The flow experts' sampler where its own paths can go wrong: contractions long
enough to be split over a cluster (F >= 2,048) with one row, one tile and two
tiles of rows a tenant, more Euler steps than the time embeddings' buffers
hold at once (few rows, and no blocks at all), and groups with more slots than
those buffers have rows."""
import copy

import numpy as np
import pytest
import torch

from oracle import flow as Fl
from paper_2607_16074_gb300 import runtime as R
from tests.gpu_helpers import f64
from tests.helpers import BF16_TOL, rel_err
from tests.test_gpu_flow import FlowSetup, built  # noqa: F401  (built: the library's fixture)

pytestmark = pytest.mark.gpu


def _sample(s, plan, hidden, noise, steps):
    g = R.DeviceGroup(plan)
    ws = torch.zeros(max(s.heads.workspace_bytes(g), 256), dtype=torch.uint8, device="cuda")
    out = torch.full_like(noise, float("nan"))
    s.heads.sample(g, hidden, noise, steps, out, ws)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("F,C,nb,steps", [(2048, 1, 1, 5), (2304, 16, 1, 3), (4096, 64, 1, 2),
                                          (256, 1, 1, 7), (256, 4, 0, 5)])
def test_sampling_vs_oracle_and_alone(F, C, nb, steps):
    s = FlowSetup(F=F, C=C, nb=nb, std=0.02)
    plan = s.plan()
    gen = torch.Generator().manual_seed(2)
    hidden = torch.randn(plan.n_tokens, 256, generator=gen).to(torch.bfloat16).cuda()
    noise = torch.randn(plan.n_samples, C, s.D, generator=gen).cuda()
    out = _sample(s, plan, hidden, noise, steps)
    H, cu, seg = f64(hidden), plan.cu_seqlens, plan.seg_offsets
    for gi, t in enumerate(plan.slot_tenant.tolist()):
        p = s.oracle_params(t)
        for i in range(seg[gi], seg[gi + 1]):
            ref = Fl.sample(p, s.nh, H[cu[i]:cu[i + 1]], f64(noise[i]), steps)
            assert rel_err(f64(out[i]), ref) < BF16_TOL, (t, i)  # bf16 operands of every product
        # the tenant alone: the same bits
        s0, s1 = seg[gi], seg[gi + 1]
        alone = _sample(s, s.plan([t]), hidden[cu[s0]:cu[s1]].contiguous(),
                        noise[s0:s1].contiguous(), steps)
        assert torch.equal(alone, out[s0:s1]), t


@pytest.mark.parametrize("nb,empty", [(0, 4), (1, 4), (2, 12)])
def test_slots_without_samples_change_nothing(nb, empty):
    """One sample, then a group that names it in its last of several slots, the others
    empty: with a chunk of one row the buffers of a step's time embeddings hold max(1, nb)
    rows, fewer than there are slots."""
    s = FlowSetup(F=256, C=1, nb=nb, std=0.05)
    plan = s.plan([1])
    many = copy.copy(plan)
    many.n_slots = empty + 1
    many.seg_offsets = np.array([0] * (empty + 1) + [1], dtype=np.int32)
    many.slot_tenant = np.array([0, 2] * (empty // 2) + [1], dtype=np.int32)
    many.sample_slot = np.array([empty], dtype=np.int32)
    gen = torch.Generator().manual_seed(2)
    hidden = torch.randn(plan.n_tokens, 256, generator=gen).to(torch.bfloat16).cuda()
    noise = torch.randn(1, 1, s.D, generator=gen).cuda()
    want = _sample(s, plan, hidden, noise, 5)
    assert torch.isfinite(want).all()
    assert torch.equal(_sample(s, many, hidden, noise, 5), want)
