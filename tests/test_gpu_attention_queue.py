"""The attention backward's work queue: CTAs claim items in any order and number,
so a sample's gradients must have the same bits alone (fewer items than CTAs) and
in a batch of many times as many, and again with the scratch the last call left."""
import numpy as np
import pytest
import torch

from paper_2607_16074_gb300 import jnx as J
from tests.gpu_helpers import randn_bf16, stream

pytestmark = pytest.mark.gpu

# one to five inner tiles of 64 rows, at and just past their edges
LENGTHS = [1, 64, 65, 128, 129, 192, 193, 320]


def _backward(lengths, rows, H, Hkv, hd, qkv, dO, lse, D, ws=None):
    cu = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    N, longest = int(cu[-1]), max(lengths)
    pos = torch.from_numpy(np.concatenate([np.arange(n) for n in lengths]).astype(np.int32)).cuda()
    cu_d = torch.from_numpy(cu).cuda()
    if ws is None:  # scratch holds anything
        ws = torch.full((J.lib().jnx_op_attention_backward_workspace_bytes(N, longest, hd),), 255,
                        dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    args = [t[rows].contiguous() for t in (qkv, dO, lse, D)]
    out = torch.full_like(args[0], float("nan"))
    J.check(J.lib().jnx_op_attention_backward(
        *(a.data_ptr() for a in args), N, H, Hkv, hd, cu_d.data_ptr(), cu.ctypes.data, len(lengths),
        longest, pos.data_ptr(), 1e4, out.data_ptr(), ws.data_ptr(), ws.numel(), status.data_ptr(),
        stream()))
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return out, ws


@pytest.mark.parametrize("H,Hkv,hd", [(4, 2, 64), (2, 2, 128), (8, 1, 256)])
def test_a_sample_has_the_same_bits_alone_and_in_a_long_queue(H, Hkv, hd):
    lengths = LENGTHS * 24  # 408 row tiles: more of each pass than SMs
    starts = np.concatenate([[0], np.cumsum(lengths)])
    N = int(starts[-1])
    qkv, dO = randn_bf16((N, (H + 2 * Hkv) * hd), 5), randn_bf16((N, H * hd), 6)
    lse = torch.full((N, H), 8.0, device="cuda")  # any: P = 2^(s - lse) stays finite
    D = torch.randn((N, H), generator=torch.Generator().manual_seed(7)).cuda()
    every = slice(0, N)
    full, ws = _backward(lengths, every, H, Hkv, hd, qkv, dO, lse, D)
    assert torch.isfinite(full.float()).all()
    again, _ = _backward(lengths, every, H, Hkv, hd, qkv, dO, lse, D, ws)
    assert torch.equal(full, again)
    for i in list(range(len(LENGTHS))) + [len(lengths) - 1]:
        rows = slice(int(starts[i]), int(starts[i + 1]))
        alone, _ = _backward([lengths[i]], rows, H, Hkv, hd, qkv, dO, lse, D)
        assert torch.equal(alone, full[rows]), (i, lengths[i])
