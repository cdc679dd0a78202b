"""The final norm's mean pool: the launch takes one of two forms by the number of
samples, and a sample's pooled features must have the same bits in both (alone, and
in a group whose CTAs fill the SMs), with and without the normed rows."""
import numpy as np
import pytest
import torch

from paper_2607_16074_gb300 import jnx as J
from tests.gpu_helpers import f64, randn_bf16, stream
from tests.helpers import rel_err

pytestmark = pytest.mark.gpu

# shares of 8 CTAs that do and do not come out in whole rounds of two and of four rows
LENGTHS = [1, 3, 8, 9, 17, 33, 272, 280, 283, 297, 300, 305, 320]


def _pool(x, gamma, lengths, hidden=None):
    cu = torch.from_numpy(np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)).cuda()
    out = torch.full((len(lengths), x.shape[1]), float("nan"), device="cuda")
    J.check(J.lib().jnx_op_final_pool(x.data_ptr(), gamma.data_ptr(), 1e-5, cu.data_ptr(),
                                      len(lengths), x.shape[1], out.data_ptr(),
                                      None if hidden is None else hidden.data_ptr(), stream()))
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("d", [256, 1024, 2048, 4096])
def test_a_sample_pools_to_the_same_bits_alone_and_in_a_large_group(d):
    lengths = LENGTHS * 9  # 117 samples
    starts = np.concatenate([[0], np.cumsum(lengths)])
    x = torch.randn((int(starts[-1]), d), generator=torch.Generator().manual_seed(3)).cuda()
    gamma = randn_bf16((d,), 4)
    full = _pool(x, gamma, lengths)
    hidden = torch.full(x.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    assert torch.equal(_pool(x, gamma, lengths, hidden), full)
    assert torch.isfinite(hidden).all()
    for i, L in enumerate(LENGTHS):
        rows = x[int(starts[i]):int(starts[i + 1])].contiguous()
        assert torch.equal(_pool(rows, gamma, [L])[0], full[i]), L
        r = f64(rows)
        want = f64(gamma) * (r / np.sqrt((r * r).mean(1, keepdims=True) + 1e-5)).mean(0)
        assert rel_err(f64(full[i]), want) < 1e-5, L  # fp32 sums of at most 320 rows
