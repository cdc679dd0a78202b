"""The GEMM's tile widths against each other and the oracle: a launch picks its
tiles by its size, and a row's result must have the same bits in all of them
(at K = 320 the fewer rows take the narrow ones, the more the wide ones; at K = 4,160
607 rows take a CTA pair's narrow ones and the full rows its wide ones)."""
import pytest
import torch

from oracle import model as M
from paper_2607_16074_gb300 import jnx as J
from tests.gpu_helpers import f64, randn_bf16, stream
from tests.helpers import check_bf16_out, rel_err

pytestmark = pytest.mark.gpu

ROWS = 5000
N = 2048
KS = 320, 4160  # five K steps, shorter than the rings, and 65: no multiple of them


def _run(A, W, rows, epi, x0, pos, hd, act):
    out = {J.JNX_EPI_F32: lambda: torch.full((rows, N), float("nan"), device="cuda"),
           J.JNX_EPI_RESID: lambda: x0[:rows].clone(),
           J.JNX_EPI_GLU: lambda: torch.zeros((rows, N // 2), dtype=torch.bfloat16, device="cuda"),
           }.get(epi, lambda: torch.zeros((rows, N), dtype=torch.bfloat16, device="cuda"))()
    ws = torch.zeros(J.lib().jnx_op_gemm_workspace_bytes(900, hd or 64), dtype=torch.uint8,
                     device="cuda")
    rope, K = epi == J.JNX_EPI_ROPE, A.shape[1]
    J.check(J.lib().jnx_op_gemm(A.data_ptr(), W.data_ptr(), rows, N, K, epi, out.data_ptr(),
                                out.shape[1], pos.data_ptr(), 900 if rope else 0,
                                N // 2 if rope else 0, hd, 10000.0, act, ws.data_ptr(), ws.numel(),
                                stream()))
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("K", KS)
@pytest.mark.parametrize("epi,hd,act", [
    (J.JNX_EPI_F32, 0, 0), (J.JNX_EPI_BF16, 0, 0), (J.JNX_EPI_RESID, 0, 0), (J.JNX_EPI_GLU, 0, 0),
    (J.JNX_EPI_GLU, 0, 1), (J.JNX_EPI_GLU_SAVE, 0, 0), (J.JNX_EPI_ROPE, 64, 0),
    (J.JNX_EPI_ROPE, 128, 0), (J.JNX_EPI_ROPE, 256, 0)])
def test_rows_have_the_same_bits_in_every_tile_width(epi, hd, act, K):
    A, W = randn_bf16((ROWS, K), 1), randn_bf16((N, K), 2, 0.05)
    x0 = torch.randn((ROWS, N), generator=torch.Generator().manual_seed(3)).cuda()
    pos = (torch.arange(ROWS, dtype=torch.int32) * 7 % 900).cuda()
    full = _run(A, W, ROWS, epi, x0, pos, hd, act)
    for rows in (1, 16, 17, 100, 129, 300, 607, 1200, 2120, 4999):
        got = _run(A, W, rows, epi, x0, pos, hd, act)
        assert torch.equal(got, full[:rows]), rows
    ref = f64(A) @ f64(W).T
    if epi == J.JNX_EPI_F32:
        assert rel_err(f64(full), ref) < 1e-4  # fp32 accumulation of exact bf16 products
    elif epi == J.JNX_EPI_RESID:
        assert rel_err(f64(full), f64(x0) + ref) < 1e-4
    elif epi == J.JNX_EPI_GLU:
        g = ref.reshape(ROWS, -1, 2, 128)
        gate, up = g[:, :, 0].reshape(ROWS, -1), g[:, :, 1].reshape(ROWS, -1)
        want = (M.silu(gate) if act == 0 else M.gelu_tanh(gate)) * up
        # the output format's own rounding, and beyond it (as the GLU epilogue's
        # other test) fp32 accumulation and the fast sigmoid's few units
        check_bf16_out(f64(full), want, 1e-3, f"glu {act}")
