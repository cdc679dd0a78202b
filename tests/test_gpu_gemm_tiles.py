"""The GEMM's tile widths against each other and the oracle: a launch picks its
tiles by its size, and a row's result must have the same bits in all of them
(at K = 320 the fewer rows take the narrow ones, the more the wide ones; at K = 4,160
607 rows take a CTA pair's narrow ones and the full rows its wide ones)."""
import pytest
import torch

import synth
from oracle import model as M
from paper_2607_16074_gb300 import jnx as J
from paper_2607_16074_gb300 import runtime as R
from tests.gpu_helpers import f64, randn_bf16, stream
from tests.helpers import check_bf16_out, oracle_requests, rel_err

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


@pytest.mark.parametrize("K", [1536, 4160])  # 1,536: lone tiles to 2,120 rows, pairs at 5,000
def test_glu_backward_rows_have_the_same_bits_in_every_tile_form(K):
    """The two GLU backward epilogues (256-wide tiles of one CTA or of a pair) at F =
    2,048: dm into stored multipliers, and dm then the recomputed gate/up product."""
    F, rows_all = 2048, 5000
    A, W = randn_bf16((rows_all, K), 1), randn_bf16((F, K), 2, 0.05)
    Wgu, m0 = randn_bf16((2 * F, K), 3, 0.05), randn_bf16((rows_all, 2 * F), 4)
    L = J.lib()

    def run(rows):
        bwd = m0[:rows].clone()
        J.check(L.jnx_op_gemm_glu_backward(A.data_ptr(), W.data_ptr(), rows, F, K, bwd.data_ptr(),
                                           0, stream()))
        dm = torch.full_like(bwd, float("nan"))
        J.check(L.jnx_op_ffn_glu_backward(A.data_ptr(), W.data_ptr(), A.data_ptr(), Wgu.data_ptr(),
                                          rows, F, K, 0, dm.data_ptr(), stream()))
        torch.cuda.synchronize()
        return bwd, dm

    full = run(rows_all)
    assert all(torch.isfinite(t.float()).all() for t in full)
    for rows in (1, 17, 129, 607, 1200, 2120, 4000):
        for got, want in zip(run(rows), full):
            assert torch.equal(got, want[:rows]), rows


@pytest.mark.parametrize("heads,kv,hd,lora", [(64, 8, 64, 0), (32, 4, 128, 0), (16, 2, 256, 0),
                                              (16, 2, 256, 16), (32, 4, 128, 16)])
def test_a_samples_rows_have_the_same_bits_alone_and_in_a_large_group(heads, kv, hd, lora):
    """Two blocks whose norms are folded into the residual products (4,096-deep: their
    epilogue also writes the norm's rows and sums of squares, which the RoPE and GLU
    epilogues read), with and without adapters: tenants of few rows alone, in narrow
    tiles, against a group of 6,000 rows, in wide ones and pairs."""
    bb = synth.Backbone(n_layers=2, d=512, n_heads=heads, n_kv_heads=kv, head_dim=hd, d_ff=4096,
                        vision_tokens=4, vocab=300, lora_rank=lora)
    lengths = [[9], [100, 1], [170, 120], [596], [600] * 8]
    tenants = [synth.Tenant(synth.HEAD_MLP, chunk=2, action_dim=3, d_hidden=64, max_images=1)
               for _ in lengths]
    w = synth.custom_workload(bb, tenants, [[synth.Sample(1, n) for n in t] for t in lengths],
                              req_batch=2, seed=5)
    weights = synth.make_backbone_weights(w)
    weights = dict(layers=[{k: v.cuda() for k, v in lw.items()} for lw in weights["layers"]],
                   final_norm=weights["final_norm"].cuda(),
                   text_table=weights["text_table"].cuda())
    inp = synth.make_inputs(w)
    vision, text = inp["vision"].cuda(), inp["text_ids"].cuda()
    dev = R.DeviceBackbone(bb, weights, len(tenants))

    def run(wsub):
        plan = J.jnx_group_plan(wsub.schemas(), oracle_requests(wsub), len(tenants), 1 << 30,
                                1 << 30)
        g = R.DeviceGroup(plan)
        ws = torch.zeros(dev.workspace_bytes(plan.n_tokens), dtype=torch.uint8, device="cuda")
        pooled = torch.full((plan.n_samples, bb.d), float("nan"), device="cuda")
        hidden = torch.full((plan.n_tokens, bb.d), float("nan"), dtype=torch.bfloat16,
                            device="cuda")
        dev.forward(g, vision, text, pooled, hidden, ws)
        R.check_status(ws)
        torch.cuda.synchronize()
        return plan, pooled, hidden

    plan, pooled, hidden = run(w)
    assert torch.isfinite(pooled).all() and torch.isfinite(hidden.float()).all()
    seg, cu = plan.seg_offsets, plan.cu_seqlens
    for slot, t in enumerate(plan.slot_tenant.tolist()):
        _, p1, h1 = run(w.subset([t]))
        assert torch.equal(p1, pooled[seg[slot]:seg[slot + 1]]), t
        assert torch.equal(h1, hidden[cu[seg[slot]]:cu[seg[slot + 1]]]), t
