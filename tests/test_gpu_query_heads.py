"""Query heads alone, on hidden rows of small ragged samples: predictions, losses,
head gradients and the gradient at the rows against the oracle, where their launches
take one path or another."""
import numpy as np
import pytest
import torch

import synth
from oracle import backward as OB
from oracle import model as M
from paper_2607_16074_gb300 import jnx as J
from paper_2607_16074_gb300 import runtime as R
from tests.gpu_helpers import f64
from tests.helpers import oracle_requests, rel_err

pytestmark = pytest.mark.gpu

# chunks of 32 keys and K steps of 64 keys: at, just below and just past their edges
LENGTHS = [[33, 1, 64], [130, 31], [65, 32, 200, 7]]


def _setup(d, lengths, kinds=(synth.HEAD_XATTN,) * 3):
    bb = synth.Backbone(n_layers=0, d=d, n_heads=4, n_kv_heads=4, head_dim=64, d_ff=1024,
                        vision_tokens=1, vocab=100)
    dims = [dict(n_queries=8, q_dim=256), dict(n_queries=8, q_dim=512),
            dict(n_queries=8, q_dim=256)]
    tenants = [synth.Tenant(k, chunk=3, action_dim=5 + 2 * i, d_hidden=64, **dims[i])
               for i, k in enumerate(kinds)]
    w = synth.custom_workload(bb, tenants, [[synth.Sample(0, n) for n in t] for t in lengths],
                              req_batch=2, seed=17)
    hw = synth.make_head_weights(w, std=0.05)
    heads = R.DeviceHeads(w.tenants, d, [{k: v.cuda() for k, v in h.items()} for h in hw])
    plan = J.jnx_group_plan(w.schemas(), oracle_requests(w), len(w.tenants), 1 << 30, 1 << 30)
    return w, hw, heads, plan


def _step(heads, plan, g, X, pooled, targets, off=0):
    """A whole step; the gradient at the rows goes to a buffer `off` floats past a
    16-byte boundary."""
    n, d = X.shape
    ws = torch.full((heads.workspace_bytes(g),), 255, dtype=torch.uint8, device="cuda")
    ws[:256] = 0  # the status word
    preds = torch.full_like(targets, float("nan"))
    loss = torch.full((heads.n,), float("nan"), device="cuda")
    dh = torch.full((n * d + off,), float("nan"), device="cuda")[off:].reshape(n, d)
    heads.forward(g, pooled, X, targets, preds, loss, ws)
    heads.backward_input(g, pooled, X, targets, dh, ws)
    R.check_status(ws)
    torch.cuda.synchronize()
    return preds, loss, dh


def _check(w, hw, heads, plan, X, targets, preds, loss, dh):
    Xn, T0, cu, seg = f64(X), f64(targets), plan.cu_seqlens, plan.seg_offsets
    for gi, t in enumerate(plan.slot_tenant.tolist()):
        tn = w.tenants[t]
        if tn.head_kind != synth.HEAD_XATTN:
            continue
        samples = [s for q in w.requests if q.tenant == t for s in q.samples]
        T = np.stack([T0[s.target_off:s.target_off + tn.width] for s in samples])
        feats = [Xn[cu[i]:cu[i + 1]] for i in range(seg[gi], seg[gi + 1])]
        p = M.widen_tree(synth.to_numpy_tree(hw[t]))
        lo, Y, gr = M.tenant_step(1, p, feats, T)
        assert abs(float(loss[t]) - lo) < 1e-4 * abs(lo)
        got = np.stack([f64(preds[s.target_off:s.target_off + tn.width]) for s in samples])
        assert rel_err(got, Y) < 1e-4, t  # as the 2B-class query heads' test
        for k, v in gr.items():
            assert rel_err(f64(heads.grads[t][k]), v) < 1e-3, (t, k)
        want = np.concatenate(OB.head_feature_grads(1, p, feats, T))
        err = np.abs(f64(dh[cu[seg[gi]]:cu[seg[gi + 1]]]) - want)
        assert (err <= _row_bound(p, feats, T)).all(), t


def _row_bound(p, feats, T):
    """What rounding dk and dv to bf16 (half a unit: 2^-9 of each) moves dk W_k + dv W_v
    by at most, twice over for what came before it."""
    caches = [M.xattn_head_forward(p, X) for X in feats]
    _, dy = M.l2_loss(np.stack([c["y"] for c in caches]), T)
    out = []
    for c, d in zip(caches, dy):
        dO = (d @ p["wout"]).reshape(c["O"].shape)
        dP = dO @ c["v"].T
        dS = c["P"] * (dP - np.sum(dP * c["P"], axis=1, keepdims=True))
        dk, dv = dS.T @ p["q"] / np.sqrt(p["q"].shape[1]), c["P"].T @ dO
        out.append(2.0 ** -8 * (np.abs(dk) @ np.abs(p["wk"]) + np.abs(dv) @ np.abs(p["wv"])))
    return np.concatenate(out)


def _features(plan, d, w):
    gen = torch.Generator().manual_seed(5)
    X = torch.randn((plan.n_tokens, d), generator=gen).to(torch.bfloat16).cuda()
    pooled = torch.randn((plan.n_samples, d), generator=gen).cuda()
    targets = torch.randn(w.n_target, generator=gen).cuda()
    return X, pooled, targets


# widths of whole 256-column tiles and not, buffers on a 16-byte boundary and not, and an
# MLP head between two query heads
@pytest.mark.parametrize("mlp", [False, True])
@pytest.mark.parametrize("d,off", [(512, 0), (512, 2), (384, 0), (640, 0), (640, 2)])
def test_step_and_feature_gradient_vs_oracle(d, off, mlp):
    kinds = [synth.HEAD_XATTN, synth.HEAD_MLP if mlp else synth.HEAD_XATTN, synth.HEAD_XATTN]
    w, hw, heads, plan = _setup(d, LENGTHS, kinds)
    g = R.DeviceGroup(plan)
    X, pooled, targets = _features(plan, d, w)
    preds, loss, dh = _step(heads, plan, g, X, pooled, targets, off)
    assert torch.isfinite(dh).all()
    _check(w, hw, heads, plan, X, targets, preds, loss, dh)


def test_weight_gradients_add_the_small_terms_while_the_sum_is_small():
    """P and dS enter the weight gradients as two bf16 operands, hi and lo; one long
    sample of positive rows, where the hi products of W_v's gradient add to one growing
    sum and the lo ones lose the more bits the later they come.  The bounds lie between
    the two orders' errors on these inputs: W_k 1.28e-5 and W_v 1.46e-5 with every lo
    product after the last hi one, 1.02e-5 and 1.26e-5 with 64 keys of each in turn."""
    d = 512
    w, hw, heads, plan = _setup(d, [[3000]], kinds=(synth.HEAD_XATTN,))
    g = R.DeviceGroup(plan)
    X, _, targets = _features(plan, d, w)
    X = X.abs()
    _step(heads, plan, g, X, None, targets)
    p = M.widen_tree(synth.to_numpy_tree(hw[0]))
    _, _, gr = M.tenant_step(1, p, [f64(X)], f64(targets)[None])
    e = {k: np.linalg.norm(f64(heads.grads[0][k]) - gr[k]) / np.linalg.norm(gr[k])
         for k in ("wk", "wv")}
    assert e["wk"] < 1.15e-5 and e["wv"] < 1.36e-5, e
