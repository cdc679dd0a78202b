"""What the framework's speed is measured on: its work as a user's program has
it done, through the classes of ``runtime`` and the C ABI that ``jnx`` binds.

Kinds of cases (the sizes are those of the repository's own workloads):

  step         one eager grouped training step of a small group: plan on the
               device, backbone forward, tenant heads, losses, head gradients.
               Latency: some twenty launches of a few microseconds each.
  infer        grouped inference of a few tenants' observations on the 2B-class
               backbone, 18 blocks deep: the serving call of a robot fleet,
               bound by reading the weights and by how few tiles a launch has.
  block        one backbone block over a packed batch (embedding gather to
               final norm), from one sample up to the largest group; with
               tenant adapters (LoRA) where ``lora`` is set.
  lora_train   one adapter training step: forward keeping the residuals, query
               heads, backward through the frozen blocks to every tenant's
               adapters.
  heads_mlp    MLP heads alone on given features: forward, loss, backward with
               the tenants' AdamW steps fused in.
  heads_query  query heads alone on given hidden rows: forward, loss, head
               gradients and the gradient at the rows.
  flow_train   flow-matching experts: forward, loss, backward, AdamW.
  flow_sample  flow-matching experts: Euler sampling of action chunks.
  attention    the varlen attention layer alone, forward with the log-sum-exp
               and backward.

Samples are ragged everywhere: whole images plus a few text tokens, their
lengths drawn from the case's own numbers, so that a case has the same shapes
for every seed; the seed draws weights and inputs.
"""
import ctypes
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2607_16074_gb300 import jnx as J
from paper_2607_16074_gb300 import runtime as R

EPS, THETA, VOCAB, RANK = 1e-6, 10000.0, 32000, 16

# The backbones of the repository's workloads, with the images and text
# lengths their samples have.
MODELS = {
    "tiny": dict(d=256, n_heads=4, n_kv_heads=4, head_dim=64, d_ff=1024, glu=0,
                 vision=64, images=(1, 1), text=(16, 24)),
    "small": dict(d=1024, n_heads=16, n_kv_heads=16, head_dim=64, d_ff=4096, glu=0,
                  vision=256, images=(1, 1), text=(8, 48)),
    "mqa2b": dict(d=2048, n_heads=8, n_kv_heads=1, head_dim=256, d_ff=16384, glu=1,
                  vision=256, images=(1, 3), text=(4, 72)),
    "llama7b": dict(d=4096, n_heads=32, n_kv_heads=32, head_dim=128, d_ff=11008, glu=0,
                    vision=256, images=(1, 1), text=(16, 64)),
}

# The flow experts of the 2B-class group.
FLOW = dict(d_model=1024, d_ff=4096, n_blocks=4, chunk=16, action_dim=32, d_in=2048)


def listed():
    return [
        # the smallest group there is: two tenants, four observations each
        dict(name="step_tiny", kind="step", model="tiny", layers=1, tenants=2, samples=4),
        # two robots ask at once: 557-odd tokens through 18 blocks
        dict(name="infer_mqa2b_2x1", kind="infer", model="mqa2b", layers=18, tenants=2,
             samples=1),
        # an ordinary group on a narrow backbone
        dict(name="block_small", kind="block", model="small", tenants=8, tokens=44000, lora=False),
        # one tenant's microbatch on the wide backbone
        dict(name="block_llama7b_tenant", kind="block", model="llama7b", tenants=1, tokens=2000,
             lora=False),
        # the largest group: the headline workload's 32 tenants
        dict(name="block_llama7b_group", kind="block", model="llama7b", tenants=32, tokens=65536,
             lora=False),
        # tenants with their own adapters, ragged samples of one to three images
        dict(name="block_mqa2b_lora", kind="block", model="mqa2b", tenants=12, tokens=20000,
             lora=True),
        # training those adapters
        dict(name="lora_train_mqa2b", kind="lora_train", model="mqa2b", layers=2, tenants=8,
             samples=16),
        # the heads of the wide backbone's tenants, trained
        dict(name="heads_mlp_train", kind="heads_mlp", tenants=14, samples=7, d=4096,
             hidden=1024, width=56),
        # the query heads of the 2B-class tenants, trained
        dict(name="heads_query_train", kind="heads_query", model="mqa2b", tenants=8, samples=8),
        # flow experts, trained: eight tenants, four observations each
        dict(name="flow_train_8x4", kind="flow_train", tenants=8, samples=4),
        # flow experts, acting: ten Euler steps for two tenants
        dict(name="flow_sample_2x1", kind="flow_sample", tenants=2, samples=1, steps=10),
        # the attention layer alone, both directions
        dict(name="attention_mqa2b", kind="attention", model="mqa2b", tokens=24000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "infer", "block", "block", "block", "lora_train", "heads_mlp",
                       "heads_query", "flow_train", "flow_sample", "attention"])
    if kind == "step":
        return dict(kind=kind, model=rng.choice(["tiny", "tiny", "small"]),
                    layers=rng.randint(1, 2), tenants=rng.randint(1, 8), samples=rng.randint(1, 9))
    if kind == "infer":
        t = rng.randint(1, 8)
        return dict(kind=kind, model="mqa2b", layers=18, tenants=t,
                    samples=rng.randint(1, max(1, 10 // t)))
    if kind == "block":
        model = rng.choice(["small", "mqa2b", "mqa2b", "llama7b"])
        most = {"small": 65536, "mqa2b": 65536, "llama7b": 65536}[model]
        tokens = _log_int(rng, 250, most)
        return dict(kind=kind, model=model, tenants=min(_log_int(rng, 1, 40), 1 + tokens // 300),
                    tokens=tokens, lora=model == "mqa2b" and rng.random() < 0.5)
    if kind == "lora_train":
        t = rng.randint(1, 8)
        return dict(kind=kind, model="mqa2b", layers=rng.randint(1, 2), tenants=t,
                    samples=max(t, _log_int(rng, 1, 32)))
    if kind == "heads_mlp":
        return dict(kind=kind, tenants=rng.randint(1, 14), samples=rng.randint(1, 13),
                    d=rng.choice([1024, 2048, 4096]), hidden=rng.choice([256, 1024]),
                    width=rng.choice([56, 112, 224]))
    if kind == "heads_query":
        return dict(kind=kind, model="mqa2b", tenants=rng.randint(1, 8), samples=rng.randint(1, 16))
    if kind == "flow_train":
        return dict(kind=kind, tenants=rng.randint(1, 8), samples=rng.randint(1, 9))
    if kind == "flow_sample":
        return dict(kind=kind, tenants=rng.randint(1, 8), samples=rng.randint(1, 4),
                    steps=rng.randint(4, 16))
    return dict(kind=kind, model=rng.choice(["small", "mqa2b", "llama7b"]),
                tokens=_log_int(rng, 250, 48000))


# ---------------------------------------------------------------------------
# shapes
# ---------------------------------------------------------------------------

def _zipf(n, total):
    share = [r ** -1.2 for r in range(1, n + 1)]
    got = [max(1, int(total * s / sum(share))) for s in share]
    got[0] += max(0, total - sum(got))
    return got


def _samples(case):
    """Per tenant its samples, each (images, text tokens)."""
    rng = random.Random(repr(sorted((k, v) for k, v in case.items() if k != "name")))
    m = MODELS[case.get("model", "mqa2b")]
    one_image = case["kind"] in ("infer", "flow_train", "flow_sample")

    def sample():
        img = 1 if one_image else rng.randint(*m["images"])
        return img, rng.randint(16, 64) if one_image else rng.randint(*m["text"])

    tenants = case.get("tenants", 1)
    if "tokens" in case:
        per, total, t = [[] for _ in range(tenants)], 0, 0
        while total < case["tokens"] or t < tenants:
            s = sample()
            per[t % tenants].append(s)
            total += s[0] * m["vision"] + s[1]
            t += 1
        return per
    if case["kind"] == "lora_train":
        return [[sample() for _ in range(n)] for n in _zipf(tenants, case["samples"])]
    return [[sample() for _ in range(case["samples"])] for _ in range(tenants)]


def _lengths(case):
    """Every sample's length in packed order (tenants in order)."""
    v = MODELS[case.get("model", "mqa2b")]["vision"]
    return [i * v + t for per in _samples(case) for i, t in per]


def _width(case, t):
    """Outputs per sample of tenant t's head."""
    if case["kind"] in ("lora_train", "heads_query"):
        return 50 * (7, 14, 32)[t % 3]
    if case["kind"] == "heads_mlp":
        return case["width"]
    return 112 if case["kind"] == "infer" else 56


def _features(case):
    """Whether a block's group reads hidden rows (query heads) and pooled
    features (MLP heads); the narrow backbone serves a mixed group."""
    return case["model"] != "llama7b", case["model"] != "mqa2b"


def _plan(case, m):
    """The group's plan: requests of up to four samples, round-robin over the
    tenants, and the samples' places in the observation buffers."""
    per = _samples(case)
    schemas = [dict(backbone_id=0, d_model=m["d"], vision_tokens=m["vision"], embed_dtype=0,
                    vocab_id=VOCAB, rope_id=int(THETA), max_images=3, action_width=_width(case, t))
               for t in range(len(per))]
    reqs, k, vrow, tpos, toff = [], 0, 0, 0, 0
    place = [[] for _ in per]
    while any(4 * k < len(p) for p in per):
        for t, p in enumerate(per):
            part = []
            for img, text in p[4 * k:4 * k + 4]:
                part.append(dict(n_img=img, text_len=text, vision_row=vrow, text_pos=tpos,
                                 target_off=toff))
                vrow, tpos, toff = vrow + img * m["vision"], tpos + text, toff + _width(case, t)
            if part:
                reqs.append(dict(tenant=t, schema=t, samples=part))
                place[t] += part
        k += 1
    return SimpleNamespace(schemas=schemas, requests=reqs, place=place, vision=vrow, text=tpos,
                           targets=toff, tenants=len(per))


def _group(p):
    return R.DeviceGroup(J.jnx_group_plan(p.schemas, p.requests, p.tenants, 1 << 30, 1 << 30))


# ---------------------------------------------------------------------------
# tensors
# ---------------------------------------------------------------------------

class _Draw:
    """The seed's random tensors, in the order they are asked for."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)

    def normal(self, *shape, std=1.0, mean=0.0, dtype=torch.bfloat16):
        x = torch.empty(shape, device="cuda", dtype=dtype)
        x.normal_(mean, std, generator=self.g)
        return x

    def uniform(self, *shape, lo=-1.0, hi=1.0):
        return torch.empty(shape, device="cuda").uniform_(lo, hi, generator=self.g)


def _backbone_weights(rnd, m, layers, lora, tenants):
    d, q, kv, F = m["d"], m["n_heads"] * m["head_dim"], m["n_kv_heads"] * m["head_dim"], m["d_ff"]
    out = []
    for _ in range(layers):
        w = dict(attn_norm=rnd.normal(d, std=0.02, mean=1.0), wq=rnd.normal(q, d, std=0.02),
                 wk=rnd.normal(kv, d, std=0.02), wv=rnd.normal(kv, d, std=0.02),
                 wo=rnd.normal(d, q, std=0.02), ffn_norm=rnd.normal(d, std=0.02, mean=1.0),
                 wg=rnd.normal(F, d, std=0.02), wu=rnd.normal(F, d, std=0.02),
                 wd=rnd.normal(d, F, std=0.02))
        if lora:
            for n, i, o in (("q", d, q), ("k", d, kv), ("v", d, kv), ("o", q, d)):
                w["lora_a_" + n] = rnd.normal(tenants, RANK, i, std=0.02)
                w["lora_b_" + n] = rnd.normal(tenants, o, RANK, std=0.02)
        out.append(w)
    return dict(layers=out, final_norm=rnd.normal(d, std=0.02, mean=1.0),
                text_table=rnd.normal(VOCAB, d))


def _inputs(rnd, p, d):
    return dict(vision=rnd.normal(max(p.vision, 1), d),
                text_ids=torch.randint(0, VOCAB, (max(p.text, 1),), generator=rnd.g, device="cuda",
                                       dtype=torch.int32),
                targets=rnd.uniform(max(p.targets, 1)))


def _mlp_weights(rnd, tenants, d, hidden, width):
    """Every tenant's head as its slice of one stacked parameter."""
    return dict(w1=rnd.normal(tenants, hidden, d, std=0.02),
                b1=rnd.normal(tenants, hidden, std=0.02),
                w2=rnd.normal(tenants, width, hidden, std=0.02),
                b2=rnd.normal(tenants, width, std=0.02))


def _query_weights(rnd, case, tenants, d):
    return [dict(q=rnd.normal(32, 256, std=0.02), wk=rnd.normal(256, d, std=0.02),
                 wv=rnd.normal(256, d, std=0.02),
                 wout=rnd.normal(_width(case, t), 32 * 256, std=0.02),
                 bout=rnd.normal(_width(case, t), std=0.02)) for t in range(tenants)]


def _flow_weights(rnd, T):
    dm, F, D, C = FLOW["d_model"], FLOW["d_ff"], FLOW["action_dim"], FLOW["chunk"]
    r = lambda *shape: rnd.normal(T, *shape, std=0.02)  # noqa: E731
    return dict(w_in=r(dm, D), b_in=r(dm), pos=r(C, dm), t1=r(dm, dm), tb1=r(dm), t2=r(dm, dm),
                tb2=r(dm), w_out=r(D, dm), b_out=r(D),
                blocks=[dict(w_qkv=r(3 * dm, dm), w_kvc=r(2 * dm, FLOW["d_in"]), w_o=r(dm, dm),
                             wg=r(F, dm), wu=r(F, dm), w_d=r(dm, F))
                        for _ in range(FLOW["n_blocks"])])


def _tensors(case, seed):
    """Everything the seed draws for a case; prepare and exact share it."""
    rnd, kind = _Draw(seed), case["kind"]
    m = MODELS[case.get("model", "mqa2b")]
    if kind in ("step", "infer", "block", "lora_train"):
        p = _plan(case, m)
        lora = kind == "lora_train" or bool(case.get("lora"))
        t = dict(p=p, m=m, lora=lora, inp=_inputs(rnd, p, m["d"]),
                 bw=_backbone_weights(rnd, m, case.get("layers", 1), lora, p.tenants))
        if kind in ("step", "infer"):
            t["hw"] = _mlp_weights(rnd, p.tenants, m["d"], 1024 if kind == "infer" else 256,
                                   _width(case, 0))
        elif kind == "lora_train":
            t["hw"] = _query_weights(rnd, case, p.tenants, m["d"])
        return SimpleNamespace(**t)
    if kind == "heads_mlp":
        m = dict(m, d=case["d"])
        p = _plan(case, m)
        n = sum(len(x) for x in p.place)
        return SimpleNamespace(p=p, m=m, pooled=rnd.normal(n, case["d"], dtype=torch.float32),
                               targets=rnd.uniform(p.targets),
                               hw=_mlp_weights(rnd, p.tenants, case["d"], case["hidden"],
                                               case["width"]))
    if kind == "heads_query":
        p = _plan(case, m)
        return SimpleNamespace(p=p, m=m, hidden=rnd.normal(sum(_lengths(case)), m["d"]),
                               targets=rnd.uniform(p.targets),
                               hw=_query_weights(rnd, case, p.tenants, m["d"]))
    if kind in ("flow_train", "flow_sample"):
        p = _plan(case, m)
        n, chunk, dim = sum(len(x) for x in p.place), FLOW["chunk"], FLOW["action_dim"]
        return SimpleNamespace(p=p, hidden=rnd.normal(sum(_lengths(case)), FLOW["d_in"]),
                               actions=rnd.uniform(n, chunk, dim),
                               noise=rnd.normal(n, chunk, dim, dtype=torch.float32),
                               tau=rnd.uniform(n, lo=0.0, hi=1.0),
                               fw=_flow_weights(rnd, p.tenants))
    n, H, Hkv, hd = sum(_lengths(case)), m["n_heads"], m["n_kv_heads"], m["head_dim"]
    return SimpleNamespace(m=m, qkv=rnd.normal(n, (H + 2 * Hkv) * hd),
                           dout=rnd.normal(n, H * hd, dtype=torch.float32))


# ---------------------------------------------------------------------------
# the passes
# ---------------------------------------------------------------------------

def _config(m, layers, lora):
    return SimpleNamespace(n_layers=layers, d=m["d"], n_heads=m["n_heads"],
                           n_kv_heads=m["n_kv_heads"], head_dim=m["head_dim"], d_ff=m["d_ff"],
                           glu=m["glu"], lora_rank=RANK if lora else 0, vocab=VOCAB,
                           vision_tokens=m["vision"], eps=EPS, rope_theta=THETA)


def _mlp_heads(t, hidden, width):
    n = t.p.tenants
    tn = SimpleNamespace(head_kind=J.JNX_HEAD_MLP, d_hidden=hidden, width=width)
    return R.DeviceHeads([tn] * n, t.m["d"], [{k: w[i] for k, w in t.hw.items()} for i in range(n)])


def _query_heads(t, case):
    tns = [SimpleNamespace(head_kind=J.JNX_HEAD_XATTN, n_queries=32, q_dim=256,
                           width=_width(case, i)) for i in range(t.p.tenants)]
    return R.DeviceHeads(tns, t.m["d"], t.hw)


def _space(n):
    return torch.zeros(max(n, 256), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    t, kind = _tensors(case, seed), case["kind"]
    s = SimpleNamespace(case=case, kind=kind, t=t)
    if kind in ("step", "infer", "block", "lora_train"):
        s.bb = R.DeviceBackbone(_config(t.m, case.get("layers", 1), t.lora), t.bw, t.p.tenants)
        s.group = _group(t.p)
        s.preds = torch.zeros_like(t.inp["targets"])
        if kind == "block":
            plan = s.group.plan
            s.ws = _space(s.bb.workspace_bytes(plan.n_tokens))
            rows, pool = _features(case)
            s.hidden = (torch.zeros((plan.n_tokens, t.m["d"]), dtype=torch.bfloat16, device="cuda")
                        if rows else None)
            s.pooled = (torch.zeros((plan.n_samples, t.m["d"]), device="cuda") if pool else None)
        elif kind == "lora_train":
            s.step = R.LoraTrainStep(s.bb, _query_heads(t, case), s.group)
        else:
            s.step = R.GroupedStep(s.bb, _mlp_heads(t, t.hw["w1"].shape[1], _width(case, 0)),
                                   s.group)
    elif kind in ("heads_mlp", "heads_query"):
        s.group = _group(t.p)
        s.heads = (_mlp_heads(t, case["hidden"], case["width"]) if kind == "heads_mlp"
                   else _query_heads(t, case))
        s.preds, s.loss = torch.zeros_like(t.targets), torch.zeros(t.p.tenants, device="cuda")
        s.ws = _space(s.heads.workspace_bytes(s.group))
        if kind == "heads_mlp":
            s.heads.init_optimizer()
        else:
            s.d_hidden = torch.zeros(t.hidden.shape, device="cuda")
    elif kind in ("flow_train", "flow_sample"):
        s.group = _group(t.p)
        s.experts = R.DeviceFlowHeads(dict(FLOW, n_tenants=t.p.tenants), t.fw)
        s.ws = _space(s.experts.workspace_bytes(s.group))
        s.out, s.loss = torch.zeros_like(t.noise), torch.zeros(t.p.tenants, device="cuda")
        if kind == "flow_train":
            s.opt = R.TenantAdamW(s.experts.param_pairs())
    else:
        _prepare_attention(s)
    return s


def _prepare_attention(s):
    t, m = s.t, s.t.m
    lens = _lengths(s.case)
    n, H, hd = sum(lens), m["n_heads"], m["head_dim"]
    s.cu_h = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    s.cu = torch.from_numpy(s.cu_h).cuda()
    s.pos = torch.from_numpy(np.concatenate([np.arange(x) for x in lens]).astype(np.int32)).cuda()
    s.n, s.longest = n, max(lens)
    new = lambda *shape, dtype=torch.bfloat16: torch.zeros(shape, dtype=dtype, device="cuda")  # noqa: E731
    s.out, s.lse, s.d_att = new(n, H * hd), new(n, H, dtype=torch.float32), new(n, H * hd)
    s.delta, s.dqkv = new(n, H, dtype=torch.float32), torch.zeros_like(t.qkv)
    s.status = new(1, dtype=torch.int32)
    s.ws = _space(J.lib().jnx_op_attention_backward_workspace_bytes(n, s.longest, hd))


def _run_attention(s):
    m, L, q = s.t.m, J.lib(), s.t.qkv.data_ptr()
    H, Hkv, hd, stream = (m["n_heads"], m["n_kv_heads"], m["head_dim"],
                          torch.cuda.current_stream().cuda_stream)
    J.check(L.jnx_op_attention_lse(q, s.n, H, Hkv, hd, s.cu.data_ptr(), len(s.cu_h) - 1, s.longest,
                                   s.out.data_ptr(), s.lse.data_ptr(), s.status.data_ptr(), stream))
    J.check(L.jnx_op_attention_backward_prep(s.t.dout.data_ptr(), s.out.data_ptr(), s.n, H, hd,
                                             s.d_att.data_ptr(), s.delta.data_ptr(), stream))
    J.check(L.jnx_op_attention_backward(
        q, s.d_att.data_ptr(), s.lse.data_ptr(), s.delta.data_ptr(), s.n, H, Hkv, hd,
        s.cu.data_ptr(), s.cu_h.ctypes.data_as(ctypes.c_void_p), len(s.cu_h) - 1, s.longest,
        s.pos.data_ptr(), THETA, s.dqkv.data_ptr(), s.ws.data_ptr(), s.ws.numel(),
        s.status.data_ptr(), stream))
    return dict(out=s.out, lse=s.lse, dqkv=s.dqkv)


def run(s):
    t, kind = s.t, s.kind
    if kind == "step":
        s.step.run(t.inp["vision"], t.inp["text_ids"], t.inp["targets"], s.preds)
        return dict(pooled=s.step.pooled, preds=s.preds, loss=s.step.loss,
                    grads=s.step.heads.grads)
    if kind == "infer":
        s.step.infer(t.inp["vision"], t.inp["text_ids"], s.preds)
        return dict(pooled=s.step.pooled, preds=s.preds)
    if kind == "block":
        s.bb.forward(s.group, t.inp["vision"], t.inp["text_ids"], s.pooled, s.hidden, s.ws)
        return dict(pooled=s.pooled, hidden=s.hidden)
    if kind == "lora_train":
        s.step.run(t.inp["vision"], t.inp["text_ids"], t.inp["targets"], s.preds)
        return dict(preds=s.preds, loss=s.step.loss, d_hidden=s.step.d_hidden,
                    grads=s.step.heads.grads, lora=s.bb.lora_grads)
    if kind == "heads_mlp":
        s.heads.forward(s.group, t.pooled, None, t.targets, s.preds, s.loss, s.ws)
        s.heads.backward_adamw(s.group, t.pooled, None, t.targets, s.ws, lr=1e-4,
                               weight_decay=0.01)
        return dict(preds=s.preds, loss=s.loss, params=t.hw,
                    m=[{k: v["m"] for k, v in st.items()} for st in s.heads.opt_state])
    if kind == "heads_query":
        s.heads.forward(s.group, None, t.hidden, t.targets, s.preds, s.loss, s.ws)
        s.heads.backward_input(s.group, None, t.hidden, t.targets, s.d_hidden, s.ws)
        return dict(preds=s.preds, loss=s.loss, d_hidden=s.d_hidden, grads=s.heads.grads)
    if kind == "flow_train":
        s.experts.forward(s.group, t.hidden, t.actions, t.noise, t.tau, s.out, s.loss, s.ws)
        s.experts.backward(s.group, t.hidden, s.ws)
        s.opt.step(range(t.p.tenants), lr=1e-4, weight_decay=0.01)
        return dict(velocity=s.out, loss=s.loss, grads=s.experts.grads,
                    blocks=s.experts.block_grads, master=s.opt.master)
    if kind == "flow_sample":
        s.experts.sample(s.group, t.hidden, t.noise, s.case["steps"], s.out, s.ws)
        return s.out
    return _run_attention(s)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _block_work(m, lens, lora, tenants):
    """(weight bytes, FLOPs) of one block's forward."""
    d, q, kv, F = m["d"], m["n_heads"] * m["head_dim"], m["n_kv_heads"] * m["head_dim"], m["d_ff"]
    w = d * (q + 2 * kv) + q * d + 3 * d * F
    extra = RANK * (2 * d + 2 * q + 2 * (d + kv)) if lora else 0
    n = sum(lens)
    return 2 * (w + tenants * extra), 2 * n * (w + extra) + 4 * q * sum(x * x for x in lens)


def work(case):
    kind = case["kind"]
    m, lens = MODELS[case.get("model", "mqa2b")], _lengths(case)
    n, T = sum(lens), case.get("tenants", 1)
    d = m["d"]
    if kind in ("step", "infer", "block"):
        layers = case.get("layers", 1)
        w, f = _block_work(m, lens, case.get("lora", False), T)
        rows, pool = _features(case) if kind == "block" else (False, True)
        out = rows * n * d * 2 + pool * len(lens) * d * 4
        b, f = layers * w + n * d * 2 + out, layers * f
        if kind != "block":
            hid, wid = (256 if kind == "step" else 1024), _width(case, 0)
            hp = T * (d * hid + hid * wid)
            b += hp * (6 if kind == "step" else 2) + len(lens) * wid * 8
            f += 2 * len(lens) * (d * hid + hid * wid) * (2 if kind == "step" else 1)
        return dict(bytes=b, flops=f)
    query_w = sum(2 * 256 * d + _width(case, t) * 8192 for t in range(T))
    if kind in ("lora_train", "heads_query"):
        # K and V projections forward; to the queries' weights and the rows backward
        per_row = 2 * 2 * 256 * d
        hf = n * (3 * per_row + 12 * 32 * 256) + sum(
            6 * len(p) * _width(case, t) * 8192 for t, p in enumerate(_samples(case)))
        hb = query_w * 6 + n * d * 6
        if kind == "heads_query":
            return dict(bytes=hb, flops=hf)
        layers = case["layers"]
        w, f = _block_work(m, lens, True, T)
        adapters = layers * T * RANK * 4 * (2 * d + 2 * 2048 + 2 * (d + 256))
        # forward, the input gradients' products, attention's five products
        return dict(bytes=layers * w + adapters + n * d * 6 + hb,
                    flops=hf + layers * (2 * f + 6 * 2048 * sum(x * x for x in lens)))
    if kind == "heads_mlp":
        hp, S = case["d"] * case["hidden"] + case["hidden"] * case["width"], T * case["samples"]
        # read g's factors once; moments and master read and written, bf16 read and written
        return dict(bytes=T * hp * 28 + S * (case["d"] + 2 * case["width"]) * 4, flops=6 * S * hp
                    - 2 * S * case["d"] * case["hidden"])
    if kind in ("flow_train", "flow_sample"):
        dm, F, C, D, B = (FLOW[k] for k in ("d_model", "d_ff", "chunk", "action_dim", "n_blocks"))
        S, di = len(lens), FLOW["d_in"]
        act, ctx = B * (4 * dm * dm + 3 * dm * F), B * 2 * dm * di
        params = act + ctx + 2 * dm * dm + 2 * D * dm + C * dm
        att = B * sum(4 * C * (x + C) * dm for x in lens)
        rows = S * C
        if kind == "flow_sample":
            k = case["steps"]
            return dict(bytes=2 * T * params + 2 * n * di + rows * D * 8,
                        flops=2 * n * ctx + k * (2 * rows * act + att))
        # products forward, to the inputs (not to the frozen rows) and to the weights; then AdamW:
        # master and moments read and written, the gradient written, bf16 read and written
        return dict(bytes=T * params * 32 + 2 * n * di + rows * D * 12,
                    flops=2 * 2 * n * ctx + 3 * 2 * rows * act + 3 * att)
    H, Hkv, hd = m["n_heads"], m["n_kv_heads"], m["head_dim"]
    # two products forward, five backward
    return dict(bytes=n * ((H + 2 * Hkv) * hd * 4 + H * hd * 6 + H * 4),
                flops=14 * H * hd * sum(x * x for x in lens))


def tolerance(case):
    """About four times what a pass was off from 64 bits on GB300 (the worst
    output of each kind).  bf16 storage between the stages sets nearly all of
    them; a 2B-class forward is 18 blocks of it, adapter and expert gradients
    are sums through several such roundings.  The MLP heads are fp32 (3e-6):
    their "max" lets a bf16 parameter that sits on a rounding boundary move by
    one unit."""
    kind, model = case["kind"], case.get("model")
    if kind == "step":
        return {"rel": 1.2e-3, "max": 8e-3} if model == "tiny" else {"rel": 6e-3, "max": 3e-2}
    if kind == "block":
        return {"rel": 1.2e-2, "max": 6.5e-2}
    return {"infer": {"rel": 3e-2, "max": 0.15}, "lora_train": {"rel": 3e-2, "max": 0.3},
            "heads_mlp": {"rel": 5e-5, "max": 8e-3}, "heads_query": {"rel": 6.6e-3, "max": 8e-2},
            "flow_train": {"rel": 3e-2, "max": 0.5}, "flow_sample": {"rel": 6e-3, "max": 3e-2},
            "attention": {"rel": 1.2e-2, "max": 0.14}}[kind]


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _d(x):
    return x.double()


def _norm(x, gamma=None):
    y = x * torch.rsqrt(x.square().mean(-1, keepdim=True) + EPS)
    return y if gamma is None else y * _d(gamma)


def _rope(x, pos, sign=1.0):
    """x [n, heads, hd]."""
    half = x.shape[-1] // 2
    inv = THETA ** (-torch.arange(half, device=x.device, dtype=torch.float64) / half)
    a = pos.double()[:, None, None] * inv
    c, s = a.cos(), sign * a.sin()
    lo, hi = x[..., :half], x[..., half:]
    return torch.cat([lo * c - hi * s, hi * c + lo * s], -1)


def _attend(q, k, v, lens):
    """Attention inside each sample; q [n, H, hd], k and v [n, Hkv, hd]."""
    out, lse, at = [], [], 0
    g = q.shape[1] // k.shape[1]
    for L in lens:
        qs, ks, vs = (x[at:at + L].transpose(0, 1) for x in (q, k, v))
        ks, vs = ks.repeat_interleave(g, 0), vs.repeat_interleave(g, 0)
        s = qs @ ks.transpose(1, 2) / math.sqrt(q.shape[-1])
        out.append((s.softmax(-1) @ vs).transpose(0, 1))
        lse.append(s.logsumexp(-1).transpose(0, 1) / math.log(2.0))
        at += L
    return torch.cat(out), torch.cat(lse)


def _backbone(t, lens, tenant_of, adapters=None):
    """The final normed rows [n, d] and the packed rows' sample offsets."""
    m, p = t.m, t.p
    rows = []
    for place in p.place:
        for s in place:
            rows.append(t.inp["vision"][s["vision_row"]:s["vision_row"] + s["n_img"] * m["vision"]])
            ids = t.inp["text_ids"][s["text_pos"]:s["text_pos"] + s["text_len"]]
            rows.append(t.bw["text_table"][ids.long()])
    x = _d(torch.cat(rows))
    n, H, Hkv, hd = len(x), m["n_heads"], m["n_kv_heads"], m["head_dim"]
    pos = torch.cat([torch.arange(L, device=x.device) for L in lens])
    for i, w in enumerate(t.bw["layers"]):
        def project(x, names, lora):
            y = x @ torch.cat([_d(w[k]) for k in names]).T
            if not t.lora:
                return y
            ad = adapters[i] if adapters else {k: _d(v) for k, v in w.items() if "lora" in k}
            add, at = [], 0
            for j in range(p.tenants):
                L = sum(a for a, b in zip(lens, tenant_of) if b == j)
                add.append(torch.cat([(x[at:at + L] @ ad["lora_a_" + k][j].T)
                                      @ ad["lora_b_" + k][j].T for k in lora], 1))
                at += L
            return y + torch.cat(add)

        y = project(_norm(x, w["attn_norm"]), ("wq", "wk", "wv"), "qkv").view(n, -1, hd)
        q, k, v = _rope(y[:, :H], pos), _rope(y[:, H:H + Hkv], pos), y[:, H + Hkv:]
        x = x + project(_attend(q, k, v, lens)[0].reshape(n, -1), ("wo",), "o")
        z = _norm(x, w["ffn_norm"])
        gate, up = z @ _d(w["wg"]).T, z @ _d(w["wu"]).T
        act = (torch.nn.functional.gelu(gate, approximate="tanh") if m["glu"]
               else torch.nn.functional.silu(gate))
        x = x + (act * up) @ _d(w["wd"]).T
    return _norm(x, t.bw["final_norm"])


def _pool(rows, lens):
    return torch.stack([r.mean(0) for r in rows.split(lens)])


def _tenant_targets(t, i, targets, width):
    return torch.stack([_d(targets[s["target_off"]:s["target_off"] + width])
                        for s in t.p.place[i]])


def _place_preds(t, ys, like):
    out = torch.zeros_like(like, dtype=torch.float64)
    for i, y in enumerate(ys):
        for s, row in zip(t.p.place[i], y):
            out[s["target_off"]:s["target_off"] + len(row)] = row
    return out


def _mlp(t, pooled, targets, leaves):
    """Every tenant's MLP head: predictions and losses from 64-bit leaves."""
    ys, losses, at = [], [], 0
    for i, h in enumerate(leaves):
        x = pooled[at:at + len(t.p.place[i])]
        at += len(t.p.place[i])
        y = torch.nn.functional.silu(x @ h["w1"].T + h["b1"]) @ h["w2"].T + h["b2"]
        ys.append(y)
        losses.append((y - _tenant_targets(t, i, targets, y.shape[1])).square().mean())
    return ys, torch.stack(losses)


def _query(t, rows, targets, leaves, lens):
    ys, losses, at = [], [], 0
    rows = rows.split(lens)
    for i, h in enumerate(leaves):
        y = []
        for x in rows[at:at + len(t.p.place[i])]:
            p = (h["q"] @ (x @ h["wk"].T).T / math.sqrt(h["q"].shape[1])).softmax(-1)
            y.append((p @ (x @ h["wv"].T)).reshape(-1) @ h["wout"].T + h["bout"])
        at += len(t.p.place[i])
        ys.append(torch.stack(y))
        losses.append((ys[-1] - _tenant_targets(t, i, targets, ys[-1].shape[1])).square().mean())
    return ys, torch.stack(losses)


def _leaf(x):
    return x.detach().double().requires_grad_()


def _grads(loss, leaves):
    """Gradients of `loss` in the layout of `leaves` (dicts and lists)."""
    flat = []

    def walk(v, f):
        if isinstance(v, dict):
            return {k: walk(x, f) for k, x in v.items()}
        if isinstance(v, list):
            return [walk(x, f) for x in v]
        return f(v)

    walk(leaves, flat.append)
    got = iter(torch.autograd.grad(loss, flat))
    return walk(leaves, lambda v: next(got))


def _flow_net(w, i, x, tau, ctx):
    """Tenant i's expert: velocity of the chunk x at time tau, given each
    block's context keys and values."""
    dm, hd = FLOW["d_model"], 64
    half = dm // 2
    a = 1000.0 * tau * 10000.0 ** (-torch.arange(half, device=x.device,
                                                 dtype=torch.float64) / half)
    s = torch.cat([a.sin(), a.cos()])
    phi = w["t2"][i] @ torch.nn.functional.silu(w["t1"][i] @ s + w["tb1"][i]) + w["tb2"][i]
    h = x @ w["w_in"][i].T + w["b_in"][i] + w["pos"][i] + phi
    for b, (kc, vc) in zip(w["blocks"], ctx):
        q, ka, va = (_norm(h) @ b["w_qkv"][i].T).split(dm, 1)
        k, v = (torch.cat(z).view(-1, dm // hd, hd).transpose(0, 1)
                for z in ((kc, ka), (vc, va)))
        q = q.view(-1, dm // hd, hd).transpose(0, 1)
        o = (q @ k.transpose(1, 2) / math.sqrt(hd)).softmax(-1) @ v
        h = h + o.transpose(0, 1).reshape(-1, dm) @ b["w_o"][i].T
        z = _norm(h)
        h = h + (torch.nn.functional.silu(z @ b["wg"][i].T) * (z @ b["wu"][i].T)) @ b["w_d"][i].T
    return _norm(h) @ w["w_out"][i].T + w["b_out"][i]


def _packed(gate, up):
    """The library's layout of a gate/up pair: 128-row blocks in turn."""
    T, F, d = gate.shape
    return torch.stack([gate.view(T, F // 128, 128, d), up.view(T, F // 128, 128, d)],
                       2).reshape(T, 2 * F, d)


def _adam(p, g):
    """A first AdamW step of 1e-4 with decay 0.01: (parameter, first moment)."""
    return p - 1e-4 * (g / (g.abs() + 1e-8) + 0.01 * p), 0.1 * g


def _exact_flow(case, t, lens):
    tenant_of = [i for i, p in enumerate(t.p.place) for _ in p]
    train = case["kind"] == "flow_train"
    blocks = [{k: _leaf(v) for k, v in b.items()} for b in t.fw["blocks"]]
    w = {k: _leaf(v) for k, v in t.fw.items() if k != "blocks"}
    w["blocks"] = blocks
    out, rows = [], t.hidden.split(lens)
    for s, i in enumerate(tenant_of):
        ctx = [(_d(rows[s]) @ b["w_kvc"][i].T).split(FLOW["d_model"], 1) for b in blocks]
        if train:
            tau = _d(t.tau[s])
            out.append(_flow_net(w, i, tau * _d(t.actions[s]) + (1 - tau) * _d(t.noise[s]), tau,
                                 ctx))
            continue
        with torch.no_grad():
            x, k = _d(t.noise[s]), case["steps"]
            for j in range(k):
                x = x + _flow_net(w, i, x, j / k, ctx) / k
            out.append(x)
    out = torch.stack(out)
    if not train:
        return out
    loss = torch.stack([(out - (_d(t.actions) - _d(t.noise)))[
        [s for s, j in enumerate(tenant_of) if j == i]].square().mean()
        for i in range(t.p.tenants)])
    g = _grads(loss.sum(), w)
    order = ("w_qkv", "w_kvc", "w_o", "w_gu", "w_d")
    names = ("w_in", "b_in", "pos", "t1", "tb1", "t2", "tb2", "w_out", "b_out")

    def lib(b):
        return dict(b, w_gu=_packed(b["wg"], b["wu"]))

    gb = [{k: lib(b)[k] for k in order} for b in g["blocks"]]
    pairs = [(w[k], g[k]) for k in names]
    pairs += [(lib(b)[k], x[k]) for b, x in zip(blocks, gb) for k in order]
    return dict(velocity=out.detach(), loss=loss.detach(), grads={k: g[k] for k in names},
                blocks=gb, master=[_adam(p, x)[0].detach() for p, x in pairs])


def _exact_attention(case, t, lens):
    m = t.m
    H, Hkv, hd = m["n_heads"], m["n_kv_heads"], m["head_dim"]
    x = _leaf(t.qkv)
    y = x.view(len(x), -1, hd)
    out, lse = _attend(y[:, :H], y[:, H:H + Hkv], y[:, H + Hkv:], lens)
    out = out.reshape(len(x), -1)
    g, = torch.autograd.grad(out, x, _d(t.dout))
    g = g.view(len(x), -1, hd)
    pos = torch.cat([torch.arange(L, device=x.device) for L in lens])
    g = torch.cat([_rope(g[:, :H + Hkv], pos, -1.0), g[:, H + Hkv:]], 1)
    return dict(out=out.detach(), lse=lse.detach(), dqkv=g.reshape(len(x), -1))


def exact(case, seed):
    kind, lens = case["kind"], _lengths(case)
    if work(case)["flops"] > 1e13:  # minutes in 64 bits
        return None
    t = _tensors(case, seed)
    if kind in ("flow_train", "flow_sample"):
        return _exact_flow(case, t, lens)
    if kind == "attention":
        return _exact_attention(case, t, lens)
    tenant_of = [i for i, p in enumerate(t.p.place) for _ in p]
    if kind in ("step", "infer", "heads_mlp"):
        with torch.no_grad():
            pooled = (_d(t.pooled) if kind == "heads_mlp"
                      else _pool(_backbone(t, lens, tenant_of), lens))
        leaves = [{k: _leaf(v[i]) for k, v in t.hw.items()} for i in range(t.p.tenants)]
        targets = t.targets if kind == "heads_mlp" else t.inp["targets"]
        ys, loss = _mlp(t, pooled, targets, leaves)
        preds = _place_preds(t, [y.detach() for y in ys], targets)
        if kind == "infer":
            return dict(pooled=pooled, preds=preds)
        g = _grads(loss.sum(), leaves)
        if kind == "step":
            return dict(pooled=pooled, preds=preds, loss=loss.detach(), grads=g)
        new = [{k: _adam(leaves[i][k].detach(), g[i][k]) for k in g[i]} for i in range(len(g))]
        return dict(preds=preds, loss=loss.detach(),
                    params={k: torch.stack([x[k][0] for x in new]) for k in t.hw},
                    m=[{k: v[1] for k, v in x.items()} for x in new])
    if kind == "block":
        with torch.no_grad():
            rows = _backbone(t, lens, tenant_of)
            keep, pool = _features(case)
            return dict(pooled=_pool(rows, lens) if pool else None, hidden=rows if keep else None)
    heads = [{k: _leaf(v) for k, v in h.items()} for h in t.hw]
    if kind == "heads_query":
        rows = _leaf(t.hidden)
        ys, loss = _query(t, rows, t.targets, heads, lens)
        g, d = _grads(loss.sum(), [heads, [rows]])
        return dict(preds=_place_preds(t, [y.detach() for y in ys], t.targets),
                    loss=loss.detach(), d_hidden=d[0], grads=g)
    adapters = [{k: _leaf(v) for k, v in w.items() if "lora" in k} for w in t.bw["layers"]]
    rows = _backbone(t, lens, tenant_of, adapters)
    ys, loss = _query(t, rows, t.inp["targets"], heads, lens)
    g, d, a = _grads(loss.sum(), [heads, [rows], adapters])
    return dict(preds=_place_preds(t, [y.detach() for y in ys], t.inp["targets"]),
                loss=loss.detach(), d_hidden=d[0], grads=g,
                lora=[{k.replace("lora_", ""): v for k, v in x.items()} for x in a])
