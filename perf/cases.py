"""Performance cases of the SMoES router framework: the calls a training or serving program makes
per MoE layer, through the public entry points of ``paper_2604_23996_gb300.binding``.

Kinds of case
  fwd         ``Router.forward_permute``: gate, top-k, Gaussian score, MI loss, bin permutation
  bwd         ``Router.backward`` after a forward: dW and dX of the MI loss (and of the top-k weights)
  step        forward_permute, optionally the bin-level balance loss, then the backward
  attn_score  ``Router.modality_score`` with the attention-accumulated score
  attn_fwd    ``smoes_attention_fwd``: attention with grouped-query heads and the score
  stats       ``smoes_gaussian_stats_update``: one step of the running modality statistics

Router inputs follow the workloads' recipe (x = alpha mu_v + (1 - alpha) mu_t + N(0, I), gate
weights N(0, 0.02^2) plus a lean of each bin towards a modality), with x rounded to multiples of
1/16 and the weights to multiples of 1/1024. Both grids are exact in bf16 and every partial sum of
a gate logit is then exact in fp32, whatever the order of the sum, so the top-k choice and the
permutation are the same whole numbers for every correct implementation of the softmax gate.
"""
import math
import random

import numpy as np
import torch

from paper_2604_23996_gb300 import binding as bd

DEV = "cuda"


# ---------------------------------------------------------------------------------------- cases

def _router(kind, name, T, samples, d, E, k, bins, **opt):
    c = dict(kind=kind, T=T, samples=samples, d=d, E=E, k=k, bins=bins, dtype="bf16", ragged=False,
             gate="softmax", renorm=False, upstream=False, balance=False, shuffled_bins=False)
    c.update(opt)
    if name:
        c["name"] = name
    return c


def _attn(kind, name, B, H, S, kv_heads, soft=False, blend=False, causal=True):
    c = dict(kind=kind, B=B, H=H, S=S, kv_heads=kv_heads, soft=soft, blend=blend, causal=causal)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # serving: one prompt of one image (576 patches) and a short question
        _router("fwd", "serve_one_prompt", 611, 1, 2048, 64, 6, 8),
        # a small fp32 layer trained for one step (the tiny_fp32 workload)
        _router("step", "tiny_step_fp32", 4096, 1, 512, 16, 2, 4, dtype="fp32"),
        # fine-tuning on a small ragged batch: sigmoid gate with a selection bias, adaptive
        # (shuffled) bins, balance loss, the language-model loss arriving through the top-k weights
        _router("step", "ragged_sigmoid_step", 6007, 7, 1416, 48, 5, 6, ragged=True, gate="sigmoid",
                upstream=True, balance=True, shuffled_bins=True),
        # the dsmoe_vlm workload: forward and backward of a DeepSeekMoE-shaped layer
        _router("fwd", "dsmoe_fwd", 16384, 8, 2048, 64, 6, 8),
        _router("bwd", "dsmoe_bwd", 16384, 8, 2048, 64, 6, 8),
        # the small_hidden workload as a training step, with the gradient of the top-k weights
        _router("step", "small_hidden_step", 32768, 16, 1280, 64, 6, 8, upstream=True),
        # the large_fine workload (Qwen3-MoE-shaped layer, 131072 tokens), each direction
        _router("fwd", "large_fwd", 131072, 32, 2048, 128, 8, 16),
        _router("bwd", "large_bwd", 131072, 32, 2048, 128, 8, 16),
        # the attn_router workload's score: 8 sequences, 16 heads, 4096 tokens, hard labels
        _attn("attn_score", "attn_score", 8, 16, 4096, 16),
        # a later layer on shorter odd sequences: carried soft score and the residual blend
        _attn("attn_score", "attn_score_ragged", 4, 16, 1111, 16, soft=True, blend=True),
        # attention forward with the score column, four query heads per key/value head
        _attn("attn_fwd", "attn_fwd", 8, 16, 4096, 4),
        # running statistics of a large batch
        _router("stats", "stats_large", 131072, 32, 2048, 128, 8, 16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fwd", "fwd", "fwd", "bwd", "bwd", "step", "step", "step", "attn_score",
                       "attn_score", "attn_fwd", "stats"])
    if kind.startswith("attn"):
        S = _log_int(rng, 128, 4096)
        if kind == "attn_fwd":
            S = max(128, S // 128 * 128)
        H = rng.choice([8, 16, 32])
        B = max(1, min(_log_int(rng, 1, 16), 8 * 16 * 4096 * 4096 // (H * S * S)))
        kv = rng.choice([1, 2, 4, H]) if kind == "attn_fwd" else H
        soft = rng.random() < 0.5
        return _attn(kind, None, B, H, S, kv, soft=soft, blend=soft and rng.random() < 0.7,
                     causal=rng.random() < 0.85)
    if kind == "step" and rng.random() < 0.25:          # fp32 layers are small
        T = _log_int(rng, 256, 8192)
        E = rng.choice([8, 16, 32, 64])
        bins = rng.choice([2, 4, 8])
        return _router(kind, None, T, max(1, min(T // 64, _log_int(rng, 1, 16))), 8 * _log_int(rng, 16, 128),
                       E, rng.choice([1, 2, 4]), bins, dtype="fp32", ragged=rng.random() < 0.5,
                       upstream=rng.random() < 0.5, renorm=rng.random() < 0.3)
    T = _log_int(rng, 512, 65536 if kind == "step" else 131072)
    d = rng.choice([1024, 1280, 1536, 2048, 8 * _log_int(rng, 64, 256), 8 * _log_int(rng, 64, 256)])
    E, bins = rng.choice([(16, 4), (32, 4), (32, 8), (48, 6), (64, 8), (64, 8), (64, 16), (72, 8), (96, 8),
                          (128, 8), (128, 16), (128, 16)])
    k = rng.choice([2, 4, 6, 8])
    samples = max(1, min(T // 128, _log_int(rng, 1, 64)))
    c = _router(kind, None, T, samples, d, E, k, bins, ragged=rng.random() < 0.5)
    if kind == "step":
        c["gate"] = "sigmoid" if rng.random() < 0.3 else "softmax"
        c["balance"] = rng.random() < 0.4
        c["shuffled_bins"] = rng.random() < 0.2
    if kind in ("step", "bwd"):
        c["upstream"] = rng.random() < 0.5
        c["renorm"] = c["gate"] == "sigmoid" or rng.random() < 0.3
    return c


# --------------------------------------------------------------------------------------- inputs

def _offsets(c):
    """Sample boundaries: equal lengths, or ragged ones that depend on the case alone."""
    T, B = c["T"], c["samples"]
    if not c["ragged"]:
        return np.array([T * i // B for i in range(B + 1)], dtype=np.int32)
    cuts = sorted(random.Random(T * 131 + B).sample(range(1, T), B - 1)) if B > 1 else []
    return np.array([0] + cuts + [T], dtype=np.int32)


def _expert_bin(c):
    eb = np.arange(c["E"]) // (c["E"] // c["bins"])
    if c["shuffled_bins"]:
        random.Random(c["E"]).shuffle(eb)
    return eb.astype(np.int32)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _router_inputs(c, seed):
    g = _gen(seed)
    T, d, E, k = c["T"], c["d"], c["E"], c["k"]
    dt = torch.float32 if c["dtype"] == "fp32" else torch.bfloat16
    offs = _offsets(c)
    # each sample starts with its image tokens (28% of it, as 576 of 2048)
    pos = torch.arange(T, device=DEV)
    start = torch.zeros(T, dtype=torch.int64, device=DEV)
    length = torch.zeros(T, dtype=torch.int64, device=DEV)
    for a, b in zip(offs[:-1].tolist(), offs[1:].tolist()):
        start[a:b] = a
        length[a:b] = b - a
    is_vision = ((pos - start) * 100 < 28 * length).to(torch.uint8)
    means = torch.randn((2, d), generator=g, device=DEV)
    means = 3.0 * means / means.norm(dim=1, keepdim=True)
    # Beta(2, 2) mixing weights: the median of three uniforms
    alpha = torch.rand((T, 3), generator=g, device=DEV).median(dim=1).values[:, None]
    X = torch.empty((T, d), dtype=dt, device=DEV)
    for s in range(0, T, 16384):
        e = min(T, s + 16384)
        x = torch.randn((e - s, d), generator=g, device=DEV)
        x += alpha[s:e] * means[0] + (1.0 - alpha[s:e]) * means[1]
        X[s:e] = (torch.round(x * 16.0).clamp_(-255, 255) / 16.0).to(dt)
    # a gate some way into training: half of the bins lean towards vision, half towards text
    eb = torch.from_numpy(_expert_bin(c)).to(DEV)
    lean = torch.where(eb < c["bins"] // 2, 1.0, -1.0)[:, None] * (means[0] - means[1]) / 3.0
    W = 0.02 * torch.randn((E, d), generator=g, device=DEV) + 0.25 * lean
    W = (torch.round(1024.0 * W) / 1024.0).to(dt)
    # running statistics as a training program has them: moments of earlier tokens
    mu = 0.5 * (means[0] + means[1]) + 0.2 * torch.stack([means[0] - means[1], means[1] - means[0]])
    var = 1.0 + 0.05 * torch.rand((2, d), generator=g, device=DEV)
    out = dict(X=X, W=W, mu=mu.contiguous(), var=var.contiguous(), is_vision=is_vision, offs=offs,
               expert_bin=_expert_bin(c), bias=None, dw=None)
    if c["gate"] == "sigmoid":
        out["bias"] = 0.05 * torch.randn(E, generator=g, device=DEV)
    if c["upstream"]:
        out["dw"] = 1e-3 * torch.randn((T, k), generator=g, device=DEV)
    if c["kind"] == "stats":
        N = torch.tensor([0.28e6, 0.72e6], dtype=torch.float64, device=DEV) * 4.0
        out["N"] = N
        out["S_mu"] = N[:, None] * mu.double()
        out["S_var"] = N[:, None] * var.double()
    return out


def _attn_inputs(c, seed):
    g = _gen(seed)
    B, H, S, kv = c["B"], c["H"], c["S"], c["kv_heads"]

    def bf16(heads):
        return torch.randn((B, heads, S, 128), generator=g, device=DEV).to(torch.bfloat16)

    out = dict(Q=bf16(H), K=bf16(kv))
    if c["kind"] == "attn_fwd":
        out["V"] = bf16(kv)
    vis = (torch.arange(S, device=DEV) < S // 4).to(torch.uint8).repeat(B)
    out["is_vision"] = vis
    out["key_bias"] = 0.5 * vis.float()
    if c["soft"]:
        out["m_prev"] = torch.rand(B * S, generator=g, device=DEV)
    if c["blend"]:
        out["xattn_norm"] = 0.5 + 1.5 * torch.rand(B * S, generator=g, device=DEV)
        out["x_norm"] = 0.5 + 1.5 * torch.rand(B * S, generator=g, device=DEV)
    return out


# ------------------------------------------------------------------------------------ the calls

class State:
    pass


def prepare(case, seed):
    c, s = case, State()
    s.case = c
    if c["kind"].startswith("attn"):
        i = _attn_inputs(c, seed)
        T = c["B"] * c["S"]
        s.router = bd.Router(T, 64, 16, 2, 4, [0, T], np.arange(16) // 4, attn_max_heads=c["H"])
        s.M = torch.empty((T, 2), device=DEV)
        s.attn = dict(Q=i["Q"], K=i["K"], B=c["B"], H=c["H"], S=c["S"], hd=128,
                      sm_scale=1.0 / math.sqrt(128), causal=int(c["causal"]), key_bias=i["key_bias"])
        s.attn["m_prev" if c["soft"] else "is_vision"] = i["m_prev"] if c["soft"] else i["is_vision"]
        if c["blend"]:
            s.attn["xattn_norm"], s.attn["x_norm"] = i["xattn_norm"], i["x_norm"]
        if c["kind"] == "attn_fwd":
            s.V = i["V"]
            s.O = torch.empty_like(i["Q"])
        return s
    i = _router_inputs(c, seed)
    s.i = i
    s.router = r = bd.Router(
        c["T"], c["d"], c["E"], c["k"], c["bins"], i["offs"], i["expert_bin"],
        bd.SMOES_F32 if c["dtype"] == "fp32" else bd.SMOES_BF16, renorm_topk=int(c["renorm"]),
        gate=bd.SMOES_GATE_SIGMOID if c["gate"] == "sigmoid" else bd.SMOES_GATE_SOFTMAX,
        score_bias=i["bias"])
    r.perm_token.zero_()                 # the entries past bin_offsets[-1] are never written
    r.perm_mask.zero_()
    s.loss_bal = torch.zeros(1, device=DEV)
    s.dW = torch.empty((c["E"], c["d"]), device=DEV)
    s.dX = torch.empty_like(i["X"])
    if c["kind"] == "stats":
        s.mu, s.var = torch.empty((2, c["d"]), device=DEV), torch.empty((2, c["d"]), device=DEV)
    if c["kind"] == "bwd":
        r.forward_permute(i["X"], i["W"], mu=i["mu"], var=i["var"], is_vision=i["is_vision"])
    return s


def run(s):
    c, r = s.case, s.router
    kind = c["kind"]
    if kind == "attn_score":
        r.modality_score(bd.SMOES_SCORE_ATTN, s.M, attn=s.attn)
        return {"M": s.M}
    if kind == "attn_fwd":
        code = bd.smoes_attention_fwd(r.plan, s.attn, s.V, c["kv_heads"], s.O, s.M, r.ws)
        assert code == bd.SMOES_OK, code
        return {"M": s.M, "O": s.O}
    i = s.i
    if kind == "stats":
        code = bd.smoes_gaussian_stats_update(r.plan, i["X"], i["is_vision"], 0.99, i["N"], i["S_mu"],
                                              i["S_var"], s.mu, s.var, r.ws)
        assert code == bd.SMOES_OK, code
        return {"N": i["N"], "S_mu": i["S_mu"], "S_var": i["S_var"], "mu": s.mu, "var": s.var}
    out = {}
    if kind in ("fwd", "step"):
        r.forward_permute(i["X"], i["W"], mu=i["mu"], var=i["var"], is_vision=i["is_vision"])
        out.update(topk_idx=r.topk_idx, topk_w=r.topk_w, M=r.M, bin_prob=r.bin_prob, joint=r.joint,
                   mi=r.mi, loss=r.loss, bin_offsets=r.bin_offsets, perm_token=r.perm_token,
                   perm_mask=r.perm_mask, dispatch=r.dispatch, expert_counts=r.expert_counts)
    if c["balance"]:
        code = bd.smoes_bin_balance(r.plan, r.topk_idx, 1e-2, s.loss_bal, r.ws)
        assert code == bd.SMOES_OK, code
        out["loss_bal"] = s.loss_bal
    if kind in ("bwd", "step"):
        r.backward(i["X"], i["W"], r.M, s.dW, dX=s.dX, d_topk_w=i["dw"])
        out.update(dW=s.dW, dX=s.dX)
    return out


def work(case):
    """Bytes and operations a pass cannot do without: every input read once, every output written
    once (X is read by the forward and again by the backward, which a step cannot avoid)."""
    c = case
    kind = c["kind"]
    if kind.startswith("attn"):
        B, H, S, kv = c["B"], c["H"], c["S"], c["kv_heads"]
        pairs = B * H * (S * (S + 1) // 2 if c["causal"] else S * S)
        nbytes = B * S * 128 * 2 * (H + kv) + B * S * (8 + 8)
        flops = 2.0 * 128 * pairs
        if kind == "attn_fwd":
            nbytes += B * S * 128 * 2 * (H + kv)
            flops *= 2.0
        return {"bytes": nbytes, "flops": flops}
    T, d, E, k, K = c["T"], c["d"], c["E"], c["k"], c["bins"]
    b = 4 if c["dtype"] == "fp32" else 2
    if kind == "stats":
        return {"bytes": T * (d * b + 1) + 2 * (2 * 2 * d * 8) + 4 * d * 4, "flops": 4.0 * T * d}
    fwd = T * (d * b + 8 * k + 8 + 4 * K + 1) + E * d * b + 8 * T * min(k, K)
    bwd = T * (2 * d * b + 8 + (8 * k if c["upstream"] else 0)) + E * d * (b + 4)
    return {"bytes": (fwd if kind in ("fwd", "step") else 0) + (bwd if kind in ("bwd", "step") else 0),
            "flops": 2.0 * T * d * E * ({"fwd": 1, "bwd": 2, "step": 3}[kind])}


def tolerance(case):
    kind = case["kind"]
    if kind == "attn_score":
        return {"rel": 1e-5, "max": 1e-3}
    if kind == "attn_fwd":               # bf16 softmax weights and bf16 output
        return {"rel": 1e-2, "max": 0.1}
    if kind == "stats":
        return {"rel": 1e-5, "max": 1e-3}
    if case["gate"] == "sigmoid":
        # sigmoid(z) + bias is not on a grid: near ties may order two experts the other way, and a
        # token with another order takes another gradient (one of 6007 tokens: 1.2e-2 of dW)
        return {"rel": 2.5e-2, "max": 1.0, "differ": 2e-3}
    # the MI rests on M - 1/2 ~ 1e-3, formed from fp32 sums over the features and the tokens
    # (1e-4 off the exact value); dX of a bf16 layer has a bf16 operand and bf16 storage
    rel = 1e-3 if kind == "fwd" or case["dtype"] == "fp32" else 1e-2
    return {"rel": rel, "max": 0.1, "differ": 0.0}


# --------------------------------------------------------------------------- the same in 64 bits

def _exact_gate(c, i):
    """Logits, gate, choice, weights and scores in float64."""
    T, k = c["T"], c["k"]
    Wd = i["W"].double()
    mu, var = i["mu"].double(), i["var"].double()
    z = torch.empty((T, c["E"]), dtype=torch.float64, device=DEV)
    dll = torch.empty(T, dtype=torch.float64, device=DEV)
    for s in range(0, T, 8192):
        x = i["X"][s:s + 8192].double()
        z[s:s + 8192] = x @ Wd.T
        ll = [-0.5 * (torch.log(var[m]) + (x - mu[m]) ** 2 / var[m]).sum(dim=1) for m in range(2)]
        dll[s:s + 8192] = ll[0] - ll[1]
    Mv = torch.sigmoid(dll / (0.5 * c["d"]))
    if c["gate"] == "sigmoid":
        raw = torch.sigmoid(z)
        key = raw + i["bias"].double()
    else:
        raw, key = torch.exp(z - z.max(dim=1, keepdim=True).values), z
    g = raw / raw.sum(dim=1, keepdim=True)
    idx = torch.sort(key, dim=1, descending=True, stable=True).indices[:, :k]
    w = torch.gather(g, 1, idx)
    if c["renorm"] or c["gate"] == "sigmoid":
        w = w / w.sum(dim=1, keepdim=True)
    return dict(z=z, raw=raw, g=g, idx=idx, w=w, dev=0.5 * torch.tanh(dll / c["d"]), Mv=Mv)


def _exact_mi(c, i, q):
    """Bin sums, per-sample joint table, mutual information and its derivative at the gate values.
    The deviations of the two rows from independence are formed from centred sums."""
    T, K, offs = c["T"], c["bins"], i["offs"]
    NB = c["E"] // K
    onehot = torch.zeros((c["E"], K), dtype=torch.float64, device=DEV)
    onehot[torch.arange(c["E"]), torch.from_numpy(i["expert_bin"].astype(np.int64))] = 1.0
    p = q["g"] @ onehot
    B = len(offs) - 1
    joint = torch.empty((B, 2, K), dtype=torch.float64, device=DEV)
    mi = torch.empty(B, dtype=torch.float64, device=DEV)
    u = torch.empty((T, K), dtype=torch.float64, device=DEV)
    for s in range(B):
        a, b = int(offs[s]), int(offs[s + 1])
        n, pk, dv = b - a, p[a:b], q["dev"][a:b]
        Q = pk.sum(dim=0)
        qk = Q / Q.sum()
        A, eps, sm = [], [], []
        for sign in (1.0, -1.0):
            d = sign * dv
            A.append(0.5 * n + d.sum())
            eps.append(((d - d.mean())[:, None] * pk).sum(dim=0) / A[-1] * n / Q)
            sm.append((qk * eps[-1]).sum())
        nbz = 2.0 + sm[0] + sm[1]
        lk, lz = torch.log1p(0.5 * (eps[0] + eps[1])), torch.log1p(0.5 * (sm[0] + sm[1]))
        P = [qk * (1.0 + e) / nbz for e in eps]
        L = [torch.log1p(eps[m]) - lk + lz - torch.log1p(sm[m]) for m in range(2)]
        I = (P[0] * L[0] + P[1] * L[1]).sum()
        joint[s, 0], joint[s, 1], mi[s] = P[0], P[1], I
        co = [(L[m] - I) / (nbz * A[m]) for m in range(2)]
        u[a:b] = (0.5 + dv)[:, None] * co[0] + (0.5 - dv)[:, None] * co[1]
    return p, joint, mi, u @ onehot.T


def _exact_balance(c, i, q, scale):
    """Bin-level balance loss and its derivative at the gate values (selection shares constant)."""
    T, E, K = c["T"], c["E"], c["bins"]
    eb = torch.from_numpy(i["expert_bin"].astype(np.int64)).to(DEV)
    sel = torch.zeros((T, E), dtype=torch.float64, device=DEV).scatter_(1, q["idx"], 1.0)
    dg = torch.zeros_like(q["g"])
    loss = torch.zeros((), dtype=torch.float64, device=DEV)
    for k in range(K):
        m = (eb == k).nonzero()[:, 0]
        chosen = sel[:, m]
        used = (chosen.sum(dim=1) > 0).double()
        if float(used.sum()) == 0:
            continue
        f = chosen.sum(dim=0) / chosen.sum()
        G = q["g"][:, m].sum(dim=1, keepdim=True)
        h = q["g"][:, m] / G
        loss += (E // K) * (f * (h * used[:, None]).sum(dim=0) / used.sum()).sum()
        dg[:, m] = scale * (E // K) / used.sum() * used[:, None] * (f - (f * h).sum(dim=1, keepdim=True)) / G
    return loss, dg


def _exact_router(c, i):
    q = _exact_gate(c, i)
    p, joint, mi, u = _exact_mi(c, i, q)
    out = {}
    if c["kind"] in ("fwd", "step"):
        out.update(topk_idx=None, topk_w=q["w"], M=torch.stack([q["Mv"], 1.0 - q["Mv"]], dim=1),
                   bin_prob=p, joint=joint, mi=mi, loss=-mi.mean().reshape(1))
    dg = -u / c["samples"]
    if c["balance"]:
        loss, more = _exact_balance(c, i, q, 1e-2)
        out["loss_bal"] = loss.reshape(1)
        dg = dg + more
    if c["kind"] == "fwd":
        return out
    g, idx = q["g"], q["idx"]
    sigmoid = c["gate"] == "sigmoid"
    fac = 1.0 - q["raw"] if sigmoid else 1.0
    dz = g * fac * (dg - (g * dg).sum(dim=1, keepdim=True))
    if c["upstream"]:
        gs, dw = torch.gather(g, 1, idx), i["dw"].double()
        if c["renorm"] or sigmoid:
            dw = (dw - (dw * q["w"]).sum(dim=1, keepdim=True)) / gs.sum(dim=1, keepdim=True)
        at = torch.zeros_like(g).scatter_(1, idx, dw)
        # the renormalised weights do not change with the common factor of the gate, so the term
        # through the softmax's (or the sigmoids') own sum is zero there
        dz = dz + g * fac * (at - (0.0 if sigmoid else (gs * dw).sum(dim=1, keepdim=True)))
    Wd = i["W"].double()
    dW = torch.zeros((c["E"], c["d"]), dtype=torch.float64, device=DEV)
    dX = torch.empty((c["T"], c["d"]), dtype=torch.float32, device=DEV) if c["T"] * c["d"] > 1 << 26 else \
        torch.empty((c["T"], c["d"]), dtype=torch.float64, device=DEV)
    for s in range(0, c["T"], 8192):
        dW += dz[s:s + 8192].T @ i["X"][s:s + 8192].double()
        dX[s:s + 8192] = (dz[s:s + 8192] @ Wd).to(dX.dtype)
    out.update(dW=dW, dX=dX)
    return out


def _exact_attn(c, i):
    B, H, S, kv = c["B"], c["H"], c["S"], c["kv_heads"]
    m = (i["m_prev"] if c["soft"] else i["is_vision"]).double().reshape(B, S)
    bias = i["key_bias"].double().reshape(B, S)
    fwd = c["kind"] == "attn_fwd"
    O = torch.empty((B, H, S, 128), dtype=torch.float64, device=DEV) if fwd else None
    mass = torch.zeros((B, S), dtype=torch.float64, device=DEV)
    later = torch.ones((S, S), dtype=torch.bool, device=DEV).triu(1) if c["causal"] else None
    for b in range(B):
        for h in range(H):
            hk = h // (H // kv)
            a = i["Q"][b, h].double() @ i["K"][b, hk].double().T / math.sqrt(128) + bias[b]
            if later is not None:
                a.masked_fill_(later, -math.inf)
            a = torch.softmax(a, dim=1)
            mass[b] += a @ m[b] / H
            if fwd:
                O[b, h] = a @ i["V"][b, hk].double()
    mv = mass.reshape(-1)
    if c["blend"]:
        an, xn = i["xattn_norm"].double(), i["x_norm"].double()
        mv = (an * mv + xn * m.reshape(-1)) / (an + xn)
    out = {"M": torch.stack([mv, 1.0 - mv], dim=1)}
    if fwd:
        out["O"] = O
    return out


def _exact_stats(c, i):
    beta = 0.99
    N0, S_mu, S_var = i["N"], i["S_mu"].clone(), i["S_var"].clone()
    N = torch.empty_like(N0)
    for m in range(2):
        rows = (i["is_vision"] == 1 - m).nonzero()[:, 0]
        n = float(len(rows))
        chunks = rows.split(8192)
        mean = sum(i["X"][r].double().sum(dim=0) for r in chunks) / n
        m2 = sum(((i["X"][r].double() - mean) ** 2).sum(dim=0) for r in chunks)
        n0 = float(N0[m])
        shift = (mean - S_mu[m] / n0) ** 2 * (beta * n0 * n / (beta * n0 + n))
        S_var[m] = beta * S_var[m] + m2 + shift
        S_mu[m] = beta * S_mu[m] + n * mean
        N[m] = beta * n0 + n
    return {"N": N, "S_mu": S_mu, "S_var": S_var, "mu": S_mu / N[:, None], "var": S_var / N[:, None]}


def exact(case, seed):
    c = case
    if c["kind"].startswith("attn"):
        return _exact_attn(c, _attn_inputs(c, seed))
    i = _router_inputs(c, seed)
    return _exact_stats(c, i) if c["kind"] == "stats" else _exact_router(c, i)
