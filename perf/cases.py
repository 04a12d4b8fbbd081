"""The layer's work as a user has it done, for timing: prefill calls and decode loops through the public entry points.

A prefill case is one hybrid_attn_fwd call on resident tensors, with the outputs and the workspace that a program
keeps from layer to layer.  A decode case is the loop that generates `steps` tokens from a kept prefix, one
hybrid_attn_step per token: it first puts the prefix's token count and linear state back (the copy by which a
program samples several continuations of one prompt), then decodes; everything else the steps write lies behind the
prefix and is written again.  steps = chunk, so every pass contains exactly one routing step.

Fields of a case: kind (prefill | decode), dtype, B, H, Hkv, d, N (prefill length, or prefix of a decode), chunk,
topk, max_salient (0: no salient-cache budget), recipe (distribution of the keys, see synth.py), gate (gate values
given), state (prefill: also builds the decode state), steps (decode).
"""
from __future__ import annotations

import math

import torch

import paper_2602_02180_b200 as still
from paper_2602_02180_b200 import synth


def _case(name, kind, dtype, B, H, Hkv, d, N, chunk, topk, recipe="iid", max_salient=0, gate=False, state=False):
    c = dict(kind=kind, dtype=dtype, B=B, H=H, Hkv=Hkv, d=d, N=N, chunk=chunk, topk=topk, max_salient=max_salient,
             recipe=recipe, gate=gate, state=state, steps=chunk if kind == "decode" else 0)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a single fp32 layer of 512 tokens (correctness work, small models); launches count
        _case("prefill fp32 tiny", "prefill", "fp32", 1, 4, 4, 64, 512, 64, 16),
        # fp32 inference of a layer with 32 heads over a ragged prompt
        _case("prefill fp32 2k", "prefill", "fp32", 1, 32, 8, 64, 2000, 64, 16, "head_scale"),
        # a chat prompt of one user, gated, that fills the decode state; latency counts
        _case("prefill prompt 1k +state", "prefill", "bf16", 1, 32, 8, 128, 1003, 64, 16, "outlier_keys", gate=True, state=True),
        # a batch of ordinary prompts at head dim 64: every token kept, and a quarter of them
        _case("prefill d64 4k all", "prefill", "bf16", 4, 32, 8, 64, 4096, 64, 64, "head_scale"),
        _case("prefill d64 4k quarter", "prefill", "bf16", 4, 32, 8, 64, 4096, 64, 16, "head_scale"),
        # long documents at head dim 128: every token kept (the benchmark's shape), and a quarter of them
        _case("prefill d128 32k all", "prefill", "bf16", 2, 32, 8, 128, 32768, 64, 64, "outlier_keys"),
        _case("prefill d128 32k quarter", "prefill", "bf16", 2, 32, 8, 128, 32768, 64, 16, "outlier_keys"),
        # the longest context, with the salient cache capped at 896 tokens
        _case("prefill d128 128k capped", "prefill", "bf16", 1, 32, 8, 128, 131072, 128, 32, "student_t_keys", max_salient=896),
        # one user's answer after a short conversation: the latency of a step
        _case("decode one user", "decode", "bf16", 1, 32, 8, 128, 2005, 64, 16),
        # a small batch over long prefixes, a quarter of the tokens kept
        _case("decode batch 16 quarter", "decode", "bf16", 16, 32, 8, 128, 16000, 64, 16),
        # a serving batch with a capped salient cache
        _case("decode batch 32 capped", "decode", "bf16", 32, 32, 8, 128, 8192, 64, 16, max_salient=448),
        # the largest decode: 64 sequences with a 32K prefix, every token kept
        _case("decode batch 64 32k all", "decode", "bf16", 64, 32, 8, 128, 32768, 64, 64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Rough cost of a case in seconds: what keeps a drawn case below the largest listed one."""
    w = work(c)
    rate = 20e12 if c["dtype"] == "fp32" else 1e15
    return w["flops"] / rate + w["bytes"] / 3e12 + 1e-5 * max(c["steps"], 1)


def draw(rng):
    while True:
        kind = rng.choice(["prefill", "prefill", "prefill", "decode", "decode"])
        dtype = "fp32" if rng.random() < 0.2 else "bf16"
        d, chunk = rng.choice([64, 128]), rng.choice([64, 64, 128])
        H, Hkv = rng.choice([(4, 4), (16, 4), (32, 8), (32, 8)])
        topk = rng.choice([chunk // 8, chunk // 4, chunk // 4, chunk // 2, chunk])
        recipe = rng.choice(["iid", "head_scale", "outlier_keys", "student_t_keys"])
        budget = topk * rng.choice([4, 14, 28]) if dtype == "bf16" and rng.random() < 0.3 else 0
        if kind == "prefill":
            B = rng.choice([1, 1, 2, 4])
            N = _log_int(rng, 200, 2500 if dtype == "fp32" else 131072 if budget else 32768)
        else:
            B = _log_int(rng, 1, 4 if dtype == "fp32" else 64)
            N = _log_int(rng, 500, 4000 if dtype == "fp32" else 32768)
        if rng.random() < 0.3:
            N = -(-N // chunk) * chunk
        c = _case(None, kind, dtype, B, H, Hkv, d, N, chunk, topk, recipe, budget, gate=rng.random() < 0.3,
                  state=kind == "prefill" and rng.random() < 0.3)
        # below the largest listed prefill / decode, and small enough to prepare three states beside each other
        if _cost(c) <= (0.05 if kind == "decode" else 0.02) and B * H * N * d * 2 <= 4 << 30:
            return c


def _params(c):
    return still.StillParams(c["B"], c["H"], c["Hkv"], c["d"], c["chunk"], c["topk"],
                             torch.float32 if c["dtype"] == "fp32" else torch.bfloat16, max_salient=c["max_salient"])


def _workload(c, seed):
    return synth.Workload("case", c["B"], c["H"], c["Hkv"], c["d"], c["N"], c["chunk"], c["topk"], c["dtype"],
                          c["recipe"], seed)


def _new_tokens(c, p, seed, dev):
    """q, k, v and gate of the decoded tokens, [steps, B, heads, d] each."""
    g = torch.Generator(device=dev)
    g.manual_seed(seed + 5000)
    kw = dict(generator=g, device=dev, dtype=torch.float32)
    n, B, H, Hkv, d = c["steps"], c["B"], c["H"], c["Hkv"], c["d"]
    q = torch.randn(n, B, H, d, **kw).to(p.dtype)
    k = torch.randn(n, B, Hkv, d, **kw).to(p.dtype)
    v = torch.randn(n, B, Hkv, d, **kw).to(p.dtype)
    return q, k, v, torch.rand(n, B, H, d, **kw).to(p.dtype) if c["gate"] else None


def prepare(case, seed):
    dev = "cuda"
    c, p, w = case, _params(case), _workload(case, seed)
    Q, K, V = synth.make_qkv(w, dev)
    Wq, Wk = synth.make_npmap_weights(w, dev)
    s = dict(case=c, p=p, Wq=Wq, Wk=Wk)
    if c["kind"] == "prefill":
        T = -(-c["N"] // c["chunk"])
        s.update(Q=Q, K=K, V=V, G=synth.make_gate(w, dev) if c["gate"] else None, Y=torch.empty_like(Q),
                 scores=torch.empty(c["B"], c["H"], c["N"], dtype=torch.float32, device=dev),
                 sel=torch.empty(c["B"], c["H"], T, c["topk"], dtype=torch.int32, device=dev),
                 workspace=torch.empty(still.workspace_bytes(p, c["N"]), dtype=torch.uint8, device=dev),
                 state=None, cap=0)
        if c["state"]:
            s["cap"] = c["N"] + 1024
            s["state"] = torch.zeros(still.state_bytes(p, s["cap"]), dtype=torch.uint8, device=dev)
            s["lay"] = still.state_layout(p, s["cap"])
        return s
    # decode: the prefix in the state, the new tokens' q, k, v
    s["cap"] = c["N"] + c["steps"]
    s["lay"] = lay = still.state_layout(p, s["cap"])
    s["state"] = torch.zeros(lay["total"], dtype=torch.uint8, device=dev)
    still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk, state=s["state"], state_max_tokens=s["cap"], want_y=False)
    del Q, K, V
    # header words and (S, z) of the prefix: what a pass puts back
    s["kept_header"] = s["state"][:256].clone()
    s["kept_sz"] = s["state"][lay["S"]: lay["scratch"]].clone()
    new = _new_tokens(c, p, seed, dev)
    s["q"], s["k"], s["v"], s["g"] = (None if x is None else x.unbind(0) for x in new)
    n, B, H, d = c["steps"], c["B"], c["H"], c["d"]
    s["y"] = torch.empty(n, B, H, d, dtype=p.dtype, device=dev)
    s["y_step"] = s["y"].unbind(0)
    cap, buf = lay["capacity"], s["state"]
    s["scores"] = buf[lay["score"]: lay["score"] + B * H * cap * 4].view(torch.float32).view(B, H, cap)[:, :, : s["cap"]]
    n_idx = B * H * (cap // c["chunk"]) * c["topk"]
    s["sel"] = buf[lay["sel_idx"]: lay["sel_idx"] + n_idx * 4].view(torch.int32).view(B, H, -1, c["topk"])
    return s


def _linear_state(s):
    """S and z as views of the decode state."""
    c, lay = s["case"], s["lay"]
    n = c["B"] * c["H"] * 2 * c["d"]
    return (s["state"][lay["S"]: lay["S"] + n * c["d"] * 4].view(torch.float32),
            s["state"][lay["z"]: lay["z"] + n * 4].view(torch.float32))


def run(state):
    s = state
    c, p = s["case"], s["p"]
    if c["kind"] == "prefill":
        Y, scores, sel = still.hybrid_attn_fwd(p, s["Q"], s["K"], s["V"], s["Wq"], s["Wk"], G=s["G"], Y=s["Y"],
                                               scores=s["scores"], sel_idx=s["sel"], state=s["state"],
                                               state_max_tokens=s["cap"], workspace=s["workspace"])
        return (Y, scores, sel) + (_linear_state(s) if s["state"] is not None else ())
    buf, lay, N, C = s["state"], s["lay"], c["N"], c["chunk"]
    buf[:256].copy_(s["kept_header"])
    buf[lay["S"]: lay["scratch"]].copy_(s["kept_sz"])
    for i in range(c["steps"]):
        still.hybrid_attn_step(p, buf, s["cap"], N + i, s["q"][i], s["k"][i], s["v"][i], s["Wq"], s["Wk"],
                               g=None if s["g"] is None else s["g"][i], y=s["y_step"][i])
    routed = -(-N // C) - 2   # the chunk routed on the way
    return (s["y"], s["scores"][:, :, N:], s["sel"][:, :, routed]) + _linear_state(s)


def work(case):
    """Operations and bytes of a pass: every input read once and every output written once; a decode step reads the
    rows of the history that some query head of the KV group selected, once for the group, and (S, z)."""
    c = case
    C, lam, d, N = c["chunk"], c["topk"], c["d"], c["N"]
    BH, BHkv, es = c["B"] * c["H"], c["B"] * c["Hkv"], 4 if c["dtype"] == "fp32" else 2
    dp, budget = 2 * d, c["max_salient"]
    la = lam < C or budget > 0
    if c["kind"] == "prefill":
        T = -(-N // C)
        p_sel = C * sum(min(t * lam, budget) if budget else t * lam for t in range(max(T - 1, 0)))
        p_loc = max(T - 1, 0) * C * C + T * C * (C + 1) // 2
        flops = 4 * d * (p_sel + p_loc) * BH + 2 * d * 2 * C * C * T * BH
        by = c["B"] * N * d * es * (2 * c["H"] + 2 * c["Hkv"]) + 4 * BH * N + 4 * BH * T * lam
        if la:
            flops += 2 * d * d * N * (BH + BHkv) + (2 * (C - lam) + 2 * C) * dp * (d + 1) * max(T - 2, 0) * BH
        if c["gate"]:
            by += BH * N * d * es
        if c["state"]:
            by += 2 * BHkv * N * d * es + BH * dp * (d + 1) * 4
        return {"bytes": by, "flops": flops}
    flops = by = 0
    union = 1 - (1 - lam / C) ** (c["H"] // c["Hkv"])
    for t in range(N, N + c["steps"]):
        routed, local = max(t // C - 1, 0), t + 1 - max(t // C - 1, 0) * C
        if budget:
            routed = min(routed, budget // lam)
        by += 2 * BHkv * d * es * (routed * C * union + local) + 2 * BH * d * es
        flops += 4 * BH * d * (routed * lam + local) + 2 * BH * d * C
        if la:
            by += BH * dp * (d + 1) * 4
            flops += BH * (2 * d * d + 2 * dp * (d + 1))
        if la and t % C == 0:
            by += 2 * BHkv * C * d * es + 2 * BH * dp * (d + 1) * 4
            flops += BHkv * 2 * C * d * d + 2 * BH * (C - lam) * dp * (d + 1)
    return {"bytes": by, "flops": flops}


def tolerance(case):
    # Against float64 (own selection on both sides, N up to 8192, every recipe): fp32 Y 3.4e-7, S 6.1e-7, scores
    # 1.8e-7, largest single difference 4.6e-6 of the RMS; bf16 (whose probabilities and features are rounded to
    # bf16) Y 2.2e-3, S 1.6e-3, largest 2.6e-2.  Indices agreed throughout: the gap at a chunk's threshold is 4e-3 in
    # the median and the scores are good to 1e-6, so one chunk in thousands may be decided the other way, which
    # shifts that chunk's ascending indices and moves one token between the branches (in a bf16 call of many chunks
    # up to half the RMS on single values of Y).
    if case["dtype"] == "fp32":
        return {"rel": 5e-6, "max": 5e-5, "differ": 1e-3}
    return {"rel": 8e-3, "max": 0.5, "differ": 1e-3}


def _phi(x, W):
    """Norm-preserved feature map of x [..., n, d] with W [..., d, d_f], in float64."""
    f = x @ W
    u = f * (x.norm(dim=-1, keepdim=True) / f.norm(dim=-1, keepdim=True).clamp_min(1e-12))
    return torch.cat([u.softmax(-1), (-u).softmax(-1)], -1)


def _exact_head_group(c, p, Q, K, V, G, Wq, Wk, row0):
    """One (batch, KV head): Q [rep, N, d], K, V [N, d], G [rep, N - row0, d], Wq [rep, d, d], Wk [d, d] in float64.
    Outputs of the rows from row0 on, scores and selection of all tokens, and the linear state after the last token."""
    C, lam, d, N, dev = c["chunk"], c["topk"], c["d"], K.shape[0], K.device
    rep, T, window = Q.shape[0], -(-N // C), c["max_salient"] // lam
    pad = lambda x: torch.nn.functional.pad(x, (0, 0, 0, T * C - x.shape[-2]))
    Qc, Kc, Vc = pad(Q).view(rep, T, C, d), pad(K).view(T, C, d), pad(V).view(T, C, d)
    # scores: row r of a chunk has the window of columns r+1 .. r+C of (previous chunk, this chunk)
    two = torch.cat([torch.cat([torch.zeros_like(Kc[:1]), Kc[:-1]]), Kc], 1)                 # [T, 2C, d]
    r, j = torch.arange(C, device=dev)[:, None], torch.arange(2 * C, device=dev)[None]
    own = j == r + C
    seen = ((j > r) & (j <= r + C))[None].expand(T, C, 2 * C).clone()
    seen[0] &= j >= C
    scores = torch.empty(rep, T * C, dtype=torch.float64, device=dev)
    for h in range(rep):
        l = (Qc[h] @ two.transpose(1, 2) * p.c().sm_scale).masked_fill(~seen, -math.inf)
        a = l.softmax(-1)
        b = l.masked_fill(own, -math.inf).softmax(-1).nan_to_num(0.0)
        scores[h] = (a * ((a + p.eps) / (b + p.eps)).log()).sum(-1).reshape(-1)
    live = (torch.arange(T * C, device=dev) < N).view(T, C)
    sc = scores.view(rep, T, C).masked_fill(~live, -math.inf)
    order = sc.sort(dim=-1, descending=True, stable=True).indices[..., :lam]
    chosen = torch.zeros(rep, T, C, dtype=torch.bool, device=dev).scatter_(2, order, True) & live
    pos = torch.arange(T * C, device=dev).view(T, C).expand(rep, T, C)
    sel = pos.masked_fill(~chosen, T * C).sort(-1).values[..., :lam]
    sel = sel.masked_fill(sel == T * C, -1).int()
    # linear state chunk by chunk; S, z before chunk t is answered hold the chunks up to t-2
    la = lam < C or window > 0
    S = torch.zeros(rep, 2 * d, d, dtype=torch.float64, device=dev)
    z = torch.zeros(rep, 2 * d, dtype=torch.float64, device=dev)
    Y = torch.empty(rep, N - row0, d, dtype=torch.float64, device=dev)
    for t in range(T):
        if la and t >= 2:
            fold = [(t - 2, ~chosen[:, t - 2])] if lam < C else []
            if window and t - 2 - window >= 0:
                fold.append((t - 2 - window, chosen[:, t - 2 - window]))
            for a, w in fold:
                f = _phi(Kc[a], Wk) * w[..., None]
                S += f.transpose(1, 2) @ Vc[a]
                z += f.sum(1)
        lo, hi = max(t * C, row0), min((t + 1) * C, N)
        if lo >= hi:
            continue
        q = Q[:, lo:hi]
        first = max(t - 1 - window, 0) if window else 0      # routed chunks before it have left the cache
        loc = max(t - 1, 0) * C
        n_c = max(t - 1 - first, 0)
        mask = torch.cat([chosen[:, first: first + n_c].reshape(rep, 1, n_c * C).expand(rep, hi - lo, n_c * C),
                          (torch.arange(loc, hi, device=dev) <= torch.arange(lo, hi, device=dev)[:, None]).expand(rep, -1, -1)], 2)
        k0 = first * C if n_c else loc
        l = (q @ K[k0: hi].T * p.c().sm_scale).masked_fill_(~mask, -math.inf)
        m = l.amax(-1, keepdim=True).clamp_min(0.0 if la else -math.inf)
        e = (l - m).exp()
        num, den = e @ V[k0: hi], e.sum(-1, keepdim=True)
        if la:
            f = _phi(q, Wq)
            n_la = f @ S
            num += (n_la if G is None else n_la * G[:, lo - row0: hi - row0]) * (-m).exp()
            den = den + (f @ z[..., None]) * (-m).exp()
        Y[:, lo - row0: hi - row0] = num / den
    return Y, scores[:, :N], sel, S, z


def exact(case, seed):
    """The outputs of run() in float64 with plain torch.  None where it would take too long."""
    c, p = case, _params(case)
    total = c["N"] + c["steps"]
    visible = min(total, (c["max_salient"] // c["topk"] + 3) * c["chunk"]) if c["max_salient"] else total
    rows = c["steps"] if c["steps"] else c["N"]
    if c["B"] * c["H"] * (rows * visible / 2 + total * c["chunk"] * 4) > 1e11:
        return None
    dev, w = "cuda", _workload(c, seed)
    Q, K, V = synth.make_qkv(w, dev)
    Wq, Wk = synth.make_npmap_weights(w, dev)
    if c["kind"] == "decode":
        *new, G = (None if x is None else x.permute(1, 2, 0, 3) for x in _new_tokens(c, p, seed, dev))
        Q, K, V = (torch.cat([x, n], 2) for x, n in zip((Q, K, V), new))
    else:
        G = synth.make_gate(w, dev) if c["gate"] else None
    rep, out = c["H"] // c["Hkv"], []
    for b in range(c["B"]):
        for kv in range(c["Hkv"]):
            hs = slice(kv * rep, (kv + 1) * rep)
            out.append(_exact_head_group(c, p, Q[b, hs].double(), K[b, kv].double(), V[b, kv].double(),
                                         None if G is None else G[b, hs].double(), Wq[hs].double(), Wk[kv].double(),
                                         c["N"] if c["kind"] == "decode" else 0))
    Y, scores, sel, S, z = (torch.cat(x).unflatten(0, (c["B"], c["H"])) for x in zip(*out))
    if c["kind"] == "decode":
        return (Y.permute(2, 0, 1, 3), scores[:, :, c["N"]:], sel[:, :, -(-c["N"] // c["chunk"]) - 2], S.flatten(), z.flatten())
    return (Y, scores, sel) + ((S.flatten(), z.flatten()) if c["state"] else ())
