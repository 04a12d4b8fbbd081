"""Parity of the CUDA decode step (still_hybrid_attn_step) with the CPU oracle, and
prefill -> decode consistency."""
import numpy as np
import pytest
import torch

import paper_2602_02180_b200 as still
from oracle import still_oracle as oracle
from paper_2602_02180_b200 import synth
from tests import util_parity as U

pytestmark = pytest.mark.gpu


def _decode_case(w, n0, n_steps, gate=False, tweak=None, expect_ties=False, n_heads=4, want_y=True, max_salient=0):
    """Prefill n0 tokens into a state, decode n_steps more, compare every decoded row of the sampled heads
    with the oracle's chunk-wise form over the whole sequence (the GPU's selection forced)."""
    dev = "cuda"
    N = n0 + n_steps
    wN = w.with_(N=N)
    Q, K, V = synth.make_qkv(wN, dev)
    if tweak is not None:
        Q, K, V = tweak(Q, K, V)
    Wq, Wk = synth.make_npmap_weights(wN, dev)
    G = synth.make_gate(wN, dev) if gate else None
    rep = w.H // w.Hkv
    heads = U.sample_heads(w, n_heads)
    # what the oracle needs of the sampled heads, and the decode steps' inputs; the whole-sequence device
    # tensors go before the prefill allocates its workspace (the full-size case would not fit otherwise)
    host = {(b, h): (U.f64(Q[b, h]), U.f64(K[b, h // rep]), U.f64(V[b, h // rep]),
                     None if G is None else U.f64(G[b, h])) for b, h in heads}
    step_in = [t[:, :, n0:].permute(2, 0, 1, 3).contiguous() if t is not None else None for t in (Q, K, V, G)]  # [steps,B,heads,d]
    pre = [t[:, :, :n0].contiguous() if t is not None else None for t in (Q, K, V, G)]
    del Q, K, V, G
    p = U.params_of(w, max_salient=max_salient)
    cap = N + 5
    lay = still.state_layout(p, cap)
    state = torch.zeros(lay["total"], dtype=torch.uint8, device=dev)
    if n0 > 0:
        still.hybrid_attn_fwd(p, pre[0], pre[1], pre[2], Wq, Wk, G=pre[3], state=state, state_max_tokens=cap,
                              want_y=want_y)
    else:
        # an empty prefill initialises the state
        c = p.c()
        import ctypes
        rc = still.binding.lib().still_hybrid_attn_fwd(
            ctypes.byref(c), 0, None, None, None, None, None, None, None, None, None, None, None,
            ctypes.c_void_p(state.data_ptr()), cap, None, 0, None)
        assert rc == 0
    torch.cuda.synchronize()
    del pre
    torch.cuda.empty_cache()
    ys = []
    for i in range(n_steps):
        y = still.hybrid_attn_step(p, state, cap, n0 + i, step_in[0][i], step_in[1][i], step_in[2][i], Wq, Wk,
                                   g=None if step_in[3] is None else step_in[3][i])
        ys.append(y)
    torch.cuda.synchronize()
    assert still.device_status(state) == (0, 0)
    Yd = torch.stack(ys, dim=2)  # [B,H,n_steps,d]
    C, lam = w.C, w.k
    capT = lay["capacity"] // C
    sc = state[lay["score"]: lay["score"] + w.B * w.H * lay["capacity"] * 4].view(torch.float32).view(w.B, w.H, -1)
    n_routed = max(0, (N - 1) // C - 1)  # chunks 0..c_last-2 have been routed
    sel = None
    if lam > 0:
        sel = state[lay["sel_idx"]: lay["sel_idx"] + w.B * w.H * capT * lam * 4].view(torch.int32).view(w.B, w.H, capT, lam)
    rows = list(range(n0, N))
    hp = oracle.HeadParams(C, lam, w.sm_scale, max_salient=max_salient)
    tie_seen = False
    worst = 0.0
    for b, h in heads:
        kv = h // rep
        q64, k64, v64, g64 = host[(b, h)]
        scores = sc[b, h, :N].cpu().numpy().astype(np.float64)
        if expect_ties and n_routed > 0:
            ch = np.sort(scores[: n_routed * C].reshape(n_routed, C)[n0 // C:], axis=1)   # chunks routed by decode steps
            tie_seen |= bool(np.any(np.diff(ch, axis=1) == 0))
        forced = None
        if lam > 0:
            want = oracle.select(scores, C, lam)
            got = sel[b, h, :n_routed].cpu().numpy()
            np.testing.assert_array_equal(got, want[:n_routed])  # bit-exact on the GPU's own scores
            forced = want.copy()
            forced[:n_routed] = got
        out = oracle.chunkwise(q64, k64, v64, U.f64(Wq[h]), U.f64(Wk[kv]), hp, g=g64, forced_idx=forced, rows=rows)
        serr = np.abs(scores - out["score"]).max()
        assert serr <= U.SCORE_TOL[w.torch_dtype], f"b={b} h={h} score max-abs {serr:.3e}"
        err = np.abs(U.f64(Yd[b, h]) - out["y"]).max()
        worst = max(worst, err)
        assert err <= U.TOL[w.torch_dtype], f"b={b} h={h} max-abs {err:.3e}"
    assert tie_seen or not expect_ties, "the constructed input produced no tie in a chunk routed by a decode step"
    return worst


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize(
    "B,H,Hkv,d,C,k,n0,steps",
    [
        (2, 4, 2, 64, 32, 8, 100, 80),     # prefill ends mid-chunk, several routings during decode
        (1, 4, 1, 128, 64, 16, 192, 70),   # prefill ends on a chunk boundary
        (1, 2, 2, 64, 32, 0, 70, 40),      # lambda = 0
        (1, 8, 2, 128, 64, 64, 130, 66),   # lambda = C
        (1, 2, 1, 64, 32, 8, 0, 100),      # decode from an empty state
        (1, 2, 2, 128, 128, 32, 300, 90),
        (1, 16, 1, 64, 32, 8, 90, 50),     # sixteen query heads on one KV head
        (1, 12, 2, 128, 64, 16, 200, 70),  # six heads per group
        (1, 2, 1, 128, 64, 16, 64 * 36 + 5, 70),   # long prefill on few heads: the state comes out of a segmented scan
    ],
)
def test_decode_matches_oracle(dtype, B, H, Hkv, d, C, k, n0, steps):
    w = synth.Workload("t", B, H, Hkv, d, n0, C, k, dtype, "iid", 999)
    _decode_case(w, n0, steps, gate=(k not in (0, C)))


@pytest.mark.parametrize("B,H,Hkv,d,C,k,budget,n0,steps", [
    (1, 4, 2, 128, 64, 16, 48, 64 * 7 + 11, 64 * 3 + 9),     # prefill already past the budget, three routings while decoding
    (2, 2, 1, 64, 64, 8, 16, 72, 64 * 7),                    # the budget is reached during the decode
    (1, 2, 2, 128, 64, 64, 128, 64 * 5, 64 * 2 + 5),         # every token selected: sliding window + linear state
    (1, 2, 1, 64, 64, 8, 8, 0, 64 * 6),                      # from an empty state
])
def test_decode_with_a_salient_cache_budget(B, H, Hkv, d, C, k, budget, n0, steps):
    # Tokens that a newly routed chunk pushes out of the capped salient cache are folded into (S, z) at that step,
    # and the split-KV pass reads only the chunks still cached.
    w = synth.Workload("t", B, H, Hkv, d, n0, C, k, "bf16", "iid", 4711)
    _decode_case(w, n0, steps, gate=True, max_salient=budget)


def test_budgeted_state_size_does_not_grow_with_the_sequence():
    # with a budget the K / V store of the state is a ring over the cached chunks, the local region and the chunk
    # being routed; what still grows with the capacity are 4-byte scores and the per-chunk index tables
    free = still.StillParams(8, 32, 8, 128, 64, 16)
    capped = still.StillParams(8, 32, 8, 128, 64, 16, max_salient=448)
    small, big = still.state_bytes(capped, 4096), still.state_bytes(capped, 65536)
    assert still.state_bytes(free, 65536) > 12 * still.state_bytes(free, 4096) > 0
    kv_ring = 8 * 8 * (448 // 16 + 3) * 64 * 128 * 2 * 2
    assert big - small < 0.1 * still.state_bytes(free, 65536) and small > kv_ring and big < 3 * small


@pytest.mark.parametrize("k", [64, 16])
def test_decode_with_growing_logits(k):
    # Logits that grow by ~7 nats per 128 tokens and one dominant key: the partial results of the key splits
    # differ by many orders of magnitude and the merge has to bring them to one reference.
    def tweak(Q, K, V):
        t = torch.arange(Q.shape[2], device=Q.device)
        Q, K = Q.float(), K.float()
        Q[..., 0] += 8.0
        K[..., 0] += (10.0 * (t // 128)).view(1, 1, -1)
        K[:, :, 128 * 3 + 100, 0] += 60.0
        return Q.to(torch.bfloat16), K.to(torch.bfloat16), V

    w = synth.Workload("t", 2, 4, 2, 128, 0, 64, k, "bf16", "iid", 77)
    _decode_case(w, 128 * 5 + 9, 70, tweak=tweak)


@pytest.mark.parametrize("dtype,C,k", [("bf16", 64, 16), ("bf16", 32, 8), ("fp32", 32, 8)])
@pytest.mark.parametrize("case", ["zero_queries", "periodic_tokens"])
def test_decode_routing_breaks_ties_like_the_oracle(dtype, C, k, case):
    # Equal scores inside a chunk (all logits zero, or tokens repeating with period 16): the chunk routed at a
    # decode step must be ranked under (score descending, position ascending), as the prefill does.
    def tweak(Q, K, V):
        if case == "zero_queries":
            return torch.zeros_like(Q), K, V
        reps = -(-Q.shape[2] // 16)
        rep = lambda x: x[:, :, :16].repeat(1, 1, reps, 1)[:, :, : x.shape[2]].contiguous()  # noqa: E731
        return rep(Q), rep(K), V

    w = synth.Workload("t", 1, 4, 2, 64, 0, C, k, dtype, "iid", 31)
    _decode_case(w, C + 7, 4 * C + 3, tweak=tweak, expect_ties=True)


@pytest.mark.parametrize("k,steps", [(64, 256), (16, 136)])
def test_c5_full_size_sampled(k, steps):
    # The decode workload as benchmarked: batch 64, 32768-token prefix summarised by the prefill into the
    # decode state, then the benchmark's 256 steps (four chunks are routed on the way) with every token
    # selected, and 136 steps (two routings) of the lambda = C/4 companion; sampled (batch, head) pairs
    # against the oracle.
    w = synth.WORKLOADS["c5"].with_(k=k)
    _decode_case(w, w.N, steps, n_heads=4 if k == 64 else 3, want_y=False)


@pytest.mark.parametrize("dtype,B,H,Hkv,d,C,k,n0,steps", [
    ("bf16", 40, 16, 4, 64, 32, 8, 70, 40),     # 640 read-outs: a warp each
    ("bf16", 12, 16, 2, 128, 64, 16, 130, 70),  # 192 read-outs: two warps each; blocks span several groups
    ("bf16", 1, 1, 1, 64, 32, 8, 2100, 40),     # one group, cut into as many partials as the scratch holds
    ("fp32", 2, 20, 2, 64, 32, 8, 70, 40),      # ten heads per group: units of four, four and two
    ("fp32", 1, 1, 1, 128, 64, 16, 1500, 70),
])
def test_decode_splits(dtype, B, H, Hkv, d, C, k, n0, steps):
    _decode_case(synth.Workload("t", B, H, Hkv, d, n0, C, k, dtype, "iid", 1234), n0, steps, gate=True)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("d,df,C,k,budget", [(64, 32, 32, 8, 0), (128, 32, 128, 16, 0), (128, 64, 64, 16, 32), (128, 128, 32, 4, 0)])
def test_decode_feature_sizes_and_bias(dtype, d, df, C, k, budget):
    # narrower maps than the head and a bias, through routing and read-out
    if dtype == "fp32":
        budget = 0
    B, H, Hkv, n0, steps = 1, 4, 2, 2 * C + 5, 2 * C
    w = synth.Workload("t", B, H, Hkv, d, n0 + steps, C, k, dtype, "iid", 8)
    Q, K, V = synth.make_qkv(w, "cuda")
    g = torch.Generator(device="cuda").manual_seed(9)
    mk = lambda *s: (torch.randn(*s, generator=g, device="cuda") * 0.05).to(w.torch_dtype)  # noqa: E731
    Wq, Wk, bq, bk = mk(H, d, df), mk(Hkv, d, df), mk(H, df), mk(Hkv, df)
    p = still.StillParams(B, H, Hkv, d, C, k, w.torch_dtype, d_f=df, sm_scale=w.sm_scale, max_salient=budget)
    cap, lay = w.N, still.state_layout(p, w.N)
    state = torch.zeros(lay["total"], dtype=torch.uint8, device="cuda")
    cut = lambda x: x[:, :, :n0].contiguous()  # noqa: E731
    still.hybrid_attn_fwd(p, cut(Q), cut(K), cut(V), Wq, Wk, bq=bq, bk=bk, state=state, state_max_tokens=cap)
    Y = torch.stack([still.hybrid_attn_step(p, state, cap, t, *(x[:, :, t].contiguous() for x in (Q, K, V)), Wq, Wk, bq=bq, bk=bk)
                     for t in range(n0, w.N)], 2)
    scores = state[lay["score"]: lay["score"] + B * H * lay["capacity"] * 4].view(torch.float32).view(B, H, -1)[:, :, : w.N]
    hp = oracle.HeadParams(C, k, w.sm_scale, max_salient=budget)
    for h in range(H):
        forced = oracle.select(scores[0, h].cpu().numpy().astype(np.float64), C, k)
        out = oracle.chunkwise(U.f64(Q[0, h]), U.f64(K[0, h // 2]), U.f64(V[0, h // 2]), U.f64(Wq[h]), U.f64(Wk[h // 2]), hp,
                               bq=U.f64(bq[h]), bk=U.f64(bk[h // 2]), forced_idx=forced, rows=list(range(n0, w.N)))
        assert np.abs(U.f64(Y[0, h]) - out["y"]).max() <= U.TOL[w.torch_dtype]


def test_state_full_and_mismatch():
    w = synth.Workload("t", 1, 2, 2, 64, 64, 32, 8, "bf16", "iid", 5)
    p = U.params_of(w)
    Q, K, V = synth.make_qkv(w, "cuda")
    Wq, Wk = synth.make_npmap_weights(w, "cuda")
    state = torch.zeros(still.state_bytes(p, 64), dtype=torch.uint8, device="cuda")
    still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk, state=state, state_max_tokens=64)
    q, k, v = synth.make_decode_inputs(w, 0, "cuda")
    with pytest.raises(still.StillError) as e:
        still.hybrid_attn_step(p, state, 64, 64, q, k, v, Wq, Wk)
    assert e.value.code == -4
    # a wrong t_pos is recorded in the state's status word; the step writes nothing else (state bytes and y
    # unchanged), the context stays usable, and later steps on that state are no-ops until it is rebuilt
    state2 = torch.zeros(still.state_bytes(p, 128), dtype=torch.uint8, device="cuda")
    still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk, state=state2, state_max_tokens=128)
    before = state2.clone()
    y = torch.full((w.B, w.H, w.d), 7.0, dtype=w.torch_dtype, device="cuda")
    still.hybrid_attn_step(p, state2, 128, 70, q, k, v, Wq, Wk, y=y)
    assert still.device_status(state2) == (-7, 1)
    still.hybrid_attn_step(p, state2, 128, 64, q, k, v, Wq, Wk, y=y)   # the right position, but the state is flagged
    assert still.device_status(state2) == (-7, 1)
    same = state2 == before
    same[14 * 4: 16 * 4] = True    # the status and detail words
    assert bool(same.all()) and bool((y == 7.0).all())
    # a state built with other parameters (another topk): detail 3
    p_other = U.params_of(w.with_(k=4))
    state3 = torch.zeros(still.state_bytes(p, 128), dtype=torch.uint8, device="cuda")
    still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk, state=state3, state_max_tokens=128)
    if still.state_bytes(p_other, 128) <= state3.numel():
        still.hybrid_attn_step(p_other, state3, 128, 64, q, k, v, Wq, Wk, y=y)
        assert still.device_status(state3) == (-7, 3)
    # and the ordinary path still works
    still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk, state=state2, state_max_tokens=128)
    still.hybrid_attn_step(p, state2, 128, 64, q, k, v, Wq, Wk, y=y)
    assert still.device_status(state2) == (0, 0) and torch.isfinite(y.float()).all()


def _dense_steps(B, Hkv, rep, d, n0, steps, edit=None):
    """Decode with every token selected (softmax attention alone, bf16) beside float64: (y, exact), [B, H, steps, d]."""
    H, C, N = Hkv * rep, 64, n0 + steps
    w = synth.Workload("t", B, H, Hkv, d, N, C, C, "bf16", "iid", 55)
    Q, K, V = synth.make_qkv(w, "cuda")
    if edit is not None:
        edit(Q, K, V)
    p = U.params_of(w)
    state = torch.zeros(still.state_bytes(p, N), dtype=torch.uint8, device="cuda")
    cut = lambda x: x[:, :, :n0].contiguous()  # noqa: E731
    still.hybrid_attn_fwd(p, cut(Q), cut(K), cut(V), state=state, state_max_tokens=N, want_y=False)
    y = torch.stack([still.hybrid_attn_step(p, state, N, t, *(x[:, :, t].contiguous() for x in (Q, K, V))) for t in range(n0, N)], 2)
    K, V = (x.double().repeat_interleave(rep, 1) for x in (K, V))
    seen = torch.arange(N, device="cuda") <= torch.arange(n0, N, device="cuda")[:, None]
    e = (Q[:, :, n0:].double() @ K.transpose(2, 3) * w.sm_scale).masked_fill(~seen, -torch.inf).softmax(-1)
    return y, e @ V, e


@pytest.mark.parametrize("d,rep", [(64, 1), (128, 3), (128, 4), (64, 5), (128, 8), (128, 9), (64, 16), (128, 16)])
def test_decode_outputs_are_float64_rounded_once(d, rep):
    # Weights rounded to bf16 (2^-9) would change about a quarter of the outputs' last bits; kept to 2^-17 they change an
    # output of the size of its terms in 2 x 2^-17 / 2^-8 = 0.4 % of the cases, the smaller ones (cancellation) in more.
    y, exact, _ = _dense_steps(2, 2, rep, d, 700, 20)
    differ = (y != exact.to(torch.bfloat16)).double().mean().item()
    assert differ <= 0.02, differ


@pytest.mark.parametrize("rep", [4, 8])
def test_decode_with_an_infinite_value(rep):
    # an infinite value under a weight that bf16 holds exactly (the maximum's, 1) and under others
    def edit(Q, K, V):
        V[:, :, 100, 3] = torch.inf
        V[:, :, 650, 7] = -torch.inf
        K[:, :, 650] = 0
        K[:, :, 650, 0] = 60.0
        Q[:, :, :, 0] = 4.0

    y, exact, _ = _dense_steps(1, 2, rep, 64, 700, 5, edit)
    assert torch.equal(y[..., 3], exact[..., 3].to(torch.bfloat16)) and bool((y[..., 3] == torch.inf).all())
    assert bool((y[..., 7] == -torch.inf).all())
    rest = [c for c in range(64) if c not in (3, 7)]
    assert bool(torch.isfinite(y[..., rest]).all())


@pytest.mark.parametrize("d", [64, 128])
def test_state_after_many_routings_is_rounded_to_nearest(d):
    # With zero maps every feature is 1 / d_f, exactly: S is then a sum of values that fp32 cannot hold exactly (large and
    # small positive ones), and its error is what the additions leave.  A routing adds a chunk's sum (error below two units
    # of the chunk's sum per product of sixteen tokens) to S, rounded to nearest: half a unit of S each.
    C, n0, routings = 64, 130, 24
    N = n0 + C * routings
    p = still.StillParams(1, 2, 1, d, C, 0, torch.bfloat16)
    g = torch.Generator(device="cuda").manual_seed(3)
    V = 1 + torch.rand(1, 1, N, d, generator=g, device="cuda")
    V[:, :, 1::2] *= 2.0 ** -12
    V = V.to(torch.bfloat16)
    Q, K = (torch.randn(1, h, N, d, generator=g, device="cuda").to(torch.bfloat16) for h in (2, 1))
    W = torch.zeros(2, d, d, dtype=torch.bfloat16, device="cuda")
    lay = still.state_layout(p, N)
    state = torch.zeros(lay["total"], dtype=torch.uint8, device="cuda")
    cut = lambda x: x[:, :, :n0].contiguous()  # noqa: E731
    still.hybrid_attn_fwd(p, cut(Q), cut(K), cut(V), W, W[:1], state=state, state_max_tokens=N, want_y=False)
    for t in range(n0, N):
        still.hybrid_attn_step(p, state, N, t, *(x[:, :, t].contiguous() for x in (Q, K, V)), W, W[:1])
    done = ((N - 1) // C - 1) * C                  # tokens that have left the local region
    S = state[lay["S"]: lay["S"] + 2 * 2 * d * d * 4].view(torch.float32).view(2, 2 * d, d).double()
    z = state[lay["z"]: lay["z"] + 2 * 2 * d * 4].view(torch.float32)
    assert bool((z == done / d).all())
    want = V[0, 0, :done].double().sum(0) / d      # every feature's row
    ulp = 2.0 ** (torch.floor(torch.log2(want)) - 23)
    chunk_ulp = 2.0 ** -23 * 2.0 ** torch.ceil(torch.log2(want / (done // C)))
    bound = routings * (0.5 * ulp + 4 * 2 * chunk_ulp)
    assert bool(((S - want).abs() <= bound).all()), ((S - want).abs() / ulp).max().item()


@pytest.mark.parametrize("dtype,n_nan", [("bf16", 16), ("fp32", 8)])
def test_decode_nan_logits_make_the_output_nan(dtype, n_nan):
    # a run of NaN keys as long as a tile of the pass: the tile's maximum is then no number, and the first of a warp's
    # tiles has no earlier one; the outputs of the group are NaN, those of the other group are not
    B, Hkv, rep, d, n0, steps, C = 1, 2, 4, 64, 700, 3, 64
    w = synth.Workload("t", B, Hkv * rep, Hkv, d, n0 + steps, C, C, dtype, "iid", 56)
    Q, K, V = synth.make_qkv(w, "cuda")
    K[:, 0, :n_nan] = torch.nan
    p = U.params_of(w)
    state = torch.zeros(still.state_bytes(p, w.N), dtype=torch.uint8, device="cuda")
    cut = lambda x: x[:, :, :n0].contiguous()  # noqa: E731
    still.hybrid_attn_fwd(p, cut(Q), cut(K), cut(V), state=state, state_max_tokens=w.N, want_y=False)
    for t in range(n0, w.N):
        y = still.hybrid_attn_step(p, state, w.N, t, *(x[:, :, t].contiguous() for x in (Q, K, V)))
        assert bool(torch.isnan(y[:, :rep]).all()) and bool(torch.isfinite(y[:, rep:]).all())


def test_decode_with_the_most_partials_a_head_can_have():
    # four KV heads of 2377 tiles as one line of blocks of 82: the second head's tiles lie in 30 blocks, the records that
    # the scratch has room for
    y, exact, _ = _dense_steps(1, 4, 1, 64, 38016, 4)
    assert (y != exact.to(torch.bfloat16)).double().mean().item() <= 0.02


@pytest.mark.parametrize("B,H,Hkv,d,df,C,k,budget", [
    (5, 16, 4, 128, 128, 64, 16, 0),     # 80 read-outs beside the cache pass: one a block, by its eight warps
    (9, 20, 4, 64, 32, 64, 32, 0),       # 180, two warps each, narrow maps; five heads a group
    (9, 20, 4, 128, 64, 64, 32, 64),     # ... tokens that leave a capped cache
    (7, 32, 4, 128, 64, 32, 8, 0),       # 224, eight heads a group
    (20, 32, 8, 64, 64, 64, 16, 0),      # 640, a warp each
    (66, 32, 8, 64, 64, 32, 8, 0),       # 2112, and few tiles: no warps for the features
    (66, 32, 8, 64, 64, 64, 16, -1),     # ... long prefixes (-1): more for some blocks than they keep features for
    (5, 32, 2, 64, 64, 64, 16, 0),       # sixteen heads a group: no warps for the features
])
def test_decode_batch_gives_each_sequence_its_own(B, H, Hkv, d, df, C, k, budget):
    # The read-outs of a batch (features by warps of their own) against those of its sequences alone, and the rounding between:
    # y differs by at most two of its roundings to bf16.
    n0, steps, budget = (1290 if budget < 0 else 2 * C + 9), 3, max(budget, 0)
    w = synth.Workload("t", B, H, Hkv, d, n0 + steps, C, k, "bf16", "iid", 21)
    Q, K, V = synth.make_qkv(w, "cuda")
    g = torch.Generator(device="cuda").manual_seed(10)
    mk = lambda *s: (torch.randn(*s, generator=g, device="cuda") * 0.05).bfloat16()  # noqa: E731
    Wq, Wk, bq, bk, G = mk(H, d, df), mk(Hkv, d, df), mk(H, df), mk(Hkv, df), torch.rand(B, H, w.N, d, generator=g, device="cuda").bfloat16()

    def run(bs):
        p = still.StillParams(len(bs), H, Hkv, d, C, k, torch.bfloat16, d_f=df, sm_scale=w.sm_scale, max_salient=budget)
        x = [t[bs] for t in (Q, K, V, G)]
        state = torch.zeros(still.state_bytes(p, w.N), dtype=torch.uint8, device="cuda")
        pre = [t[:, :, :n0].contiguous() for t in x]
        still.hybrid_attn_fwd(p, *pre[:3], Wq, Wk, G=pre[3], bq=bq, bk=bk, state=state, state_max_tokens=w.N)
        return torch.stack([still.hybrid_attn_step(p, state, w.N, t, *(y[:, :, t].contiguous() for y in x[:3]), Wq, Wk,
                                                   g=x[3][:, :, t].contiguous(), bq=bq, bk=bk) for t in range(n0, w.N)], 2).float()

    Y = run(list(range(B)))
    for b in {0, B // 2, B - 1}:
        alone = run([b])[0]
        assert bool(((Y[b] - alone).abs() <= 2 ** -7 * alone.abs() + 1e-4).all())


@pytest.mark.parametrize("B,H,Hkv,d,n0", [
    # with few tiles a block the features of the read-outs are formed by the warps of the cache pass, with more by warps of their own
    (5, 16, 4, 128, 2500), (5, 16, 4, 128, 2800),      # one a block: 23 and 26 tiles
    (18, 32, 8, 128, 900), (18, 32, 8, 128, 1100),     # four: 56 and 68
    (10, 32, 8, 64, 1300), (10, 32, 8, 64, 1600),      # three, d = 64: 45 and 55
    (20, 32, 8, 128, 2350), (20, 32, 8, 128, 2700),    # five: 160 and 183
])
def test_decode_batch_on_both_sides_of_the_limits(B, H, Hkv, d, n0):
    # Sequences of a batch against the same sequences alone, and the rounding between.
    C, k, steps = 64, 16, 2
    w = synth.Workload("t", B, H, Hkv, d, n0 + steps, C, k, "bf16", "iid", 27)
    Q, K, V = synth.make_qkv(w, "cuda")
    Wq, Wk = synth.make_npmap_weights(w, "cuda")

    def run(bs):
        p = still.StillParams(len(bs), H, Hkv, d, C, k, torch.bfloat16, sm_scale=w.sm_scale)
        x = [t[bs] for t in (Q, K, V)]
        state = torch.zeros(still.state_bytes(p, w.N), dtype=torch.uint8, device="cuda")
        still.hybrid_attn_fwd(p, *(t[:, :, :n0].contiguous() for t in x), Wq, Wk, state=state, state_max_tokens=w.N)
        y = torch.stack([still.hybrid_attn_step(p, state, w.N, t, *(z[:, :, t].contiguous() for z in x), Wq, Wk) for t in range(n0, w.N)], 2)
        assert still.device_status(state) == (0, 0)
        return y.float()

    Y = run(list(range(B)))
    for b in (0, B - 1):
        alone = run([b])[0]
        assert bool(((Y[b] - alone).abs() <= 2 ** -7 * alone.abs() + 1e-4).all())   # two roundings of y to bf16 apart
