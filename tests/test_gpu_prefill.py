"""Parity of the CUDA prefill (still_hybrid_attn_fwd, through the C ABI) with the CPU oracle."""
import numpy as np
import pytest
import torch

import paper_2602_02180_b200 as still
from paper_2602_02180_b200 import synth
from tests import util_parity as U

pytestmark = pytest.mark.gpu


def _small(name, dtype, B, H, Hkv, d, N, C, k, recipe="iid", seed=1):
    return synth.Workload(name, B, H, Hkv, d, N, C, k, dtype, recipe, 4242 + seed)


def test_c1_fp32_every_row():
    w = synth.WORKLOADS["c1"]
    r = U.run_prefill(w)
    heads = U.sample_heads(w, 99)
    U.check_selection(r["scores"], r["sel"], w.C, w.k, heads)
    worst, serr = U.check_outputs(w, r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], r["Y"], r["scores"], r["sel"], heads)
    assert serr < 1e-4
    print(f"c1 max-abs {worst:.2e} score err {serr:.2e}")


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize(
    "B,H,Hkv,d,N,C,k",
    [
        (1, 2, 1, 64, 200, 32, 8),      # ragged tail, GQA
        (2, 4, 2, 64, 64 * 5 + 17, 64, 16),
        (1, 4, 4, 128, 128 * 3 + 1, 128, 32),
        (1, 2, 2, 64, 300, 64, 0),      # lambda = 0: local softmax + linear attention
        (1, 2, 1, 128, 333, 64, 1),
        (1, 2, 2, 64, 260, 64, 64),     # lambda = C: causal softmax attention
        (1, 2, 1, 128, 40, 64, 16),     # shorter than one chunk
        (1, 1, 1, 64, 1, 32, 4),        # a single token
        (1, 8, 2, 128, 128 * 4, 128, 128),
        (1, 4, 2, 64, 128 * 3 + 70, 128, 32),   # d = 64 with C = 128: two 64-token sub-chunks per chunk
        (1, 2, 1, 128, 64 * 40 + 17, 64, 16),   # many chunks, few heads: the state scan runs as four segments
        (1, 2, 2, 64, 128 * 33 + 5, 128, 32),   # the same with two sub-chunks per chunk (two segments)
    ],
)
def test_small_shapes(dtype, B, H, Hkv, d, N, C, k):
    w = _small("t", dtype, B, H, Hkv, d, N, C, k)
    r = U.run_prefill(w, gate=True, bias=True)
    heads = U.sample_heads(w, 4)
    if k:
        U.check_selection(r["scores"], r["sel"], C, k, heads)
    U.check_outputs(w, r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], r["Y"], r["scores"], r["sel"], heads,
                    G=r["G"], bq=r["bq"], bk=r["bk"])


@pytest.mark.parametrize(
    "B,H,Hkv,d,N,C,k,budget",
    [
        (1, 4, 2, 128, 64 * 12 + 9, 64, 16, 48),      # three chunks' selections stay cached
        (2, 2, 1, 64, 128 * 9 + 40, 128, 32, 64),     # two sub-chunks per chunk
        (1, 2, 2, 128, 64 * 10 + 3, 64, 64, 128),     # every token selected: a sliding window of two chunks + linear state
        (1, 2, 1, 128, 64 * 40 + 17, 64, 16, 64),     # the state scan in four segments
        (1, 4, 2, 128, 64 * 9, 64, 16, 16 * 64),      # a budget that is never reached
        (1, 2, 2, 64, 64 * 30, 64, 8, 8),             # a single chunk's selections
    ],
)
def test_salient_cache_budget(B, H, Hkv, d, N, C, k, budget):
    # max_salient: per head at most `budget` selected tokens stay in the softmax branch; the oldest leave for the
    # linear state when a newly routed chunk pushes them out (this library's rule; the paper caps the cache
    # without stating one).  The oracle applies the same rule.
    w = _small("t", "bf16", B, H, Hkv, d, N, C, k)
    r = U.run_prefill(w, gate=True, max_salient=budget)
    heads = U.sample_heads(w, 4)
    U.check_selection(r["scores"], r["sel"], C, k, heads)
    U.check_outputs(w, r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], r["Y"], r["scores"], r["sel"], heads, G=r["G"],
                    max_salient=budget)
    if budget >= (N // C) * k:   # never reached: the same bits as without a budget
        free = U.run_prefill(w, gate=True)
        assert torch.equal(free["Y"], r["Y"])


def test_salient_cache_budget_must_be_whole_chunks_of_selections():
    p = still.StillParams(1, 2, 2, 64, 64, 16, max_salient=40)
    assert still.workspace_bytes(p, 256) == 0
    assert still.workspace_bytes(still.StillParams(1, 2, 2, 64, 64, 16, torch.float32, max_salient=32), 256) == 0   # FMA path
    assert still.workspace_bytes(still.StillParams(1, 2, 2, 64, 64, 16, max_salient=32), 256) > 0


def _has_tie(scores, C):
    """True when some chunk holds two equal finite scores (so the tie arm of the ranking decided)."""
    sc = scores.cpu().numpy()
    n = sc.shape[-1] // C * C
    ch = np.sort(sc[..., :n].reshape(-1, C), axis=1)
    return bool(np.any((np.diff(ch, axis=1) == 0) & np.isfinite(ch[:, 1:])))


@pytest.mark.parametrize("dtype,d,C,k", [("bf16", 128, 64, 16), ("bf16", 64, 128, 32), ("bf16", 64, 64, 64 - 1),
                                         ("bf16", 64, 32, 8), ("fp32", 64, 64, 16), ("fp32", 128, 32, 8)])
@pytest.mark.parametrize("case", ["zero_queries", "periodic_tokens", "nan_key"])
def test_constructed_ties_and_nan_rank_like_the_oracle(dtype, d, C, k, case):
    # Top-lambda under the total order (score descending, position ascending), NaN lowest: the tie arm of the
    # ranking only runs when two scores of a chunk are equal, which random inputs never produce.
    #   zero_queries     every logit is 0, so every full window has the same score: whole chunks tie
    #   periodic_tokens  q, k repeat with period 16: tokens 16 apart see the same window contents
    #   nan_key          one key is NaN: the C rows whose window holds it have NaN scores
    w = _small("t", dtype, 1, 4, 2, d, C * 6 + C // 2 + 3, C, k)
    Q, K, V = synth.make_qkv(w, "cuda")
    if case == "zero_queries":
        Q = torch.zeros_like(Q)
    elif case == "periodic_tokens":
        reps = -(-w.N // 16)
        Q = Q[:, :, :16].repeat(1, 1, reps, 1)[:, :, : w.N].contiguous()
        K = K[:, :, :16].repeat(1, 1, reps, 1)[:, :, : w.N].contiguous()
    else:
        K = K.clone()
        K[0, 1, 2 * C + 5, 3] = float("nan")
    Wq, Wk = synth.make_npmap_weights(w, "cuda")
    Y, scores, sel = still.hybrid_attn_fwd(U.params_of(w), Q, K, V, Wq, Wk)
    torch.cuda.synchronize()
    heads = U.sample_heads(w, 99)
    U.check_selection(scores, sel, C, k, heads)
    if case == "nan_key":
        sc = scores.cpu().numpy()
        assert np.isnan(sc[0, 2:, 2 * C + 5: 3 * C + 5]).all() and np.isfinite(sc[0, :2]).all()
        assert np.isfinite(sc[0, 2:, : 2 * C + 5]).all() and np.isfinite(sc[0, 2:, 3 * C + 5:]).all()
        # a NaN score ranks below every number: the five finite rows of the chunk (positions 2C .. 2C+4) are
        # taken before any of its NaN rows
        picked = sel[0, 2:, 2].cpu().numpy()
        n_finite = 5
        assert ((picked < 2 * C + 5) & (picked >= 0)).sum(axis=1).min() == min(k, n_finite)
        heads = [(0, 0), (0, 1)]   # the heads of the KV head without the NaN stay finite and are compared
    else:
        assert _has_tie(scores, C), "the constructed input produced no tie"
    U.check_outputs(w, Q, K, V, Wq, Wk, Y, scores, sel, heads)


def test_feature_width_smaller_than_head_dim():
    # d_f = 64 with d = 128: feature dim d' = 128 (other template instance of the NP-Map and scan kernels)
    w = _small("t", "bf16", 1, 4, 2, 128, 64 * 7 + 5, 64, 16)
    Q, K, V = synth.make_qkv(w, "cuda")
    g = torch.Generator(device="cuda").manual_seed(11)
    Wq = (torch.randn(w.H, w.d, 64, generator=g, device="cuda") * 0.02).to(torch.bfloat16)
    Wk = (torch.randn(w.Hkv, w.d, 64, generator=g, device="cuda") * 0.02).to(torch.bfloat16)
    p = still.StillParams(w.B, w.H, w.Hkv, w.d, w.C, w.k, torch.bfloat16, d_f=64)
    Y, scores, sel = still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk)
    torch.cuda.synchronize()
    heads = U.sample_heads(w, 4)
    U.check_selection(scores, sel, w.C, w.k, heads)
    U.check_outputs(w, Q, K, V, Wq, Wk, Y, scores, sel, heads)


def test_paper_literal_scale_one():
    # sm_scale = 1 is the main text's exp(q k^T); inputs are scaled down so the softmaxes stay soft.
    w = _small("t", "fp32", 1, 2, 2, 64, 256, 64, 16)
    Q, K, V = synth.make_qkv(w, "cuda")
    Q, K = Q * 0.35, K * 0.35
    Wq, Wk = synth.make_npmap_weights(w, "cuda")
    p = still.StillParams(w.B, w.H, w.Hkv, w.d, w.C, w.k, torch.float32, sm_scale=1.0)
    Y, scores, sel = still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk)
    heads = U.sample_heads(w, 2)
    U.check_selection(scores, sel, w.C, w.k, heads)
    from oracle import still_oracle as oracle
    for b, h in heads:
        out = oracle.chunkwise(U.f64(Q[b, h]), U.f64(K[b, h]), U.f64(V[b, h]), U.f64(Wq[h]), U.f64(Wk[h]),
                               oracle.HeadParams(w.C, w.k, 1.0), forced_idx=sel[b, h].cpu().numpy())
        assert np.abs(U.f64(Y[b, h]) - out["y"]).max() < 1e-4


@pytest.mark.parametrize("dtype,d,df,C,k,N", [
    ("fp32", 64, 32, 32, 8, 32 * 11 + 5), ("fp32", 128, 64, 64, 64 - 1, 64 * 9 + 1), ("fp32", 128, 32, 128, 32, 128 * 6 + 127),
    ("bf16", 128, 128, 32, 8, 32 * 9 + 31), ("bf16", 64, 32, 64, 16, 64 * 7),   # bf16 shapes of the FMA kernels
])
def test_fma_kernels_feature_sizes_and_bias(dtype, d, df, C, k, N):
    # maps narrower than the head and a bias, scan segments of one and two chunks, ragged ends
    B, H, Hkv = 1, 4, 2
    w = _small("t", dtype, B, H, Hkv, d, N, C, k)
    Q, K, V = synth.make_qkv(w, "cuda")
    G = synth.make_gate(w, "cuda")
    g = torch.Generator(device="cuda").manual_seed(10)
    mk = lambda *s: (torch.randn(*s, generator=g, device="cuda") * 0.05).to(w.torch_dtype)  # noqa: E731
    Wq, Wk, bq, bk = mk(H, d, df), mk(Hkv, d, df), mk(H, df), mk(Hkv, df)
    p = still.StillParams(B, H, Hkv, d, C, k, w.torch_dtype, d_f=df, sm_scale=w.sm_scale)
    Y, scores, sel = still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk, G=G, bq=bq, bk=bk)
    heads = [(0, h) for h in range(H)]
    U.check_selection(scores, sel, C, k, heads)
    U.check_outputs(w, Q, K, V, Wq, Wk, Y, scores, sel, heads, G=G, bq=bq, bk=bk)


@pytest.mark.parametrize("d,C", [(64, 64), (128, 128)])
def test_scores_with_a_subnormal_eps(d, C):
    # every logarithm's argument contains eps; a subnormal one takes the form that scales its argument.  Scores reach
    # log(1 / eps) = 90 here, seven times the range the score tolerance is stated for.
    w = _small("t", "bf16", 1, 4, 2, d, C * 3 + 9, C, C // 4)
    Q, K, V = synth.make_qkv(w, "cuda")
    Wq, Wk = synth.make_npmap_weights(w, "cuda")
    p = still.StillParams(w.B, w.H, w.Hkv, d, C, w.k, torch.bfloat16, sm_scale=w.sm_scale, eps=1e-39)
    Y, scores, sel = still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk)
    heads = [(0, h) for h in range(4)]
    U.check_selection(scores, sel, C, w.k, heads)
    U.check_outputs(w, Q, K, V, Wq, Wk, Y, scores, sel, heads, eps=float(np.float32(1e-39)), score_tol=7 * U.SCORE_TOL[torch.bfloat16])


@pytest.mark.parametrize("d,B,H,Hkv,N", [(64, 3, 6, 2, 700), (128, 1, 8, 4, 1100), (64, 1, 8, 4, 128 * 1024 + 70), (128, 1, 4, 2, 64 * 1024 + 200)])
def test_row_blocks_of_all_heads(d, B, H, Hkv, N):
    # every row block of every head is worked on once, with the heads in one set and in several (65536 keys of a KV group
    # at d = 128, 131072 at d = 64, fill a set): rows that were left out would keep the NaN they start with
    w = _small("t", "bf16", B, H, Hkv, d, N, 64, 64)
    Q, K, V = synth.make_qkv(w, "cuda")
    p = U.params_of(w)
    Y, scores, sel = still.hybrid_attn_fwd(p, Q, K, V, Y=torch.full_like(Q, float("nan")))
    heads = U.sample_heads(w, 3)
    rows = U.sample_rows(N, 12, 64)
    U.check_outputs(w, Q, K, V, *synth.make_npmap_weights(w, "cuda"), Y, scores, sel, heads, rows=rows)
    assert bool(torch.isfinite(Y.float()).all())


@pytest.mark.parametrize("k", [64, 16])
def test_growing_logits_rescale_the_accumulator(k):
    # The tensor-core kernel keeps a row's softmax reference until a tile's maximum exceeds it by 2^8 and then
    # rescales the output accumulator.  Logits that grow by ~7 nats per 128-key tile, plus one key far above the
    # rest in the second half of a tile, make that happen in every tile and in both halves.
    w = _small("t", "bf16", 1, 4, 2, 128, 128 * 7 + 40, 64, k)
    Q, K, V = synth.make_qkv(w, "cuda")
    t = torch.arange(w.N, device="cuda")
    Q = Q.float()
    K = K.float()
    Q[..., 0] += 8.0
    K[..., 0] += (10.0 * (t // 128)).view(1, 1, -1)
    K[:, :, 128 * 3 + 100, 0] += 60.0
    Q, K = Q.to(torch.bfloat16), K.to(torch.bfloat16)
    Wq, Wk = synth.make_npmap_weights(w, "cuda")
    Y, scores, sel = still.hybrid_attn_fwd(U.params_of(w), Q, K, V, Wq, Wk)
    torch.cuda.synchronize()
    assert torch.isfinite(Y.float()).all()
    heads = U.sample_heads(w, 4)
    U.check_selection(scores, sel, w.C, w.k, heads)
    U.check_outputs(w, Q, K, V, Wq, Wk, Y, scores, sel, heads)


def test_run_to_run_determinism():
    w = _small("t", "bf16", 1, 4, 2, 64, 500, 64, 16)
    a = U.run_prefill(w)
    b = U.run_prefill(w)
    assert torch.equal(a["Y"], b["Y"]) and torch.equal(a["sel"], b["sel"]) and torch.equal(a["scores"], b["scores"])


def test_constant_value_rows():
    # y is a positive-weight average of the values: constant V gives constant y (gate = 1).
    w = _small("t", "fp32", 1, 2, 2, 64, 320, 64, 16)
    Q, K, V = synth.make_qkv(w, "cuda")
    V = torch.ones_like(V) * 0.75
    Wq, Wk = synth.make_npmap_weights(w, "cuda")
    Y, _, _ = still.hybrid_attn_fwd(U.params_of(w), Q, K, V, Wq, Wk)
    assert (Y - 0.75).abs().max().item() < 1e-5


def test_c2_sampled():
    w = synth.WORKLOADS["c2"]
    r = U.run_prefill(w)
    heads = U.sample_heads(w, 6, seed=2)
    rows = U.sample_rows(w.N, 96, w.C, seed=2)
    U.check_selection(r["scores"], r["sel"], w.C, w.k, heads)
    worst, serr = U.check_outputs(w, r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], r["Y"], r["scores"], r["sel"],
                                  heads, rows=rows)
    print(f"c2 max-abs {worst:.2e} score err {serr:.2e}")
    # companion with a non-degenerate selection (lambda = C/4)
    w4 = w.with_(k=w.C // 4)
    r = U.run_prefill(w4)
    U.check_selection(r["scores"], r["sel"], w4.C, w4.k, heads)
    U.check_outputs(w4, r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], r["Y"], r["scores"], r["sel"], heads, rows=rows)


@pytest.mark.parametrize("name,n_heads,n_rows", [("c3", 3, 40), ("c4", 2, 24)])
def test_full_size_workloads_sampled(name, n_heads, n_rows):
    # The benchmark's own shapes and launch configuration; the oracle checks sampled heads and rows
    # (all O(N) steps -- scores, selection -- in full for those heads).
    w = synth.WORKLOADS[name]
    r = U.run_prefill(w)
    assert still.device_status is not None
    heads = U.sample_heads(w, n_heads, seed=3)
    rows = set(U.sample_rows(w.N, n_rows, w.C, seed=3))
    # rows that sit on a key of unusual norm (c3: the 5x outlier keys, c4: the heavy tail) and the rows right
    # after one, where that key dominates the window: the positions these workloads exist for
    for b, h in heads:
        kn = r["K"][b, h // (w.H // w.Hkv)].float().norm(dim=-1)
        top = torch.topk(kn, 4).indices.cpu().tolist()
        for t in top:
            rows.update(x for x in (t, t + 1, t + w.C - 1, t + w.C, t + 2 * w.C) if x < w.N)
    rows = sorted(rows)
    U.check_selection(r["scores"], r["sel"], w.C, w.k, heads)
    rep = {}
    worst, serr = U.check_outputs(w, r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], r["Y"], r["scores"], r["sel"],
                                  heads, rows=rows, report=rep)
    print(f"{name} max-abs {worst:.2e} score err {serr:.2e} on {len(rows)} rows of {len(heads)} heads; "
          f"selection Jaccard (oracle's own vs GPU) {np.mean(rep['jaccard']):.4f}")


def test_c3_companion_quarter_selection_sampled():
    # lambda = C / 4 at the 32K shape: selection, NP-Map, state scan and merge at scale
    w = synth.WORKLOADS["c3"].with_(B=1, k=16)
    r = U.run_prefill(w)
    heads = U.sample_heads(w, 2, seed=4)
    rows = U.sample_rows(w.N, 32, w.C, seed=4)
    U.check_selection(r["scores"], r["sel"], w.C, w.k, heads)
    rep = {}
    worst, serr = U.check_outputs(w, r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], r["Y"], r["scores"], r["sel"],
                                  heads, rows=rows, report=rep)
    print(f"c3 k16 max-abs {worst:.2e} score err {serr:.2e}; selection Jaccard (oracle's own vs GPU) "
          f"{np.mean(rep['jaccard']):.4f}")


def test_invalid_arguments_are_rejected():
    w = _small("t", "bf16", 1, 2, 2, 64, 128, 64, 16)
    Q, K, V = synth.make_qkv(w, "cuda")
    Wq, Wk = synth.make_npmap_weights(w, "cuda")
    p = U.params_of(w)
    with pytest.raises(still.StillError) as e:
        still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk, workspace=torch.empty(1024, dtype=torch.uint8, device="cuda"))
    assert e.value.code == -3
    bad = still.StillParams(1, 3, 2, 64, 64, 16)
    assert still.workspace_bytes(bad, 128) == 0
    with pytest.raises(still.StillError):
        still.hybrid_attn_fwd(still.StillParams(1, 2, 2, 64, 64, 65), Q, K, V, Wq, Wk,
                              workspace=torch.empty(1 << 20, dtype=torch.uint8, device="cuda"))
    ws = torch.empty(still.workspace_bytes(p, 128) + 16, dtype=torch.uint8, device="cuda")
    with pytest.raises(still.StillError) as e:  # misaligned workspace pointer
        still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk, workspace=ws[1:])
    assert e.value.code == -1


def test_bounded_device_wait_runs_out_and_is_reported():
    # The tensor-core kernels wait on mbarriers with a cycle limit; when a wait runs out the kernel records
    # STILL_ERR_DEVICE_TIMEOUT in the status block and returns.  The self-test kernel is that wait alone, on a
    # barrier nothing arrives on, with a limit of about a millisecond: it must come back, report (-6, 99) and
    # leave the context usable.
    block = torch.full((256,), 0x5A, dtype=torch.uint8, device="cuda")
    still.selftest_wait_timeout(block, 2_000_000)
    assert still.device_status(block) == (-6, 99)
    w = _small("t", "bf16", 1, 2, 2, 64, 300, 64, 16)
    r = U.run_prefill(w)
    assert torch.isfinite(r["Y"].float()).all()
    ws = torch.empty(still.workspace_bytes(r["p"], w.N), dtype=torch.uint8, device="cuda")
    still.hybrid_attn_fwd(r["p"], r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], workspace=ws)
    assert still.device_status(ws) == (0, 0)


def test_prefills_back_to_back_on_one_workspace():
    # Calls enqueued without waiting: the kernels of a call are resident while the call before, or the kernel that fills
    # its inputs, still runs, and all use the same input, output and workspace buffers.  Every output has to be the one of
    # the call made by itself.
    for dtype, d, C, k, budget in [("bf16", 128, 64, 16, 0), ("bf16", 64, 128, 32, 64), ("fp32", 64, 32, 8, 0), ("bf16", 64, 32, 8, 0)]:
        w = _small("t", dtype, 1, 4, 2, d, C * 9 + 5, C, k)
        p = U.params_of(w, max_salient=budget)
        ins = [(*synth.make_qkv(w.with_(seed=s), "cuda"), synth.make_gate(w.with_(seed=s), "cuda"), *synth.make_npmap_weights(w.with_(seed=s), "cuda"))
               for s in range(4)]
        call = lambda x, **kw: still.hybrid_attn_fwd(p, *x[:3], *x[4:], G=x[3], **kw)  # noqa: E731
        alone = []
        for x in ins:
            alone.append(call(x))
            torch.cuda.synchronize()
        buf, out = [torch.empty_like(t) for t in ins[0]], [torch.empty_like(t) for t in alone[0]]
        ws = torch.empty(still.workspace_bytes(p, w.N), dtype=torch.uint8, device="cuda")
        got = []
        torch.cuda.synchronize()
        for x in ins * 2:
            for dst, src in zip(buf, x):
                dst.copy_(src)
            got.append([t.clone() for t in call(buf, Y=out[0], scores=out[1], sel_idx=out[2], workspace=ws)])
        torch.cuda.synchronize()
        for want, have in zip(alone * 2, got):
            assert all(torch.equal(a, b) for a, b in zip(want, have)), (dtype, d, C)


def test_fp32_nan_logits_make_the_output_nan():
    # the first tile of keys (64 at d = 64) NaN for one KV head: every row of its query heads sees a NaN
    w = _small("t", "fp32", 1, 4, 2, 64, 300, 64, 64)
    Q, K, V = synth.make_qkv(w, "cuda")
    K[:, 0, :64] = torch.nan
    Y = still.hybrid_attn_fwd(U.params_of(w), Q, K, V)[0]
    assert bool(torch.isnan(Y[:, :2]).all()) and bool(torch.isfinite(Y[:, 2:]).all())


@pytest.mark.parametrize("H,Hkv,d,df,C,k,N", [
    (16, 4, 64, 64, 64, 16, 1024),     # 14 segments wanted, room for three beside the workspace: eight in N_LA
    (16, 4, 64, 64, 64, 16, 1150),     # no room at all
    (16, 4, 64, 64, 64, 16, 1200),     # past the static workspace: a place of their own again
    (8, 4, 128, 128, 64, 16, 1000),    # segments of four chunks (2 d_f = 256 tokens) and a longer last one
    (32, 4, 64, 32, 128, 32, 640 + 127),   # segments of one chunk: the second one's rows are answered with zeros
    (16, 4, 128, 64, 32, 8, 515),
])
def test_fp32_scan_segments_without_room_for_their_sums(H, Hkv, d, df, C, k, N):
    # Below the 16 MiB of the static workspace the sums of the scan's segments have no place of their own; they then lie in
    # rows of N_LA and D_LA.  Parity on every head, with the state, and no fall back to one serial pass.
    w = _small("t", "fp32", 1, H, Hkv, d, N, C, k)
    p = still.StillParams(1, H, Hkv, d, C, k, torch.float32, d_f=df, sm_scale=w.sm_scale)
    Q, K, V = synth.make_qkv(w, "cuda")
    g = torch.Generator(device="cuda").manual_seed(12)
    Wq, Wk = (torch.randn(n, d, df, generator=g, device="cuda") * 0.05 for n in (H, Hkv))
    G = synth.make_gate(w, "cuda")
    lay = still.state_layout(p, N)
    state = torch.zeros(lay["total"], dtype=torch.uint8, device="cuda")
    ws = torch.full((still.workspace_bytes(p, N) + 4096,), 255, dtype=torch.uint8, device="cuda")   # (NaN wherever nothing is written)
    Y, scores, sel = still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk, G=G, state=state, state_max_tokens=N, workspace=ws[:-4096])
    assert still.last_launch_count() == 8      # score, two maps, sums, prefix, scan, attention, state
    assert bool((ws[-4096:] == 255).all())
    heads = [(0, h) for h in range(0, H, 3)]
    U.check_selection(scores, sel, C, k, heads)
    U.check_outputs(w, Q, K, V, Wq, Wk, Y, scores, sel, heads, G=G, tol=1e-5)
    # S and z: phi(K)^T [V, 1] over the unselected tokens of the routed chunks, in float64
    n = (-(-N // C) - 2) * C
    S = state[lay["S"]: lay["S"] + H * 2 * df * d * 4].view(torch.float32).view(H, 2 * df, d)
    z = state[lay["z"]: lay["z"] + H * 2 * df * 4].view(torch.float32).view(H, 2 * df)
    for _, h in heads:
        x, W = K[0, h // (H // Hkv), :n].double(), Wk[h // (H // Hkv)].double()
        f = x @ W
        u = f * (x.norm(dim=1, keepdim=True) / f.norm(dim=1, keepdim=True))
        phi = torch.cat([u.softmax(1), (-u).softmax(1)], 1)
        idx = sel[0, h].flatten().long()
        phi[idx[(idx >= 0) & (idx < n)]] = 0
        for got, want in ((S[h], phi.T @ V[0, h // (H // Hkv), :n].double()), (z[h], phi.sum(0))):
            assert float((got - want).norm() / want.norm()) <= 2e-6   # (fp32 features and sums of up to 1100 terms)


def test_a_refused_launch_does_not_fail_the_next_call():
    # 65536 KV heads exceed a grid dimension: the launch is refused on the host and the call says so.  The next call, which
    # checks for launch errors itself, must not find that one.
    many = still.StillParams(1, 65536, 65536, 64, 64, 16)
    x, w = torch.zeros(1, 65536, 4, 64, dtype=torch.bfloat16, device="cuda"), torch.zeros(65536, 64, 64, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(still.StillError) as e:
        still.hybrid_attn_fwd(many, x, x, x, w, w)
    assert e.value.code == -5
    del x, w
    r = U.run_prefill(_small("t", "bf16", 1, 2, 1, 64, 200, 64, 16))
    assert bool(torch.isfinite(r["Y"].float()).all())


@pytest.mark.parametrize("B,H,Hkv,d,df,C,k,N", [
    (1, 4, 4, 64, 64, 64, 16, 512),      # one launch for score and maps, a chunk a segment
    (1, 4, 2, 64, 32, 64, 16, 577),      # ... a last block of one row, narrow maps
    (2, 2, 1, 128, 128, 64, 8, 190),     # head dim 128, a ragged chunk; three chunks: one pass of the scan
    (1, 4, 2, 64, 64, 64, 16, 256),      # ... the last such size
    (1, 4, 2, 64, 64, 64, 16, 257),      # five: three passes
    (1, 2, 2, 128, 64, 128, 32, 700),    # wide blocks take half of a chunk of 128
    (1, 3, 1, 64, 64, 32, 8, 333),       # chunks of 32: plain blocks
    (1, 8, 2, 64, 64, 64, 16, 1030),     # 222 blocks of score and maps, the most that are one launch ...
    (1, 8, 2, 64, 64, 64, 16, 1100),     # ... and more
])
def test_fp32_small_calls(B, H, Hkv, d, df, C, k, N):
    w = _small("t", "fp32", B, H, Hkv, d, N, C, k)
    p = still.StillParams(B, H, Hkv, d, C, k, torch.float32, d_f=df, sm_scale=w.sm_scale)
    Q, K, V = synth.make_qkv(w, "cuda")
    g = torch.Generator(device="cuda").manual_seed(13)
    Wq, Wk = (torch.randn(n, d, df, generator=g, device="cuda") * 0.05 for n in (H, Hkv))
    bq, bk = (torch.randn(n, df, generator=g, device="cuda") * 0.05 for n in (H, Hkv))
    ws = torch.full((still.workspace_bytes(p, N) + 4096,), 255, dtype=torch.uint8, device="cuda")   # (NaN wherever nothing is written)
    Y, scores, sel = still.hybrid_attn_fwd(p, Q, K, V, Wq, Wk, bq=bq, bk=bk, workspace=ws[:-4096])
    chunks, rows = -(-N // C), -(-N // (64 if C == 32 else 128))
    one = B * H * chunks + B * (H + Hkv) * rows <= 222
    assert still.last_launch_count() == (1 if one else 3) + (3 if chunks > 4 else 1) + 1 and bool((ws[-4096:] == 255).all())
    heads = [(0, 0), (B - 1, H - 1)]
    U.check_selection(scores, sel, C, k, heads)
    U.check_outputs(w, Q, K, V, Wq, Wk, Y, scores, sel, heads, bq=bq, bk=bk, tol=1e-5)


@pytest.mark.parametrize("N,rides", [(200, True), (1400, True), (1500, False)])
def test_state_written_among_the_gathered_rows(N, rides):
    # 505 and 545 blocks of copies: the last size that rides along with the gather, and one with a launch of its own
    B, H, Hkv, d, C, k = 1, 32, 8, 128, 64, 16
    w = _small("t", "bf16", B, H, Hkv, d, N, C, k)
    p, cap = U.params_of(w), N + 70
    lay = still.state_layout(p, cap)
    state = torch.full((lay["total"],), 255, dtype=torch.uint8, device="cuda")
    r = U.run_prefill(w, state=state, state_max_tokens=cap)
    with_state = still.last_launch_count()
    U.run_prefill(w)
    assert with_state - still.last_launch_count() == (0 if rides else 1)
    n_cap, part = lay["capacity"], lambda at, n, dt: state[lay[at]: lay[at] + n * dt.itemsize].view(dt)
    for at, x in (("k_cache", r["K"]), ("v_cache", r["V"])):
        assert torch.equal(part(at, B * Hkv * n_cap * d, torch.bfloat16).view(B, Hkv, n_cap, d)[:, :, :N], x)
    assert torch.equal(part("score", B * H * n_cap, torch.float32).view(B, H, n_cap)[:, :, :N], r["scores"])
    T = -(-N // C)
    assert torch.equal(part("sel_idx", B * H * (n_cap // C) * k, torch.int32).view(B, H, -1, k)[:, :, :T], r["sel"])
    words = part("sel_mask", B * H * (n_cap // C) * (C // 32), torch.int32).view(B, H, -1)[:, :, : T * (C // 32)].cpu()
    bits = ((words[..., None] >> torch.arange(32)) & 1).flatten(2)
    want = torch.zeros(B, H, T * C, dtype=torch.int32)
    sel = r["sel"].cpu().flatten(2).long()
    want.scatter_add_(2, sel.clamp_min(0), (sel >= 0).int())
    assert torch.equal(bits, want)
    assert part("header", 14, torch.int32)[12].item() == N


@pytest.mark.parametrize("H,Hkv,d,N", [
    (32, 8, 128, 320), (32, 8, 128, 330),   # a chunk a segment, and two from 321 (chunks x heads x d / 64) on
    (28, 4, 64, 1024), (28, 4, 64, 1030),   # ... from 449 on: 16 and 17 chunks
])
def test_fp32_segments_of_one_chunk_and_of_two(H, Hkv, d, N):
    C, k = 64, 16
    w = _small("t", "fp32", 1, H, Hkv, d, N, C, k)
    lay = still.state_layout(U.params_of(w), N)
    state = torch.zeros(lay["total"], dtype=torch.uint8, device="cuda")
    r = U.run_prefill(w, state=state, state_max_tokens=N)
    heads = [(0, 0), (0, H - 1)]
    U.check_selection(r["scores"], r["sel"], C, k, heads)
    U.check_outputs(w, r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], r["Y"], r["scores"], r["sel"], heads, tol=1e-5)
    # z: the features of the unselected tokens of the routed chunks, which sum to 2 each
    z = state[lay["z"]: lay["z"] + H * 2 * d * 4].view(torch.float32).view(H, 2 * d)
    n = -(-N // C) - 2
    want = 2.0 * n * (C - k)
    assert float((z.double().sum(1) - want).abs().max()) <= want * n * C * 2 ** -24   # (fp32 sums of up to n C terms)
