"""Edges of the tensor-core prefill: the key streams of the attention kernels' query tiles, and the segments of the linear
branch's scan."""
import pytest
import torch

import paper_2602_02180_b200 as still
from paper_2602_02180_b200 import synth

from . import util_parity as U

pytestmark = pytest.mark.gpu


def _workload(H, Hkv, d, N, C, k):
    return synth.Workload("t", 1, H, Hkv, d, N, C, k, "bf16", "head_scale", 31)


@pytest.mark.parametrize("d,N,C,k,budget", [
    # one query tile; a second one of a single row; a CTA (256 rows; a pair: 512) that is just full, and one row more
    (64, 1, 64, 16, 0), (64, 128, 64, 16, 0), (64, 129, 64, 16, 0), (64, 256, 64, 64, 0), (64, 257, 128, 32, 0),
    (128, 1, 64, 16, 0), (128, 256, 64, 64, 0), (128, 257, 128, 32, 0), (128, 512, 64, 16, 0), (128, 513, 64, 16, 0),
    # shared tiles that run through the ring several times, and own tiles of both query tiles behind them
    (64, 2111, 64, 64, 0), (128, 2303, 64, 64, 0), (128, 2200, 128, 1, 0),
    # a CTA pair whose last rows are few: the first query tile goes on after the second has no more
    (128, 820, 64, 16, 0), (128, 1836, 64, 16, 64), (128, 1836, 64, 32, 64),
    # windows of the capped cache that two query tiles share in part, or not at all (then every tile is one's own)
    (64, 1500, 64, 16, 64), (64, 1500, 64, 64, 64), (128, 2000, 64, 64, 64), (128, 2000, 128, 32, 32), (128, 2100, 64, 32, 896),
])
def test_key_streams(d, N, C, k, budget):
    w = _workload(4, 2, d, N, C, k)
    r = U.run_prefill(w, max_salient=budget)
    heads = [(0, 0), (0, 3)]
    U.check_selection(r["scores"], r["sel"], C, k, heads)
    U.check_outputs(w, r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], r["Y"], r["scores"], r["sel"], heads, max_salient=budget)


@pytest.mark.parametrize("H,Hkv,d,N,C,k,budget,gate", [
    (32, 8, 128, 1003, 64, 16, 0, True),      # two segments that fold again, gated
    (32, 8, 64, 1090, 64, 16, 0, False),      # rows that are no whole sub-chunk, without a gate
    (16, 4, 128, 2048, 64, 16, 0, False),     # four segments, 48 tiles before the last: folded again
    (16, 4, 128, 2752, 64, 16, 0, False),     # 72 tiles: a pass of sums, pieces of three chunks
    (4, 4, 64, 3000, 64, 32, 0, False),       # ... a ring of eleven stages
    (16, 4, 128, 4200, 128, 32, 128, False),  # ... with tokens leaving a capped cache
    (4, 2, 128, 4300, 128, 128, 256, False),  # ... every token selected: the state holds the leaving ones alone
])
def test_linear_scan_segments(H, Hkv, d, N, C, k, budget, gate):
    w = _workload(H, Hkv, d, N, C, k)
    p = U.params_of(w, max_salient=budget)
    lay = still.state_layout(p, N)
    state = torch.zeros(lay["total"], dtype=torch.uint8, device="cuda")
    r = U.run_prefill(w, gate=gate, max_salient=budget, state=state, state_max_tokens=N)
    heads = [(0, 0), (0, H - 1)]
    U.check_outputs(w, r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], r["Y"], r["scores"], r["sel"], heads, G=r["G"],
                    rows=U.sample_rows(N, 200, C), max_salient=budget)
    # S and z: phi(K)^T [V, 1] over the tokens that have left for the state, in float64.  The features are rounded to bf16, by at
    # most 2^-9 each, independently of the signs of V: twice that for S, once for sums of positive terms.
    T, window = -(-N // C), budget // k
    n = (T - 2) * C
    S = state[lay["S"]: lay["S"] + H * 2 * d * d * 4].view(torch.float32).view(H, 2 * d, d)
    z = state[lay["z"]: lay["z"] + H * 2 * d * 4].view(torch.float32).view(H, 2 * d)
    for _, h in heads:
        kv = h // (H // Hkv)
        x, W = r["K"][0, kv, :n].double(), r["Wk"][kv].double()
        f = x @ W
        u = f * (x.norm(dim=1, keepdim=True) / f.norm(dim=1, keepdim=True))
        phi = torch.cat([u.softmax(1), (-u).softmax(1)], 1)
        still_cached = r["sel"][0, h, max(T - 2 - window, 0) if window else 0: T - 2].flatten().long()
        phi[still_cached] = 0
        for got, want, tol in ((S[h], phi.T @ r["V"][0, kv, :n].double(), 2 ** -8), (z[h], phi.sum(0), 2 ** -9)):
            assert float((got - want).norm() / want.norm()) <= tol


@pytest.mark.parametrize("N,C,k,budget", [
    (700, 64, 64, 0), (2303, 64, 64, 0), (1500, 128, 32, 0),
    # windows of the capped cache: none, one or two tiles that the first query tile alone sees ahead of the shared ones
    (1100, 64, 64, 256), (1500, 64, 64, 640), (2000, 128, 32, 64), (3000, 128, 32, 896), (1836, 64, 16, 64), (2100, 64, 32, 896),
])
def test_both_head_dims_give_the_same_rows(N, C, k, budget):
    # A head of 64 dims, and the same head with 64 more that add nothing to its logits and features and hold its values once
    # more: the kernels of both head dims weigh and sum the same numbers in the same order, so the rows are equal, bit for bit.
    w = _workload(4, 2, 64, N, C, k)
    Q, K, V = synth.make_qkv(w, "cuda")
    Wq, Wk = synth.make_npmap_weights(w, "cuda")
    call = lambda d, *x: still.hybrid_attn_fwd(still.StillParams(1, 4, 2, d, C, k, torch.bfloat16, d_f=64, sm_scale=w.sm_scale,  # noqa: E731
                                                                 max_salient=budget), *x)
    wide = lambda x: torch.cat([x, torch.zeros_like(x)], -1)  # noqa: E731
    Y, scores, sel = call(64, Q, K, V, Wq, Wk)
    Y2, scores2, sel2 = call(128, wide(Q), wide(K), torch.cat([V, V], -1), torch.cat([Wq, torch.zeros_like(Wq)], 1),
                             torch.cat([Wk, torch.zeros_like(Wk)], 1))
    assert torch.equal(scores, scores2) and torch.equal(sel, sel2)
    assert torch.equal(torch.cat([Y, Y], -1), Y2)


@pytest.mark.parametrize("H,d,df,N", [
    (32, 64, 64, 1003), (32, 128, 128, 1003),   # two segments; pieces of two chunks, the first of them empty
    (37, 128, 64, 2100),                        # the most heads that are cut
    (16, 128, 128, 2048),                       # four segments: eleven pieces
    (16, 64, 64, 2500),                         # pieces of five chunks
    (32, 128, 128, 3000),                       # pieces of six chunks
    (4, 128, 128, 2048), (8, 64, 64, 2048),     # 48 tiles, folded again in one wave at d = 128 and in two
    (4, 64, 64, 2048), (4, 64, 64, 3000),       # ... a pass of sums at d = 64; 72 tiles
])
def test_linear_state_is_the_fp32_sum_of_its_pieces(H, d, df, N):
    # W_k = 0 makes every feature 1 / d_f exactly.  Chunk 0 brings 2^24 into the state of every head, whose neighbours in fp32
    # are 2 apart; the chunks of a later piece bring 1 each, 1/4 at most in one step of the tensor cores.  A piece of 2 n
    # chunks then adds 2 n exactly, if it is summed by itself and added in fp32; step by step it would be rounded away.
    # (With an odd number of chunks a piece's sum is odd, and 1 is lost to rounding.)
    C = 64
    T = -(-N // C)
    n_seg = 4 if H <= 18 and T >= 32 else 2
    per = -(-T // n_seg)
    per += per & 1                                                   # chunks of a segment
    parts = 4 if per % 4 == 0 and per >= 8 else 2 if per >= 4 else 1
    own = (n_seg - 1) * per - 2                                      # first chunk of the last segment's own updates
    p = still.StillParams(1, H, 1, d, C, C // 2, torch.bfloat16, d_f=df)
    g = torch.Generator(device="cuda").manual_seed(7)
    Q, K = (torch.randn(1, n, N, d, generator=g, device="cuda").bfloat16() for n in (H, 1))
    Wq = (torch.randn(H, d, df, generator=g, device="cuda") * 0.02).bfloat16()
    V = torch.zeros(1, 1, N, d, device="cuda", dtype=torch.bfloat16)
    first = per // parts - 2 if per // parts > 2 else per // parts   # chunks of the first piece
    V[:, :, :C] = 2.0 ** 19 * df                                     # (32 unselected tokens of a chunk)
    V[:, :, first * C: own * C] = df / 32
    lay = still.state_layout(p, N)
    state = torch.zeros(lay["total"], dtype=torch.uint8, device="cuda")
    still.hybrid_attn_fwd(p, Q, K, V, Wq, torch.zeros(1, d, df, device="cuda", dtype=torch.bfloat16), state=state, state_max_tokens=N)
    S = state[lay["S"]: lay["S"] + H * 2 * df * d * 4].view(torch.float32)
    pieces, chunks = (own - first) // (per // parts), per // parts
    want = torch.tensor(2.0 ** 24, dtype=torch.float32)
    for _ in range(pieces):
        want = want + chunks
    assert S.unique().tolist() == [float(want)]


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("d,N,key", [
    (64, 400, 0), (64, 400, 8), (64, 400, 131), (128, 700, 0), (128, 700, 17), (128, 700, 250), (128, 1300, 70),
])
def test_nan_and_infinite_logits_make_the_output_nan(d, N, key, bad):
    # One key of one KV head, also in columns whose exponential is the cubic: every row that sees it is NaN in every column, as
    # inf - inf and NaN are, and no other row.  (Q > 0, so that the logit is +inf and not -inf.)
    w = _workload(4, 2, d, N, 64, 64)
    Q, K, V = synth.make_qkv(w, "cuda")
    K[:, 0, key] = bad
    Y = still.hybrid_attn_fwd(U.params_of(w), Q.abs() + 1, K, V)[0]
    assert bool(torch.isnan(Y[:, :2, key:]).all())
    assert bool(torch.isfinite(Y[:, :2, :key]).all()) and bool(torch.isfinite(Y[:, 2:]).all())


@pytest.mark.parametrize("d,B,N,k,budget", [
    # more items than CTAs: of 256 rows (d = 64) or 512; the last one of a head without a second query tile, with whole rows
    # only, with one row
    (64, 5, 300, 16, 0), (64, 5, 512, 64, 0), (64, 3, 641, 16, 64), (128, 5, 700, 16, 0), (128, 3, 700, 32, 64), (128, 3, 1024, 64, 0),
    (128, 3, 1025, 64, 0),
])
def test_items_of_a_cta_do_not_mix(d, B, N, k, budget):
    # A head's rows are those of the call with this head alone, bit for bit, whatever its CTAs worked on before.
    w = synth.Workload("t", B, 32, 32, d, N, 64, k, "bf16", "head_scale", 33)
    r = U.run_prefill(w, gate=k < 64, max_salient=budget)
    one = synth.Workload("t", 1, 1, 1, d, N, 64, k, "bf16", "head_scale", 33)
    p = U.params_of(one, max_salient=budget)
    for b, h in ((0, 0), (0, 31), (B // 2, 7), (B - 1, 30), (B - 1, 31)):
        x = [None if t is None else t[b: b + 1, h: h + 1].contiguous() for t in (r["Q"], r["K"], r["V"], r["G"])]
        Y, _, _ = still.hybrid_attn_fwd(p, x[0], x[1], x[2], r["Wq"][h: h + 1].contiguous(), r["Wk"][h: h + 1].contiguous(), G=x[3])
        assert torch.equal(Y[0, 0], r["Y"][b, h])


@pytest.mark.parametrize("d,C,N", [(64, 64, 900), (128, 64, 1000), (64, 128, 900), (128, 64, 2305)])
def test_score_tiles_of_a_cta(d, C, N):
    # several tiles for every CTA of the score kernel, in turn by its groups of warps: not as many for every CTA, and a ragged one
    # at the end of every head
    w = synth.Workload("t", 2, 32, 8, d, N, C, C // 4, "bf16", "head_scale", 35)
    r = U.run_prefill(w)
    heads = [(0, 0), (0, 13), (1, 7), (1, 31)]
    U.check_selection(r["scores"], r["sel"], C, C // 4, heads)
    U.check_outputs(w, r["Q"], r["K"], r["V"], r["Wq"], r["Wk"], r["Y"], r["scores"], r["sel"], heads[1:], rows=U.sample_rows(N, 100, C))


def _items_as_alone(d, B, N, C, k, df):
    # More items than CTAs (pairs), of few tiles each: the rows of every sequence are those of the call with this sequence alone, where
    # a CTA has one item, bit for bit, and every wait ended.
    w = synth.Workload("t", B, 32, 32, d, N, C, k, "bf16", "head_scale", 37)
    Q, K, V = synth.make_qkv(w, "cuda")
    G = synth.make_gate(w, "cuda")
    g = torch.Generator(device="cuda").manual_seed(8)
    Wq, Wk = ((torch.randn(32, d, df, generator=g, device="cuda") * 0.05).bfloat16() for _ in range(2))

    def run(b0, b1):
        p = still.StillParams(b1 - b0, 32, 32, d, C, k, torch.bfloat16, d_f=df, sm_scale=w.sm_scale)
        ws = torch.empty(still.workspace_bytes(p, N), dtype=torch.uint8, device="cuda")
        x = [t[b0:b1].contiguous() for t in (Q, K, V, G)]
        Y = still.hybrid_attn_fwd(p, *x[:3], Wq, Wk, G=x[3] if k < C else None, workspace=ws)[0]
        assert still.device_status(ws) == (0, 0)
        return Y

    Y = run(0, B)
    for b in range(B):
        assert torch.equal(Y[b], run(b, b + 1)[0])


@pytest.mark.parametrize("N", [200, 600])
def test_short_items_of_a_pair(N):
    # five ring entries: the first CTA's producer can be through with an item while the second has not seen that it may begin with it
    _items_as_alone(128, 5, N, 64, 16, 128)


@pytest.mark.parametrize("d,B,N,C,k,df", [
    # without a linear branch, with one part, with two; no token kept; CTAs that get two items, and three
    (64, 10, 1, 64, 64, 64), (64, 5, 100, 64, 64, 64), (64, 10, 100, 64, 16, 32), (64, 10, 128, 64, 16, 64), (64, 10, 129, 64, 64, 64),
    (64, 10, 200, 64, 0, 64), (64, 5, 200, 64, 16, 32), (64, 10, 300, 64, 0, 64), (64, 10, 300, 128, 128, 64), (64, 10, 384, 64, 64, 64),
    (64, 10, 384, 128, 32, 64),
    (128, 5, 1, 64, 16, 128), (128, 5, 100, 64, 64, 128), (128, 5, 100, 64, 16, 32), (128, 10, 128, 64, 16, 128), (128, 5, 129, 128, 128, 128),
    (128, 10, 200, 64, 64, 128), (128, 5, 200, 64, 16, 32), (128, 10, 250, 128, 128, 128), (128, 5, 256, 64, 0, 128), (128, 5, 600, 64, 0, 64),
    (128, 5, 600, 64, 64, 128),
])
def test_short_items_of_a_cta(d, B, N, C, k, df):
    # one to three key tiles: the producers can be ahead of the softmax and the output warps by more than an item
    _items_as_alone(d, B, N, C, k, df)
