// fp32 FMA kernels of the STILL layer: the path for fp32 inputs and for bf16
// shapes the tensor-core kernels do not cover.  Arithmetic is fp32 throughout;
// T is the storage type of Q/K/V/G/W/Y and of the NP-Map features kept in the
// workspace.
//
// All of them are register-tiled products over shared memory: a thread owns a tile
// of outputs and takes 16-byte pieces of its rows, so that one shared-memory access
// serves 8 or more multiply-adds, and the multiply-adds are the packed form (two per
// instruction), which leaves issue slots for the loads.  At B = 1, H = 32, d = 64 and
// 2000 tokens a quarter of which stays selected (4.5 G multiply-adds, 120 us at the
// FMA pipes' rate) the layer took 1930 us with one shared-memory access per operand
// and a scan over the chunks in one block per 32 value columns; see each kernel.
#pragma once
#include "still_common.cuh"

namespace still {

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16 *p) {
    const uint2 r = *reinterpret_cast<const uint2 *>(p);
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                       __uint_as_float(r.y & 0xffff0000u));
}
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ void st4(__nv_bfloat16 *p, float4 v) {
    st_f(p, v.x); st_f(p + 1, v.y); st_f(p + 2, v.z); st_f(p + 3, v.w);
}
__device__ __forceinline__ float2 lo2(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4 &v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float2 dup2(float x) { return make_float2(x, x); }
// Four values of a row into shared memory: fp32 rows as an asynchronous copy, bf16 rows converted on the way.
__device__ __forceinline__ void stage4(float *dst, const float *src, bool valid) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    const int bytes = valid ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void stage4(float *dst, const __nv_bfloat16 *src, bool valid) {
    *reinterpret_cast<float4 *>(dst) = valid ? ld4(src) : make_float4(0.f, 0.f, 0.f, 0.f);
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Self-Saliency Score (Sec. 3.1) + per-chunk top-k (Sec. 3.3, delayed selection).
// One block per (chunk, head, batch): 8 (16) warps take the logits of 32 (64) rows at a time
// against the keys their windows cover: a warp owns four rows of a group of 32, a lane NJ =
// C / 32 + 1 keys of each.  Then the warp scores its tokens: lane j holds the logits of
// window slots j, j+32, ...; slot C-1 is the token itself (window_score).
// Selection: rank under (score descending, position ascending), NaN as -inf;
// the k best are written in ascending position order, -1 padded.
// ---------------------------------------------------------------------------
template <int NJ, bool kWide>
struct ScorePlan {
    static constexpr int C = 32 * (NJ - 1), kThreads = kWide && C > 32 ? 512 : 256, kRows = kThreads / 8;   // rows of a pass
    static size_t smem(int d) { return ((size_t)(2 * C + kRows) * (d + 4) + (size_t)kRows * (C + 33) + C) * 4 + (size_t)C * 4; }
};
template <typename T, int NJ, bool kWide>
__device__ __forceinline__ void score_block(const T *Q, const T *K, float *scores, int32_t *sel_idx, int c, int h, int b, int H, int Hkv,
                                            long long N, int d, int lam, float scale, float eps) {
    using P = ScorePlan<NJ, kWide>;
    constexpr int C = P::C, kThreads = P::kThreads, kRows = P::kRows;
    extern __shared__ __align__(16) float smem[];
    const int kv = h / (H / Hkv), ds = d + 4;
    const long long base = (long long)c * C, Tn = (N + C - 1) / C;
    float *kbuf = smem;                       // [2C][d + 4]: previous chunk, then this chunk
    float *qbuf = kbuf + 2 * C * ds;          // [kRows][d + 4]
    float *lg = qbuf + kRows * ds;            // [kRows][C + 33]
    float *sc = lg + kRows * (C + 33);        // [C]
    int *flag = reinterpret_cast<int *>(sc + C);  // [C]
    const T *Qh = Q + ((long long)b * H + h) * N * d;
    const T *Kh = K + ((long long)b * Hkv + kv) * N * d;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, d4 = d >> 2;

    for (int i = threadIdx.x; i < 2 * C * d4; i += kThreads) {
        const int row = i / d4, col = (i - row * d4) * 4;
        const long long pos = base - C + row;
        const bool in = pos >= 0 && pos < N;
        stage4(kbuf + row * ds + col, Kh + (in ? pos * d : 0) + col, in);
    }
    for (int p0 = 0; p0 < C; p0 += kRows) {
        if (base + p0 >= N) {   // (rows past the end of a ragged chunk)
            if (threadIdx.x < kRows) sc[p0 + threadIdx.x] = 0.f;
            continue;
        }
        for (int i = threadIdx.x; i < kRows * d4; i += kThreads) {
            const int row = i / d4, col = (i - row * d4) * 4;
            const long long pos = base + p0 + row;
            stage4(qbuf + row * ds + col, Qh + (pos < N ? pos * d : 0) + col, pos < N);
        }
        stage_commit();
        stage_wait();
        __syncthreads();
        // rows p0 + 4 warp + i, keys (rows of kbuf) r0 + lane + 32 j, where r0 starts the group of 32 rows
        const int r0 = p0 + (warp >> 3) * 32, in_group = 4 * (warp & 7);
        float2 acc[4][NJ];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < NJ; ++j) acc[i][j] = make_float2(0.f, 0.f);
        const float *qr = qbuf + 4 * warp * ds, *kr = kbuf + (r0 + lane) * ds;
#pragma unroll 4
        for (int x = 0; x < d; x += 4) {
            float4 q[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) q[i] = *reinterpret_cast<const float4 *>(qr + i * ds + x);
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const float4 k = *reinterpret_cast<const float4 *>(kr + 32 * j * ds + x);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    acc[i][j] = __ffma2_rn(lo2(q[i]), lo2(k), acc[i][j]);
                    acc[i][j] = __ffma2_rn(hi2(q[i]), hi2(k), acc[i][j]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < NJ; ++j) lg[(4 * warp + i) * (C + 33) + lane + 32 * j] = (acc[i][j].x + acc[i][j].y) * scale;
        __syncwarp();   // a warp scores the rows it has the logits of
#pragma unroll (kWide ? 4 : 1)   // (wide: four rows' chains of shuffles side by side)
        for (int i = 0; i < 4; ++i) {
            const int r = r0 + in_group + i;
            if (base + r >= N) {
                if (lane == 0) sc[r] = 0.f;
                continue;
            }
            float l[4];
#pragma unroll
            for (int s = 0; s < 4; ++s) {   // slot lane + 32 s is row r + 1 + slot of kbuf
                const int slot = lane + 32 * s;
                l[s] = s < NJ - 1 && base + r - (C - 1) + slot >= 0 ? lg[(4 * warp + i) * (C + 33) + in_group + i + 1 + slot] : -INFINITY;
            }
            const float s = window_score(l, lane, NJ - 1, C, eps);
            if (lane == 0) {
                sc[r] = s;
                if (scores) scores[((long long)b * H + h) * N + base + r] = s;
            }
        }
        __syncthreads();
    }
    __syncthreads();
    if (lam <= 0) return;

    const int n_c = (int)((N - base < C) ? (N - base) : C);
    select_chunk(sc, flag, n_c, C, lam, base, sel_idx + (((long long)b * H + h) * Tn + c) * lam);
}
template <typename T, int NJ>
__global__ void __launch_bounds__(256)
score_select_kernel(const T *Q, const T *K, float *scores,
                    int32_t *sel_idx, int *status, int H, int Hkv, long long N, int d, int lam, float scale, float eps) {
    grid_dep_wait();
    grid_dep_launch();
    clear_status(status);
    score_block<T, NJ, false>(Q, K, scores, sel_idx, blockIdx.x, blockIdx.y, blockIdx.z, H, Hkv, N, d, lam, scale, eps);
}

// ---------------------------------------------------------------------------
// Norm-Preserved Feature Map (Sec. 3.2, Eq. feature_map) of every row of X.
// u = f(x) ||x|| / ||f(x)||, f(x) = xW + b; phi = [softmax(u), softmax(-u)].
// kThreads / 4 rows a block as a product with W; thread (tr, tc) owns four rows and
// DF / 16 features, the sixteen threads of a row form its norms, extrema and sums.
// (2000 tokens x 40 heads: 38 us; a warp per row: 159 us.)
// ---------------------------------------------------------------------------
inline size_t npmap_smem(int d, int df, int threads) { return ((size_t)d * df + (size_t)(threads / 4) * (d + 4)) * 4; }
template <typename T, int DF, int kThreads>
__device__ __forceinline__ void npmap_block(const T *X, const T *W, const T *bias, T *phi, uint32_t rb, int hd, int b, int heads, long long N,
                                            int d) {
    constexpr int kRows = kThreads / 4;
    constexpr int VC = DF >= 64 ? 4 : 2, NV = DF / (16 * VC);   // columns VC (tc + 16 j) .. + VC
    extern __shared__ __align__(16) float smem[];
    const int ds = d + 4, d4 = d >> 2;
    float *Ws = smem;             // [d][DF]
    float *xs = Ws + d * DF;      // [kRows][d + 4]
    const int tid = threadIdx.x, tr = tid >> 4, tc = tid & 15;
    const T *Wh = W + (long long)hd * d * DF;
    const long long row0 = (long long)rb * kRows, head0 = ((long long)b * heads + hd) * N;
    for (int i = tid; i < d * DF / 4; i += kThreads) stage4(Ws + 4 * i, Wh + 4 * i, true);
    for (int i = tid; i < kRows * d4; i += kThreads) {
        const int r = i / d4, col = (i - r * d4) * 4;
        const bool in = row0 + r < N;
        stage4(xs + r * ds + col, X + (head0 + (in ? row0 + r : 0)) * d + col, in);
    }
    stage_commit();
    stage_wait();
    __syncthreads();
    float f[4][NV * VC];
#pragma unroll
    for (int j = 0; j < NV; ++j)
#pragma unroll
        for (int e = 0; e < VC; ++e) {
            const float bv = bias ? ld_f(bias + (long long)hd * DF + VC * (tc + 16 * j) + e) : 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) f[i][j * VC + e] = bv;
        }
#pragma unroll 2
    for (int x = 0; x < d; x += 4) {
        float4 q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = *reinterpret_cast<const float4 *>(xs + (4 * tr + i) * ds + x);
#pragma unroll
        for (int xx = 0; xx < 4; ++xx) {
            float2 w[NV * VC / 2];
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                const float *wr = Ws + (x + xx) * DF + VC * (tc + 16 * j);
                if constexpr (VC == 4) {
                    const float4 v = *reinterpret_cast<const float4 *>(wr);
                    w[2 * j] = lo2(v);
                    w[2 * j + 1] = hi2(v);
                } else {
                    w[j] = *reinterpret_cast<const float2 *>(wr);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 qq = dup2(xx == 0 ? q[i].x : xx == 1 ? q[i].y : xx == 2 ? q[i].z : q[i].w);
#pragma unroll
                for (int j = 0; j < NV * VC / 2; ++j) {
                    const float2 r = __ffma2_rn(qq, w[j], make_float2(f[i][2 * j], f[i][2 * j + 1]));
                    f[i][2 * j] = r.x;
                    f[i][2 * j + 1] = r.y;
                }
            }
        }
    }
    auto over_row = [](float v, auto op) {   // over the sixteen threads of a row
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
        return v;
    };
    auto add = [](float a, float c) { return a + c; };
    auto mx = [](float a, float c) { return fmaxf(a, c); };
    auto mn = [](float a, float c) { return fminf(a, c); };
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const long long row = row0 + 4 * tr + i;
        float nx2 = 0.f, nf2 = 0.f, umax = -INFINITY, umin = INFINITY;
        for (int x = tc; x < d; x += 16) {
            const float v = xs[(4 * tr + i) * ds + x];
            nx2 = fmaf(v, v, nx2);
        }
#pragma unroll
        for (int j = 0; j < NV * VC; ++j) nf2 = fmaf(f[i][j], f[i][j], nf2);
        nx2 = over_row(nx2, add);
        nf2 = over_row(nf2, add);
        const float ratio = sqrtf(nx2) / fmaxf(sqrtf(nf2), 1e-12f);
#pragma unroll
        for (int j = 0; j < NV * VC; ++j) {
            f[i][j] *= ratio;
            umax = fmaxf(umax, f[i][j]);
            umin = fminf(umin, f[i][j]);
        }
        umax = over_row(umax, mx);
        umin = over_row(umin, mn);
        float p[NV * VC], n[NV * VC], zp = 0.f, zn = 0.f;
#pragma unroll
        for (int j = 0; j < NV * VC; ++j) {
            p[j] = expf(f[i][j] - umax);
            n[j] = expf(umin - f[i][j]);
            zp += p[j];
            zn += n[j];
        }
        zp = over_row(zp, add);
        zn = over_row(zn, add);
        if (row < N) {
            T *pr = phi + (head0 + row) * 2 * DF;
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                T *dst = pr + VC * (tc + 16 * j);
                if constexpr (VC == 4) {
                    st4(dst, make_float4(p[4 * j] / zp, p[4 * j + 1] / zp, p[4 * j + 2] / zp, p[4 * j + 3] / zp));
                    st4(dst + DF, make_float4(n[4 * j] / zn, n[4 * j + 1] / zn, n[4 * j + 2] / zn, n[4 * j + 3] / zn));
                } else {
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        st_f(dst + e, p[2 * j + e] / zp);
                        st_f(dst + DF + e, n[2 * j + e] / zn);
                    }
                }
            }
        }
    }
}
// grid (ceil(N/64), heads, B)
template <typename T, int DF>
__global__ void __launch_bounds__(256, DF == 128 ? 2 : 3)
npmap_kernel(const T *X, const T *W, const T *bias,
             T *phi, int heads, long long N, int d) {
    grid_dep_wait();
    grid_dep_launch();
    npmap_block<T, DF, 256>(X, W, bias, phi, blockIdx.x, blockIdx.y, blockIdx.z, heads, N, d);
}

// ---------------------------------------------------------------------------
// The score and the two feature maps, which need nothing of one another, in one launch: blocks of the score first, which take
// longest, then those of Q, then of K.  For calls of few blocks (kFrontBlocks), which wait for one another's chains: 4 heads x
// 512 tokens 15 + 7 + 7 us in three launches, 12 in one.
// ---------------------------------------------------------------------------
template <typename T>
struct FrontArgs {
    const T *Q, *K, *Wq, *bq, *Wk, *bk;
    T *phiQ, *phiK;
    float *scores;
    int32_t *sel_idx;
    int *status;
    long long N;
    int B, H, Hkv, d, lam, n_score, n_q, row_blocks;   // n_score, n_q: blocks of the score, of phi(Q)
    float scale, eps;
};
template <typename T, int NJ, int DF>
__global__ void __launch_bounds__(ScorePlan<NJ, true>::kThreads)
score_npmap_kernel(const __grid_constant__ FrontArgs<T> a) {
    grid_dep_wait();
    grid_dep_launch();
    clear_status(a.status);
    using P = ScorePlan<NJ, true>;
    int i = blockIdx.x;
    if (i < a.n_score) {
        const int Tn = (int)((a.N + P::C - 1) / P::C), bh = i / Tn;
        score_block<T, NJ, true>(a.Q, a.K, a.scores, a.sel_idx, i - bh * Tn, bh % a.H, bh / a.H, a.H, a.Hkv, a.N, a.d, a.lam, a.scale, a.eps);
        return;
    }
    i -= a.n_score;
    const bool q = i < a.n_q;
    if (!q) i -= a.n_q;
    const int heads = q ? a.H : a.Hkv, unit = i / a.row_blocks;
    npmap_block<T, DF, P::kThreads>(q ? a.Q : a.K, q ? a.Wq : a.Wk, q ? a.bq : a.bk, q ? a.phiQ : a.phiK, i - unit * a.row_blocks, unit % heads,
                                 unit / heads, heads, a.N, a.d);
}

// ---------------------------------------------------------------------------
// Linear-attention branch (Algorithm 1 "Linear Attention Branch"; Eq.
// cache_routing_sum) as a two-level scan over the chunks of one (batch, head).  The
// chunks are cut into n_seg segments that run side by side.  Before chunk c is
// answered, chunk c-2 is folded:  S += sum_{i in M^LA_{c-2}} phi_k(k_i)^T v_i,
// z += sum phi_k(k_i)^T;  then N_LA = (phi_q(q) S) . g and D_LA = phi_q(q) z for the
// rows of chunk c.
//   sum_only = 1: what segment blockIdx.y folds, into sums (blockIdx.y < n_seg - 1)
//   sum_only = 0: the scan of a segment, from sums made exclusive prefixes by
//                 la_prefix_kernel
// The sums may lie in the segment's own rows of N_LA and D_LA (SegSums): a block takes
// its columns of them into registers before it writes any of its rows.
// grid (B*H, segments, d / 64), 256 threads: thread (tf, te) owns DP / 16 features x
// four of the block's 64 value columns of S in registers; for the read-out S passes
// through shared memory and a thread owns four rows x four columns of N_LA.  The same
// 2000 tokens: 32 + 71 us and 5 us for the prefix, against 833 us for the scan of all
// chunks by one block per 32 value columns.
// Final S, z go to the decode state when asked.
// ---------------------------------------------------------------------------
struct SegSums {   // of segment seg of head bh: S [DP][d] at S + bh S_bh + seg S_seg, z [DP] at z + bh z_bh + seg z_seg
    float *S, *z;
    long long S_bh, S_seg, z_bh, z_seg;
};
inline size_t la_seg_smem(int dp) { return ((size_t)64 * dp + 64 * 64 + (size_t)dp * 64 + dp) * 4 + 64 * 4 + 16; }
template <typename T, int DP>
__global__ void __launch_bounds__(256)
la_seg_kernel(const T *phiQ, const T *phiK, const T *V,
              const T *G, const int32_t *sel_idx, float *N_LA,
              float *D_LA, SegSums sums, float *S_out,
              float *z_out, int H, int Hkv, long long N, int d, int C, int lam, int seg_chunks,
              int n_seg, int sum_only) {
    grid_dep_wait();
    grid_dep_launch();
    constexpr int FPT = DP / 16;
    extern __shared__ __align__(16) float smem[];
    float *ph = smem;                 // [64][DP] feature rows of the current sub-tile
    float *vs = ph + 64 * DP;         // [64][64]
    float *Ss = vs + 64 * 64;         // [DP][64]
    float *zs = Ss + DP * 64;         // [DP]
    int *list = reinterpret_cast<int *>(zs + DP);   // [64] tokens of the sub-tile to fold; their number
    int *n_list = list + 64;
    const int bh = blockIdx.x, seg = blockIdx.y, b = bh / H, h = bh % H, kv = h / (H / Hkv);
    const int e0 = blockIdx.z * 64, tid = threadIdx.x, te = tid & 15, tf = tid >> 4, warp = tid >> 5, lane = tid & 31;
    const long long Tn = (N + C - 1) / C;
    const T *pq = phiQ + (long long)bh * N * DP;
    const T *pk = phiK + ((long long)b * Hkv + kv) * N * DP;
    const T *vh = V + ((long long)b * Hkv + kv) * N * d;
    float *mine_S = sums.S + bh * sums.S_bh + seg * sums.S_seg, *mine_z = sums.z + bh * sums.z_bh + seg * sums.z_seg;
    float2 S[FPT / 2][4];   // features tf * FPT + 2 i, + 1; columns e0 + 4 te + e
#pragma unroll
    for (int i = 0; i < FPT / 2; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) S[i][e] = make_float2(0.f, 0.f);
    for (int i = tid; i < DP; i += 256) zs[i] = 0.f;
    if (!sum_only && seg > 0) {
#pragma unroll
        for (int i = 0; i < FPT / 2; ++i) {
            const float4 a = ld4(mine_S + (long long)(tf * FPT + 2 * i) * d + e0 + 4 * te);
            const float4 c = ld4(mine_S + (long long)(tf * FPT + 2 * i + 1) * d + e0 + 4 * te);
            S[i][0] = make_float2(a.x, c.x);
            S[i][1] = make_float2(a.y, c.y);
            S[i][2] = make_float2(a.z, c.z);
            S[i][3] = make_float2(a.w, c.w);
        }
        if (blockIdx.z == 0)   // (z is used by these blocks alone, which also write the rows of D_LA that it may lie in)
            for (int i = tid; i < DP; i += 256) zs[i] = mine_z[i];
        __syncthreads();       // the sums are taken before any row is written
    }
    const int W = C < 64 ? C : 64;    // tokens of a sub-tile
    const long long c1 = seg == n_seg - 1 ? Tn : (long long)(seg + 1) * seg_chunks;
    for (long long c = (long long)seg * seg_chunks; c < c1; ++c) {
        if (c >= 2) {
            const long long ub = (c - 2) * C;  // chunk c-2 is complete
            const int32_t *si = sel_idx + ((long long)bh * Tn + (c - 2)) * lam;
            for (int sub = 0; sub < C; sub += W) {
                __syncthreads();
                if (warp == 0) {   // the sub-tile's tokens that were not selected, in order
                    int n = 0;
                    uint64_t out = 0;   // bit r: token sub + r was selected
                    for (int i = lane; i < lam; i += 32) {
                        const long long r = si[i] - ub - sub;
                        if (r >= 0 && r < W) out |= 1ull << r;
                    }
                    const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)out), hi = __reduce_or_sync(0xffffffffu, (uint32_t)(out >> 32));
                    for (int r0 = 0; r0 < W; r0 += 32) {
                        const uint32_t keep = ~(r0 == 0 ? lo : hi);
                        if ((keep >> lane) & 1u) list[n + __popc(keep & ((1u << lane) - 1u))] = sub + r0 + lane;
                        n += __popc(keep);
                    }
                    if (lane == 0) *n_list = n;
                }
                __syncthreads();
                const int n = *n_list;
                for (int i = tid; i < n * (DP / 4); i += 256) {
                    const int row = i / (DP / 4), col = (i % (DP / 4)) * 4;
                    stage4(ph + row * DP + col, pk + (ub + list[row]) * DP + col, true);
                }
                for (int i = tid; i < n * 16; i += 256) {
                    const int row = i >> 4, col = (i & 15) * 4;
                    stage4(vs + row * 64 + col, vh + (ub + list[row]) * d + e0 + col, true);
                }
                stage_commit();
                stage_wait();
                __syncthreads();
#pragma unroll 2
                for (int i = 0; i < n; ++i) {
                    const float4 v = *reinterpret_cast<const float4 *>(vs + i * 64 + 4 * te);
                    const float2 v2[4] = {dup2(v.x), dup2(v.y), dup2(v.z), dup2(v.w)};
#pragma unroll
                    for (int q = 0; q < FPT / 4; ++q) {
                        const float4 p = *reinterpret_cast<const float4 *>(ph + i * DP + tf * FPT + 4 * q);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            S[2 * q][e] = __ffma2_rn(lo2(p), v2[e], S[2 * q][e]);
                            S[2 * q + 1][e] = __ffma2_rn(hi2(p), v2[e], S[2 * q + 1][e]);
                        }
                    }
                }
                if (tid < DP) {
                    float a = zs[tid];
                    for (int i = 0; i < n; ++i) a += ph[i * DP + tid];
                    zs[tid] = a;
                }
            }
        }
        if (sum_only) continue;
        if (c < 2) {   // nothing has left the local region yet: the branch is zero
            for (long long i = tid; i < (long long)C * 16; i += 256) {
                const long long pos = c * C + i / 16;
                if (pos < N) st4(N_LA + ((long long)bh * N + pos) * d + e0 + (i % 16) * 4, make_float4(0.f, 0.f, 0.f, 0.f));
            }
            if (blockIdx.z == 0)
                for (int r = tid; r < C; r += 256)
                    if (c * C + r < N) D_LA[(long long)bh * N + c * C + r] = 0.f;
            continue;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < FPT / 2; ++i) {
            *reinterpret_cast<float4 *>(Ss + (tf * FPT + 2 * i) * 64 + 4 * te) = make_float4(S[i][0].x, S[i][1].x, S[i][2].x, S[i][3].x);
            *reinterpret_cast<float4 *>(Ss + (tf * FPT + 2 * i + 1) * 64 + 4 * te) = make_float4(S[i][0].y, S[i][1].y, S[i][2].y, S[i][3].y);
        }
        for (int sub = 0; sub < C; sub += W) {
            const long long base = c * C + sub;
            if (base >= N) break;
            const int rows = (int)min((long long)W, N - base);
            if (sub > 0) __syncthreads();
            for (int i = tid; i < rows * (DP / 4); i += 256) {
                const int row = i / (DP / 4), col = (i % (DP / 4)) * 4;
                stage4(ph + row * DP + col, pq + (base + row) * DP + col, true);
            }
            stage_commit();
            stage_wait();
            __syncthreads();
            if (4 * tf < rows) {   // rows 4 tf .. + 3 (rows past the end hold stale features and are not stored)
                float4 gate[4];    // (requested ahead of the products and of the stores)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    gate[i] = G && 4 * tf + i < rows ? ld4(G + ((long long)bh * N + base + 4 * tf + i) * d + e0 + 4 * te) : make_float4(1.f, 1.f, 1.f, 1.f);
                float2 acc[4][2];
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
#pragma unroll 2
                for (int f = 0; f < DP; f += 4) {
                    float4 p[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) p[i] = *reinterpret_cast<const float4 *>(ph + (4 * tf + i) * DP + f);
#pragma unroll
                    for (int ff = 0; ff < 4; ++ff) {
                        const float4 s = *reinterpret_cast<const float4 *>(Ss + (f + ff) * 64 + 4 * te);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float2 pp = dup2(ff == 0 ? p[i].x : ff == 1 ? p[i].y : ff == 2 ? p[i].z : p[i].w);
                            acc[i][0] = __ffma2_rn(pp, lo2(s), acc[i][0]);
                            acc[i][1] = __ffma2_rn(pp, hi2(s), acc[i][1]);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (4 * tf + i < rows) {
                        const long long o = ((long long)bh * N + base + 4 * tf + i) * d + e0 + 4 * te;
                        float4 v = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
                        if (G) v = make_float4(v.x * gate[i].x, v.y * gate[i].y, v.z * gate[i].z, v.w * gate[i].w);
                        st4(N_LA + o, v);
                    }
            }
            if (blockIdx.z == 0) {
                for (int r = warp; r < rows; r += 8) {
                    float acc = 0.f;
                    for (int f = lane; f < DP; f += 32) acc = fmaf(ph[r * DP + f], zs[f], acc);
                    acc = warp_sum(acc);
                    if (lane == 0) D_LA[(long long)bh * N + base + r] = acc;
                }
            }
        }
    }
    const bool last = !sum_only && seg == n_seg - 1;
    if (sum_only || (last && S_out)) {
        __syncthreads();
        float *So = sum_only ? mine_S : S_out + (long long)bh * DP * d, *zo = sum_only ? mine_z : z_out + (long long)bh * DP;
#pragma unroll
        for (int i = 0; i < FPT / 2; ++i) {
            st4(So + (long long)(tf * FPT + 2 * i) * d + e0 + 4 * te, make_float4(S[i][0].x, S[i][1].x, S[i][2].x, S[i][3].x));
            st4(So + (long long)(tf * FPT + 2 * i + 1) * d + e0 + 4 * te, make_float4(S[i][0].y, S[i][1].y, S[i][2].y, S[i][3].y));
        }
        if (blockIdx.z == 0)
            for (int i = tid; i < DP; i += 256) zo[i] = zs[i];
    }
}
// Segment s receives the sum of the segments before it (the last segment's own sum is not needed).  n_S = DP d / 4 and n_z =
// DP threads per head.
template <typename T>
__device__ __forceinline__ void prefix_over_segments(T *p, long long stride, int n_seg) {
    auto add = [](const T &a, const T &b) -> T {
        if constexpr (sizeof(T) == 16) return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
        else return a + b;
    };
    T run{};
    for (int s0 = 0; s0 < n_seg; s0 += 8) {   // eight independent loads in flight, then the running sum
        T v[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) v[s] = s0 + s < n_seg - 1 ? p[(s0 + s) * stride] : T{};
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            if (s0 + s < n_seg) p[(s0 + s) * stride] = run;
            run = add(run, v[s]);
        }
    }
}
__global__ void __launch_bounds__(256)
la_prefix_kernel(SegSums sums, int n_S, int n_z, long long n_threads, int n_seg) {
    grid_dep_wait();
    grid_dep_launch();
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    if (i >= n_threads) return;
    const long long bh = i / (n_S + n_z);
    const int r = (int)(i - bh * (n_S + n_z));
    if (r < n_S) prefix_over_segments(reinterpret_cast<float4 *>(sums.S + bh * sums.S_bh) + r, sums.S_seg / 4, n_seg);
    else prefix_over_segments(sums.z + bh * sums.z_bh + (r - n_S), sums.z_seg, n_seg);
}

// ---------------------------------------------------------------------------
// Softmax-attention branch + merge (Algorithm 1 "Softmax Attention Branch" and
// the output line; Sec. 3.3 merge equation).  One block of 16 ROWS / RT threads per
// ROWS queries of a chunk, head and batch.  The keys of chunk c are the selected tokens of
// chunks 0..c-2 (through sel_idx), all of chunk c-1 and the causal part of chunk c;
// they pass through two buffers of KT keys.  Thread (ty, tx) owns RT rows: of the
// logits the keys tx, tx + 16, ..., of the output the columns 4 tx .. + 3 (and + 64).
// The rows' probabilities go from one product to the other through shared memory that
// only the half warp of the row reads.  Bound by shared-memory reads (57 % of the rate, issue slots 53 %):
// 32 heads x 2000 tokens, d = 64, a quarter selected take 250 us with RT = 4 (16 warps an
// SM), 264 us with RT = 8 (8 warps); with one read per operand and multiply 756 us.
// Merge: with m the running max, ms = max(m, 0):
//   y = (o e^{m-ms} + e^{-ms} N_LA) / (l e^{m-ms} + e^{-ms} D_LA).
// ---------------------------------------------------------------------------
template <int D, int ROWS, int RT>
struct SaPlan {
    static constexpr int kThreads = ROWS / RT * 16;
    static constexpr int KT = D == 64 ? 64 : 32;
    static constexpr int kQ = 0, kK = ROWS * (D + 4), kV = kK + 2 * KT * (D + 4), kP = kV + 2 * KT * D;   // in floats
    static constexpr int kPos = kP + ROWS * (KT + 4);
    static constexpr int kBytes = (kPos + 2 * KT) * 4;
};
template <typename T, int D, int ROWS, int RT>
__global__ void __launch_bounds__(SaPlan<D, ROWS, RT>::kThreads)
sa_merge_kernel(const T *Q, const T *K, const T *V,
                const int32_t *sel_idx, const float *N_LA,
                const float *D_LA, T *Y, int H, int Hkv, long long N, int C,
                int lam, float scale) {
    grid_dep_wait();
    grid_dep_launch();
    using P = SaPlan<D, ROWS, RT>;
    constexpr int KT = P::KT, kThreads = P::kThreads, NK = KT / 16, NV = D / 64, DS = D + 4, PS = KT + 4;
    extern __shared__ __align__(16) float smem[];
    float *qs = smem + P::kQ, *ps = smem + P::kP;
    int *kpos = reinterpret_cast<int *>(smem + P::kPos);   // [2][KT]
    const int h = blockIdx.y, b = blockIdx.z, tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int kv = h / (H / Hkv);
    const long long row0 = (long long)(gridDim.x - 1 - blockIdx.x) * ROWS;   // the longest key streams first
    const long long c = row0 / C, Tn = (N + C - 1) / C, bh = (long long)b * H + h;
    const T *Qh = Q + bh * N * D;
    const T *Kh = K + ((long long)b * Hkv + kv) * N * D;
    const T *Vh = V + ((long long)b * Hkv + kv) * N * D;
    const int32_t *si = sel_idx + bh * Tn * lam;
    const long long n_sel = c >= 2 ? (c - 1) * lam : 0, loc0 = c >= 1 ? (c - 1) * C : 0;
    const long long loc1 = min(row0 + ROWS, N), L = n_sel + (loc1 - loc0);

    auto load_tile = [&](long long t0, int buf) {
        float *ks = smem + P::kK + buf * KT * DS, *vs = smem + P::kV + buf * KT * D;
        for (int i = tid; i < KT * (D / 4); i += kThreads) {
            const int row = i / (D / 4), col = (i % (D / 4)) * 4;
            const long long e = t0 + row;
            const long long p = e < n_sel ? (long long)si[e] : e < L ? loc0 + (e - n_sel) : -1;
            stage4(ks + row * DS + col, Kh + (p >= 0 ? p * D : 0) + col, p >= 0);
            stage4(vs + row * D + col, Vh + (p >= 0 ? p * D : 0) + col, p >= 0);
            if (col == 0) kpos[buf * KT + row] = (int)p;
        }
        stage_commit();
    };
    for (int i = tid; i < ROWS * (D / 4); i += kThreads) {
        const int row = i / (D / 4), col = (i % (D / 4)) * 4;
        const bool in = row0 + row < N;
        stage4(qs + row * DS + col, Qh + (in ? row0 + row : 0) * D + col, in);
    }
    load_tile(0, 0);
    float m[RT], l[RT];
    float2 o[RT][2 * NV];
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        m[r] = -INFINITY;
        l[r] = 0.f;
#pragma unroll
        for (int e = 0; e < 2 * NV; ++e) o[r][e] = make_float2(0.f, 0.f);
    }
    int buf = 0;
    for (long long t0 = 0; t0 < L; t0 += KT, buf ^= 1) {
        stage_wait();
        __syncthreads();   // the tile is there, and everybody has left the other buffer
        if (t0 + KT < L) load_tile(t0 + KT, buf ^ 1);
        const float *ks = smem + P::kK + buf * KT * DS, *vs = smem + P::kV + buf * KT * D;
        float2 acc[RT][NK];
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int j = 0; j < NK; ++j) acc[r][j] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int x = 0; x < D; x += 4) {
            float4 k[NK];
#pragma unroll
            for (int j = 0; j < NK; ++j) k[j] = *reinterpret_cast<const float4 *>(ks + (tx + 16 * j) * DS + x);
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                const float4 q = *reinterpret_cast<const float4 *>(qs + (ty * RT + r) * DS + x);
#pragma unroll
                for (int j = 0; j < NK; ++j) {
                    acc[r][j] = __ffma2_rn(lo2(q), lo2(k[j]), acc[r][j]);
                    acc[r][j] = __ffma2_rn(hi2(q), hi2(k[j]), acc[r][j]);
                }
            }
        }
        int kp[NK];
#pragma unroll
        for (int j = 0; j < NK; ++j) kp[j] = kpos[buf * KT + tx + 16 * j];
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            const long long t = row0 + ty * RT + r;
            float s[NK], mx = -INFINITY;
#pragma unroll
            for (int j = 0; j < NK; ++j) {
                s[j] = kp[j] >= 0 && kp[j] <= t ? (acc[r][j].x + acc[r][j].y) * scale : -INFINITY;
                mx = max_nan(mx, s[j]);
            }
#pragma unroll
            for (int w = 8; w > 0; w >>= 1) mx = max_nan(mx, __shfl_xor_sync(0xffffffffu, mx, w));
            const float mnew = max_nan(m[r], mx);
            const float alpha = mnew == -INFINITY ? 1.f : expf(m[r] - mnew);
            m[r] = mnew;
            float sum = 0.f;
#pragma unroll
            for (int j = 0; j < NK; ++j) {
                const float p = kp[j] >= 0 && kp[j] <= t && mnew != -INFINITY ? expf(s[j] - mnew) : 0.f;
                sum += p;
                ps[(ty * RT + r) * PS + tx + 16 * j] = p;
            }
            l[r] = l[r] * alpha + sum;   // (this thread's keys only)
#pragma unroll
            for (int e = 0; e < 2 * NV; ++e) o[r][e] = __fmul2_rn(o[r][e], dup2(alpha));
        }
        __syncwarp();
#pragma unroll 1
        for (int k = 0; k < KT; k += 4) {
            float4 p[RT];
#pragma unroll
            for (int r = 0; r < RT; ++r) p[r] = *reinterpret_cast<const float4 *>(ps + (ty * RT + r) * PS + k);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
#pragma unroll
                for (int e = 0; e < NV; ++e) {
                    const float4 v = *reinterpret_cast<const float4 *>(vs + (k + kk) * D + 64 * e + 4 * tx);
#pragma unroll
                    for (int r = 0; r < RT; ++r) {
                        const float2 pp = dup2(kk == 0 ? p[r].x : kk == 1 ? p[r].y : kk == 2 ? p[r].z : p[r].w);
                        o[r][2 * e] = __ffma2_rn(pp, lo2(v), o[r][2 * e]);
                        o[r][2 * e + 1] = __ffma2_rn(pp, hi2(v), o[r][2 * e + 1]);
                    }
                }
            }
        }
        __syncwarp();
    }
    float dlas[RT];
    float4 nla[RT][NV];   // the linear branch's rows, requested together
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        const long long t = row0 + ty * RT + r;
        dlas[r] = D_LA && t < N ? D_LA[bh * N + t] : 0.f;
#pragma unroll
        for (int e = 0; e < NV; ++e) nla[r][e] = dlas[r] > 0.f ? ld4(N_LA + (bh * N + t) * D + 64 * e + 4 * tx) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        const long long t = row0 + ty * RT + r;
#pragma unroll
        for (int w = 8; w > 0; w >>= 1) l[r] += __shfl_xor_sync(0xffffffffu, l[r], w);
        if (t >= N) continue;
        const float dla = dlas[r];
        float fs = 1.f, fl = 0.f;
        if (dla > 0.f) {
            const float ms = fmaxf(m[r], 0.f);
            fs = expf(m[r] - ms);
            fl = expf(-ms);
        }
        const float den = l[r] * fs + fl * dla;
#pragma unroll
        for (int e = 0; e < NV; ++e) {
            const long long oidx = (bh * N + t) * D + 64 * e + 4 * tx;
            float4 num = make_float4(o[r][2 * e].x * fs, o[r][2 * e].y * fs, o[r][2 * e + 1].x * fs, o[r][2 * e + 1].y * fs);
            if (dla > 0.f) {
                const float4 n = nla[r][e];
                num = make_float4(num.x + fl * n.x, num.y + fl * n.y, num.z + fl * n.z, num.w + fl * n.w);
            }
            st4(Y + oidx, make_float4(num.x / den, num.y / den, num.z / den, num.w / den));
        }
    }
}

}  // namespace still
