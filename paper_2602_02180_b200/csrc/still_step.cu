// Decode: one step of the Recurrent Form (Sec. 3.3) on the decode state.
//
//   step_route  : (one step in chunk) when the new token opens a chunk, the chunk that has just left the two-chunk
//                 local region is routed (Eq. delayed_selection, Eq. cache_routing_sum): top-k positions into
//                 sel_idx, every other token into (S, z) through the NP-Map.
//   step_main   : everything that reads much: the split-KV pass over the salient cache h_t (selected rows of the
//                 routed chunks + the local region; one partial (max, sum, numerator) per block and KV group) and the
//                 linear branch's read-out phi(q) (S, z).  The pass leaves the new token's logits against its window.
//   step_merge  : combines the partials under one denominator, y = (N_SA + N_LA) / (D_SA + D_LA), appends (k_t, v_t) to
//                 the history, scores the new token (Sec. 3.1) and counts it.
//
// A step of a small batch is bound by latency, not by bytes, so the three are launched with programmatic stream
// serialization: a kernel's blocks are resident before its predecessor has ended and wait for it in
// griddepcontrol.wait.  Every block of every kernel executes that wait, so the end of a kernel still implies the end
// of all before it; and nothing is read before the wait.
#include "still_common.cuh"
#include "still_step_f32.cuh"
#include "still_step_mma.cuh"
#include "still_tc.h"

#include <algorithm>
#include <type_traits>

namespace still {

// Records of a head in the scratch of the state, d + 2 floats each: partials of the history, the linear branch, and in
// the last two the new token's logits against its window (at most 128).
constexpr int kRecords = 33, kMaxSplits = 30, kLinRecord = 30, kLogitRecord = 31;
constexpr int kStepThreads = kStepWarps * 32;

long long state_kv_rows(const still_params_t *p, long long capacity) {
    if (p->max_salient <= 0 || p->topk <= 0) return capacity;
    const long long window = p->max_salient / p->topk;   // chunks whose selections stay cached
    return std::min<long long>(capacity, (window + 3) * p->chunk);
}

size_t step_scratch_bytes(const still_params_t *p, long long) {
    return (size_t)p->B * p->H * kRecords * (p->d + 2) * sizeof(float);
}

// What a step expects to find in the header of the decode state.
struct StateKey {
    int32_t B, H, Hkv, d, d_f, chunk, topk, dtype;
    long long cap, t;
};

// Header words 0-13 against the call: 0 if they agree, else a detail code (1: token count, 2: not a
// state / other layout version, 3: built with other parameters or another capacity, 4: an earlier step
// has already failed).  Nothing writes these words while the first kernel of a step runs.
__device__ __forceinline__ int state_mismatch(const int32_t *words, const StateKey &k) {
    const int4 *w4 = reinterpret_cast<const int4 *>(words);   // (four loads in flight, not a chain of comparisons)
    const int4 w0 = w4[0], w1 = w4[1], w2 = w4[2], w3 = w4[3];
    const int32_t hdr[16] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w, w2.x, w2.y, w2.z, w2.w, w3.x, w3.y, w3.z, w3.w};
    if (hdr[0] != 0x5354494c || hdr[1] != 1) return 2;
    if (hdr[2] != k.B || hdr[3] != k.H || hdr[4] != k.Hkv || hdr[5] != k.d || hdr[6] != k.d_f || hdr[7] != k.chunk ||
        hdr[8] != k.topk || hdr[9] != k.dtype)
        return 3;
    const long long cap = ((long long)hdr[11] << 32) | (unsigned int)hdr[10];
    if (cap != k.cap) return 3;
    if (hdr[14] != 0) return 4;
    const long long have = ((long long)hdr[13] << 32) | (unsigned int)hdr[12];
    return have != k.t ? 1 : 0;
}

// fp32 states; grid (H, B), 256 threads.  Routes chunk cr (complete, C tokens): top-k into sel_idx / sel_mask, the other tokens
// into (S, z).  With a salient-cache budget of `window` chunks the selected tokens of chunk cr - window leave the
// cache at the same moment and are folded into (S, z) as well.
__global__ void __launch_bounds__(256)
step_route_kernel(float *kc, float *vc, float *score,
                  int32_t *sel_idx, uint32_t *sel_mask, float *S,
                  float *z, float *Wk, float *bk, int32_t *hdr, StateKey key,
                  int H, int Hkv, long long cap, long long kvr, int d, int df, int C, int lam, long long cr, int window,
                  int w_in_smem) {
    extern __shared__ __align__(16) float smem[];
    grid_dep_wait();
    grid_dep_launch();
    {   // the step's first kernel when there is a chunk to route: the header against the call
        const int bad = state_mismatch(hdr, key);
        if (bad != 0) {
            if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && bad != 4)
                report_status(hdr + 14, STILL_ERR_STATE_MISMATCH, bad);
            return;
        }
    }
    const int dp = 2 * df;
    float *ph = smem;                 // [C][dp]
    float *vs = ph + C * dp;          // [C][d]
    float *xs = vs + C * d;           // [8][d]
    float *sc = xs + 8 * d;           // [C]
    int *flag = reinterpret_cast<int *>(sc + C);  // [C]
    float *Ws = reinterpret_cast<float *>(flag + C);  // [d][df] the head's W_k (read once per row of the chunk otherwise)
    const int h = blockIdx.x, b = blockIdx.y, kv = h / (H / Hkv);
    const long long bh = (long long)b * H + h;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < C; i += blockDim.x) {
        sc[i] = score[bh * cap + cr * C + i];
        flag[i] = 0;
    }
    __syncthreads();
    if (lam > 0) select_chunk(sc, flag, C, C, lam, cr * C, sel_idx + (bh * (cap / C) + cr) * lam);
    __syncthreads();
    if (threadIdx.x < C / 32) {  // the same selection as bit masks (read by the split-KV pass)
        uint32_t bits = 0u;
        for (int j = 0; j < 32; ++j) bits |= (flag[threadIdx.x * 32 + j] ? 1u : 0u) << j;
        sel_mask[(bh * (cap / C) + cr) * (C / 32) + threadIdx.x] = bits;
    }
    const float *Wh = Wk + (long long)kv * d * df;
    const float *bh_ = bk ? bk + (long long)kv * df : nullptr;
    float *Sh = S + bh * dp * d;
    const float *Wuse = Wh;   // W_k from shared memory when it fits beside the chunk's tiles, else from global memory
    if (w_in_smem && (lam < C || window > 0)) {
        for (int i = threadIdx.x; i < d * df; i += blockDim.x) Ws[i] = Wh[i];
        Wuse = Ws;
    }
    // pass 0: the unselected tokens of chunk cr; pass 1: the selected tokens of the chunk that leaves the cache
    for (int pass = 0; pass < 2; ++pass) {
        const long long chunk = pass == 0 ? cr : cr - window;
        if (pass == 0 ? lam >= C : (window <= 0 || chunk < 0)) continue;   // nothing to fold in this pass
        __syncthreads();
        if (pass == 1) {   // fold[r] = 1 for the tokens to fold: here the chunk's selected ones, recorded when it was routed
            for (int i = threadIdx.x; i < C; i += blockDim.x)
                flag[i] = !((sel_mask[(bh * (cap / C) + chunk) * (C / 32) + i / 32] >> (i & 31)) & 1u);
            __syncthreads();
        }
        const long long base = chunk * C;
        const float *kh = kc + (((long long)b * Hkv + kv) * kvr + base % kvr) * d;   // (a chunk never straddles the ring's end)
        const float *vh = vc + (((long long)b * Hkv + kv) * kvr + base % kvr) * d;
        for (int i = threadIdx.x; i < C * d; i += blockDim.x) vs[i] = vh[i];
        float *xw = xs + warp * d;
        for (int r = warp; r < C; r += 8) {   // flag[r] != 0: the token stays out of this pass
            float ep[4], en[4];
            if (!flag[r]) {
                for (int i = lane; i < d; i += 32) xw[i] = kh[(long long)r * d + i];
                __syncwarp();
                npmap_row(xw, Wuse, bh_, d, df, lane, ep, en);
            }
#pragma unroll
            for (int jj = 0; jj < 4; ++jj)
                if (jj < (df >> 5)) {
                    int j = lane + 32 * jj;
                    ph[r * dp + j] = flag[r] ? 0.f : ep[jj];
                    ph[r * dp + df + j] = flag[r] ? 0.f : en[jj];
                }
            __syncwarp();
        }
        __syncthreads();
        // S[f][e] += sum_i phi[i][f] v[i][e]: a thread owns 4 features x 8 value columns at a time, so that a token
        // costs 3 shared-memory reads for 32 multiply-adds
        for (int blk = threadIdx.x; blk < (dp / 4) * (d / 8); blk += blockDim.x) {
            const int f0 = (blk / (d / 8)) * 4, e0 = (blk % (d / 8)) * 8;
            float acc[4][8];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[a][c] = Sh[(f0 + a) * d + e0 + c];
            for (int i = 0; i < C; ++i) {
                const float4 pf = *reinterpret_cast<const float4 *>(ph + i * dp + f0);
                const float4 v0 = *reinterpret_cast<const float4 *>(vs + i * d + e0);
                const float4 v1 = *reinterpret_cast<const float4 *>(vs + i * d + e0 + 4);
                const float pa[4] = {pf.x, pf.y, pf.z, pf.w};
                const float vv[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int c = 0; c < 8; ++c) acc[a][c] = fmaf(pa[a], vv[c], acc[a][c]);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < 8; ++c) Sh[(f0 + a) * d + e0 + c] = acc[a][c];
        }
        for (int f = threadIdx.x; f < dp; f += blockDim.x) {
            float acc = z[bh * dp + f];
            for (int i = 0; i < C; ++i) acc += ph[i * dp + f];
            z[bh * dp + f] = acc;
        }
    }
}

// The same for bf16 states on the tensor cores; grid (H, B), 256 threads.  f = K W_k and S += phi(K)^T V are bf16
// products with fp32 accumulation (the features are bf16 in the prefill as well); f is kept in fp32 and a row of f is
// replaced in place by the row's features, zero for a token that stays out.  The chunk's sum is formed by itself and
// then added to the state in fp32: carried through the accumulators, the state would take their rounding (not to
// nearest) sixteen tokens at a time for a whole generation.  What bounds it is the read and write of S (128 KB a head each way) and, for
// few heads, the chain of loads, two products and the row-wise softmax.  (A quarter kept, C = 64, d = 128: 512 heads 70 us,
// 1024 heads with a chunk leaving the cache as well 235 us, 32 heads 25 us; on the FMA pipes 416, 1168 and 95 us.)
template <int D>
struct RoutePlan {
    int k, v, w, f, sc, flag, total;   // byte offsets
    __host__ __device__ RoutePlan(int C, int df) {
        k = 0;
        v = k + C * D * 2;
        w = v + C * D * 2;
        f = w + D * df * 2;              // f [C][df] fp32, then phi [C][2 df] bf16
        sc = f + C * df * 4;
        flag = sc + C * 4;
        total = flag + C * 4;
    }
};
template <int D>
__global__ void __launch_bounds__(256)
step_route_mma_kernel(__nv_bfloat16 *kc, __nv_bfloat16 *vc, float *score, int32_t *sel_idx, uint32_t *sel_mask, float *S,
                      float *z, __nv_bfloat16 *Wk, __nv_bfloat16 *bk, int32_t *hdr, StateKey key, int H, int Hkv, long long cap,
                      long long kvr, int df, int C, int lam, long long cr, int window) {
    extern __shared__ __align__(128) uint8_t route_smem[];
    grid_dep_wait();
    grid_dep_launch();
    {   // the step's first kernel when there is a chunk to route: the header against the call
        const int bad = state_mismatch(hdr, key);
        if (bad != 0) {
            if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && bad != 4)
                report_status(hdr + 14, STILL_ERR_STATE_MISMATCH, bad);
            return;
        }
    }
    const RoutePlan<D> plan(C, df);
    uint8_t *ks = route_smem + plan.k, *vs = route_smem + plan.v, *ws = route_smem + plan.w, *fs = route_smem + plan.f;
    float *sc = reinterpret_cast<float *>(route_smem + plan.sc);
    int *flag = reinterpret_cast<int *>(route_smem + plan.flag);
    const int h = blockIdx.x, b = blockIdx.y, kv = h / (H / Hkv), dp = 2 * df;
    const long long bh = (long long)b * H + h, row0 = (long long)b * Hkv + kv;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tig = lane & 3;
    // 16-byte pieces of a row are swizzled by the row: ldmatrix reads eight rows of one piece without conflicts
    constexpr int kRowB = D * 2, kPieces = D / 8;
    const int w_pieces = df / 8, f_row = df * 4;
    auto w_off = [&](int row, int piece) { return row * df * 2 + ((w_pieces >= 8 ? piece ^ (row & 7) : piece ^ ((row >> 1) & 3)) << 4); };

    const bool fold0 = lam < C, fold1 = window > 0 && cr >= window;
    auto load_chunk = [&](long long chunk) {   // (a chunk never straddles the ring's end)
        const long long r = chunk * C % kvr;
        const __nv_bfloat16 *kh = kc + (row0 * kvr + r) * D, *vh = vc + (row0 * kvr + r) * D;
        for (int i = tid; i < C * kPieces; i += 256) {
            const int row = i / kPieces, piece = i % kPieces, dst = row * kRowB + ((piece ^ (row & 7)) << 4);
            cp_async16(ks + dst, kh + (long long)row * D + piece * 8, true);
            cp_async16(vs + dst, vh + (long long)row * D + piece * 8, true);
        }
    };
    if (fold0 || fold1) {
        for (int i = tid; i < D * w_pieces; i += 256) {
            const int row = i / w_pieces, piece = i % w_pieces;
            cp_async16(ws + w_off(row, piece), Wk + ((long long)kv * D + row) * df + piece * 8, true);
        }
        load_chunk(fold0 ? cr : cr - window);
    }
    cp_async_commit();
    for (int i = tid; i < C; i += 256) {
        sc[i] = score[bh * cap + cr * C + i];
        flag[i] = 0;
    }
    __syncthreads();
    if (lam > 0) select_chunk(sc, flag, C, C, lam, cr * C, sel_idx + (bh * (cap / C) + cr) * lam);
    __syncthreads();
    if (tid < C / 32) {  // the same selection as bit masks (read by the split-KV pass)
        uint32_t bits = 0u;
        for (int j = 0; j < 32; ++j) bits |= (flag[tid * 32 + j] ? 1u : 0u) << j;
        sel_mask[(bh * (cap / C) + cr) * (C / 32) + tid] = bits;
    }
    for (int pass = 0; pass < 2; ++pass) {   // the unselected tokens of chunk cr; the selected ones of the chunk that leaves
        if (!(pass == 0 ? fold0 : fold1)) continue;
        __syncthreads();
        if (pass == 1) {
            const long long chunk = cr - window;
            if (fold0) {
                load_chunk(chunk);
                cp_async_commit();
            }
            for (int i = tid; i < C; i += 256)
                flag[i] = !((sel_mask[(bh * (cap / C) + chunk) * (C / 32) + i / 32] >> (i & 31)) & 1u);
        }
        cp_async_wait<0>();
        __syncthreads();
        // f = K W_k: 16 tokens x 32 features at a time
        for (int u = warp; u < (C / 16) * (df / 32); u += 8) {
            const int mt = u / (df / 32), n0 = u % (df / 32) * 32;
            float acc[4][4] = {};
#pragma unroll
            for (int k16 = 0; k16 < D / 16; ++k16) {
                uint32_t af[4], bf[4];
                const int arow = mt * 16 + ((lane >> 3) & 1) * 8 + (lane & 7), apiece = k16 * 2 + (lane >> 4);
                ldmatrix_x4(af, ks + arow * kRowB + ((apiece ^ (arow & 7)) << 4));
#pragma unroll
                for (int np = 0; np < 2; ++np) {
                    ldmatrix_x4_trans(bf, ws + w_off(k16 * 16 + ((lane >> 3) & 1) * 8 + (lane & 7), n0 / 8 + np * 2 + (lane >> 4)));
                    mma_16816(acc[np * 2], af, bf[0], bf[1]);
                    mma_16816(acc[np * 2 + 1], af, bf[2], bf[3]);
                }
            }
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int hr = 0; hr < 2; ++hr) {
                    const int row = mt * 16 + g + hr * 8, col = n0 + nt * 8 + tig * 2;
                    *reinterpret_cast<float2 *>(fs + row * f_row + (((col >> 2) ^ (row & 7)) << 4) + (col & 3) * 4) =
                        make_float2(acc[nt][hr * 2], acc[nt][hr * 2 + 1]);
                }
        }
        __syncthreads();
        // a warp per row: u = f ||x|| / ||f||, phi = [softmax(u), softmax(-u)], rounded as the prefill stores it
        for (int r = warp; r < C; r += 8) {
            const bool out = flag[r] != 0;   // the token stays out of this pass
            float f[4], ep[4], en[4];
            float nx2 = 0.f, nf2 = 0.f, umax = -INFINITY, umin = INFINITY;
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                f[jj] = 0.f;
                if (jj * 32 < df) {
                    const int j = lane + 32 * jj;
                    f[jj] = *reinterpret_cast<const float *>(fs + r * f_row + (((j >> 2) ^ (r & 7)) << 4) + (j & 3) * 4);
                    if (bk) f[jj] += ld_f(bk + (long long)kv * df + j);
                    nf2 = fmaf(f[jj], f[jj], nf2);
                }
                if (jj * 32 < D) {
                    const int j = lane + 32 * jj;
                    const float x = ld_f(reinterpret_cast<const __nv_bfloat16 *>(ks + r * kRowB + (((j >> 3) ^ (r & 7)) << 4)) + (j & 7));
                    nx2 = fmaf(x, x, nx2);
                }
            }
            nx2 = warp_sum(nx2);
            nf2 = warp_sum(nf2);
            const float ratio = sqrtf(nx2) / fmaxf(sqrtf(nf2), 1e-12f);
#pragma unroll
            for (int jj = 0; jj < 4; ++jj)
                if (jj * 32 < df) {
                    f[jj] *= ratio;
                    umax = fmaxf(umax, f[jj]);
                    umin = fminf(umin, f[jj]);
                }
            umax = warp_max(umax);
            umin = warp_min(umin);
            float zp = 0.f, zn = 0.f;
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                ep[jj] = en[jj] = 0.f;
                if (jj * 32 < df) {
                    ep[jj] = expf(f[jj] - umax);
                    en[jj] = expf(umin - f[jj]);
                    zp += ep[jj];
                    zn += en[jj];
                }
            }
            zp = warp_sum(zp);   // (also: every lane has read its f before any lane overwrites the row)
            zn = warp_sum(zn);
#pragma unroll
            for (int jj = 0; jj < 4; ++jj)
                if (jj * 32 < df) {
                    const int j = lane + 32 * jj, jn = df + j;
                    st_f(reinterpret_cast<__nv_bfloat16 *>(fs + r * f_row + (((j >> 3) ^ (r & 7)) << 4)) + (j & 7), out ? 0.f : ep[jj] / zp);
                    st_f(reinterpret_cast<__nv_bfloat16 *>(fs + r * f_row + (((jn >> 3) ^ (r & 7)) << 4)) + (jn & 7), out ? 0.f : en[jj] / zn);
                }
        }
        __syncthreads();
        // S += phi^T V: 16 features x 64 value columns at a time
        for (int u = warp; u < (dp / 16) * (D / 64); u += 8) {
            const int mt = u / (D / 64), e0 = u % (D / 64) * 64;
            float acc[8][4] = {};
            float2 lo[8], hi[8];   // the state, requested ahead of the products
            float *Sr = S + (bh * dp + mt * 16 + g) * D + e0 + tig * 2;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                lo[nt] = *reinterpret_cast<const float2 *>(Sr + nt * 8);
                hi[nt] = *reinterpret_cast<const float2 *>(Sr + 8 * D + nt * 8);
            }
            for (int k16 = 0; k16 < C / 16; ++k16) {
                uint32_t af[4], bf[4];
                const int arow = k16 * 16 + (lane >> 4) * 8 + (lane & 7), apiece = mt * 2 + ((lane >> 3) & 1);
                ldmatrix_x4_trans(af, fs + arow * f_row + ((apiece ^ (arow & 7)) << 4));
                const int brow = k16 * 16 + ((lane >> 3) & 1) * 8 + (lane & 7);
#pragma unroll
                for (int np = 0; np < 4; ++np) {
                    const int bpiece = e0 / 8 + np * 2 + (lane >> 4);
                    ldmatrix_x4_trans(bf, vs + brow * kRowB + ((bpiece ^ (brow & 7)) << 4));
                    mma_16816(acc[np * 2], af, bf[0], bf[1]);
                    mma_16816(acc[np * 2 + 1], af, bf[2], bf[3]);
                }
            }
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                *reinterpret_cast<float2 *>(Sr + nt * 8) = make_float2(lo[nt].x + acc[nt][0], lo[nt].y + acc[nt][1]);
                *reinterpret_cast<float2 *>(Sr + 8 * D + nt * 8) = make_float2(hi[nt].x + acc[nt][2], hi[nt].y + acc[nt][3]);
            }
        }
        for (int f = tid; f < dp; f += 256) {
            float acc = 0.f;
            for (int r = 0; r < C; ++r)
                acc += ld_f(reinterpret_cast<const __nv_bfloat16 *>(fs + r * f_row + (((f >> 3) ^ (r & 7)) << 4)) + (f & 7));
            z[bh * dp + f] += acc;
        }
    }
    cp_async_wait<0>();
}

template <uint32_t kRegs>
__device__ __forceinline__ void reg_inc_step() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegs)); }
template <uint32_t kRegs>
__device__ __forceinline__ void reg_dec_step() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegs)); }

// Arguments of step_main_kernel / step_merge_kernel.  (Their contents come from kernels that may still run when a block
// becomes resident, and must not be loaded ahead of the wait: see grid_dep_wait.)
template <typename T>
struct StepArgs {
    T *kc, *vc;
    float *score;
    uint32_t *sel_mask;
    float *S, *z, *part;
    int32_t *hdr;
    T *q, *k, *v, *g, *Wq, *bq, *y;
    StateKey key;
    AttendView view;             // view.rep: query heads of a KV group
    long long cap, kvr, t;
    int B, H, Hkv, df, la;
    float eps;
    // Plan.  A unit is what shares its K / V rows: the query heads of one (batch, KV head) (fp32: up to four of them).
    // The units' tiles form one line of units * unit_len, of which block i takes [i * per, (i + 1) * per): blocks that
    // divide the line evenly, whatever the number of groups.  unit_len is the number of tiles of a unit, or that
    // rounded up so that no block has tiles of two units.  Items: the linear read-outs, one per (batch, query head).
    int heads_per_unit, units_per_group, tiles, unit_len, per, total;
    int first_item_block, n_items;   // blocks from first_item_block on share the items evenly
    int item_warps;                  // warps that work on an item together
};

// First block that works on unit u, and how many do.
__device__ __forceinline__ int unit_first_block(int per, int unit_len, int u) { return u * unit_len / per; }
__device__ __forceinline__ int unit_blocks(int per, int unit_len, int tiles, int u) {
    return (u * unit_len + tiles - 1) / per - u * unit_len / per + 1;
}

// Eight (bf16) or four (fp32) consecutive values as fp32.
__device__ __forceinline__ void load16(const __nv_bfloat16 *p, float (&o)[8]) {
    const uint4 r = *reinterpret_cast<const uint4 *>(p);
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        o[2 * i] = __uint_as_float(w[i] << 16);
        o[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}
__device__ __forceinline__ void load16(const float *p, float (&o)[4]) {
    const float4 r = *reinterpret_cast<const float4 *>(p);
    o[0] = r.x; o[1] = r.y; o[2] = r.z; o[3] = r.w;
}

// Read-outs are worked on by groups of NW warps (1, 2 or all 8 of a block).
template <int NW, bool kOthers = false>
__device__ __forceinline__ void group_sync() {
    if constexpr (NW == 1) __syncwarp();
    else if constexpr (NW == kStepWarps) step_sync<kOthers>();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)(threadIdx.x >> 5) / NW), "n"(NW * 32) : "memory");
}
// Shared memory of a group beside the rings, in floats: q [D], phi [2 d_f], sums of z [8], partial sums [NW][D].
constexpr int kItemFloats = 128 + 256 + 8;
constexpr int kItemSmem = kStepWarps * (kItemFloats + 128) * 4;

// phi(q) [softmax(u), softmax(-u)] of a row by a warp, from its f + b: lane j holds features j, j + 32, ...  nx2: ||q||^2.  The
// features are rounded to the storage type, as the prefill stores them.
template <typename T>
__device__ __forceinline__ void features_of_row(float (&f)[4], float nx2, int df, float *ph) {
    const int lane = threadIdx.x & 31, jpl = df >> 5;
    float nf2 = 0.f, umax = -INFINITY, umin = INFINITY;
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) nf2 += f[jj] * f[jj];
    nf2 = warp_sum(nf2);
    const float ratio = sqrtf(nx2) / fmaxf(sqrtf(nf2), 1e-12f);
#pragma unroll
    for (int jj = 0; jj < 4; ++jj)
        if (jj < jpl) {
            f[jj] *= ratio;
            umax = fmaxf(umax, f[jj]);
            umin = fminf(umin, f[jj]);
        }
    umax = warp_max(umax);
    umin = warp_min(umin);
    float zp = 0.f, zn = 0.f, ep[4], en[4];
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
        ep[jj] = en[jj] = 0.f;
        if (jj < jpl) {
            ep[jj] = expf(f[jj] - umax);
            en[jj] = expf(umin - f[jj]);
            zp += ep[jj];
            zn += en[jj];
        }
    }
    zp = warp_sum(zp);
    zn = warp_sum(zn);
    if (ph == nullptr) return;
#pragma unroll
    for (int jj = 0; jj < 4; ++jj)
        if (jj < jpl) {
            T p0, p1;
            st_f(&p0, ep[jj] / zp);
            st_f(&p1, en[jj] / zn);
            ph[lane + 32 * jj] = ld_f(&p0);
            ph[df + lane + 32 * jj] = ld_f(&p1);
        }
}

// Linear read-out of one (batch, query head): N_LA = phi(q) S, D_LA = phi(q) z into the head's last record.  S [2 d_f, D]
// fp32 (128 KB at d = d_f = 128) and W_q are what it costs.  A warp takes a contiguous slice of either through its
// cp.async ring, first W_q, then S, so that the whole ring is in flight also while phi(q) is formed.  (With the rows
// requested into registers instead, a warp had too little in flight: 512 read-outs took 60 us, 1.1 TB/s.)
// Of a read-out apart (kApart), which a step of few sequences waits for, state_ok() is asked before anything of the state is read,
// but behind the requests for q and W_q.  (One user, 2000 tokens: 10.5 us a step with the header first, 10.0 like this.)
template <typename T, int D, int NW, bool kApart, class Ring, class StateOk>
__device__ __forceinline__ void linear_item(const StepArgs<T> &a, long long bh, uint8_t *ring, float *smem, StateOk state_ok) {
    constexpr int V = 16 / (int)sizeof(T);
    constexpr int LPR = D / 4, RPW = 32 / LPR;        // lanes per row of S (16 bytes each), rows per warp and load
    constexpr int kStage = Ring::kStage, kStages = Ring::kStages;
    const int warp = (threadIdx.x >> 5) % NW, lane = threadIdx.x & 31, tid = warp * 32 + lane;
    const int df = a.df, dp = 2 * df, h = (int)(bh % a.H), jpl = df >> 5;
    float *qs = smem, *ph = qs + D, *redz = ph + 256, *red = redz + 8;
    const int w_bytes = D * df * (int)sizeof(T) / NW, s_bytes = dp * D * 4 / NW;   // this warp's slices
    const int n_w = (w_bytes + kStage - 1) / kStage, n_s = (s_bytes + kStage - 1) / kStage;
    const char *w_src = reinterpret_cast<const char *>(a.Wq + (long long)h * D * df) + (long long)warp * w_bytes;
    const char *s_src = reinterpret_cast<const char *>(a.S + bh * dp * D) + (long long)warp * s_bytes;
    auto issue = [&](int c) {
        if (c < n_w + n_s) {
            const bool is_w = c < n_w;
            const int off = (is_w ? c : c - n_w) * kStage, bytes = min(kStage, (is_w ? w_bytes : s_bytes) - off);
            const char *src = (is_w ? w_src : s_src) + off;
            uint8_t *dst = ring + c % kStages * kStage;
#pragma unroll 4
            for (int i = lane * 16; i < bytes; i += 512) cp_async16(dst + i, src + i, true);
        }
        cp_async_commit();
    };
    if constexpr (kApart) {
        const int early = min(n_w, kStages);
        for (int c = 0; c < early; ++c) issue(c);
        for (int i = tid; i < D; i += NW * 32) qs[i] = ld_f(a.q + bh * D + i);
        if (!state_ok()) {
            cp_async_wait<0>();
            return;
        }
        for (int c = early; c < kStages; ++c) issue(c);
    } else {
#pragma unroll
        for (int c = 0; c < kStages; ++c) issue(c);
        for (int i = tid; i < D; i += NW * 32) qs[i] = ld_f(a.q + bh * D + i);
    }
    float dz = 0.f, zv[8];
#pragma unroll
    for (int i = 0; i < 8 / NW + (8 % NW ? 1 : 0); ++i) zv[i] = tid + i * NW * 32 < dp ? a.z[bh * dp + tid + i * NW * 32] : 0.f;
    group_sync<NW>();
    auto norm2_of_q = [&] {
        float x2 = 0.f;
        for (int i = lane; i < D; i += 32) x2 += qs[i] * qs[i];
        return warp_sum(x2);
    };
    float nx2 = 0.f;
    if constexpr (kApart) nx2 = norm2_of_q();   // (while W_q comes in)
    {   // f = q W_q: 16 bytes of a row per lane
        const int lpr = df / V, rpl = 32 / lpr, cg = lane % lpr;
        float acc[V];
#pragma unroll
        for (int e = 0; e < V; ++e) acc[e] = 0.f;
        for (int c = 0; c < n_w; ++c) {
            cp_async_wait<kStages - 1>();
            __syncwarp();
            const T *wr = reinterpret_cast<const T *>(ring + c % kStages * kStage) + cg * V;
            const int r0 = (warp * w_bytes + c * kStage) / (df * (int)sizeof(T));
            const int rows = min(kStage, w_bytes - c * kStage) / (df * (int)sizeof(T));
#pragma unroll 4
            for (int r = lane / lpr; r < rows; r += rpl) {
                float w[V];
                load16(wr + r * df, w);
                const float x = qs[r0 + r];
#pragma unroll
                for (int e = 0; e < V; ++e) acc[e] = fmaf(x, w[e], acc[e]);
            }
            __syncwarp();
            issue(c + kStages);
        }
        for (int o = lpr; o < 32; o <<= 1) {
#pragma unroll
            for (int e = 0; e < V; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
        }
        if (lane < lpr) {
#pragma unroll
            for (int e = 0; e < V; ++e) red[warp * df + cg * V + e] = acc[e];
        }
        group_sync<NW>();
    }
    {   // every warp forms the norms and sums
        float f[4];
        if constexpr (!kApart) nx2 = norm2_of_q();
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            f[jj] = 0.f;
            if (jj < jpl) {
                if (a.bq) f[jj] = ld_f(a.bq + (long long)h * df + lane + 32 * jj);
#pragma unroll
                for (int w = 0; w < NW; ++w) f[jj] += red[w * df + lane + 32 * jj];
            }
        }
        features_of_row<T>(f, nx2, df, warp == 0 ? ph : nullptr);
        group_sync<NW>();
    }
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c = n_w; c < n_w + n_s; ++c) {
        cp_async_wait<kStages - 1>();
        __syncwarp();
        const int off = (c - n_w) * kStage, rows = min(kStage, s_bytes - off) / (D * 4);
        const float *sr = reinterpret_cast<const float *>(ring + c % kStages * kStage) + lane * 4;
        const float *pr = ph + (warp * s_bytes + off) / (D * 4) + lane / LPR;
#pragma unroll 4
        for (int r = 0; r < rows; r += RPW) {
            const float4 x = *reinterpret_cast<const float4 *>(sr + r * D);
            const float p = pr[r];
            acc.x = fmaf(p, x.x, acc.x);
            acc.y = fmaf(p, x.y, acc.y);
            acc.z = fmaf(p, x.z, acc.z);
            acc.w = fmaf(p, x.w, acc.w);
        }
        __syncwarp();
        issue(c + kStages);
    }
    cp_async_wait<0>();
    if constexpr (RPW == 2) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 16);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 16);
        acc.z += __shfl_xor_sync(0xffffffffu, acc.z, 16);
        acc.w += __shfl_xor_sync(0xffffffffu, acc.w, 16);
    }
    if (lane < LPR) *reinterpret_cast<float4 *>(red + warp * D + lane * 4) = acc;
#pragma unroll
    for (int i = 0; i < 8 / NW + (8 % NW ? 1 : 0); ++i)
        if (tid + i * NW * 32 < dp) dz = fmaf(ph[tid + i * NW * 32], zv[i], dz);
    dz = warp_sum(dz);
    if (lane == 0) redz[warp] = dz;
    group_sync<NW>();
    float *rec = a.part + (bh * kRecords + kLinRecord) * (D + 2);
    for (int i = tid; i < D; i += NW * 32) {
        float n = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) n += red[w * D + i];
        rec[2 + i] = n;
    }
    if (tid == 0) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) s += redz[w];
        rec[1] = s;
    }
    group_sync<NW>();
}

// This block's share of the read-outs, by groups of NW warps, from the first-th of the block on: its j-th is item j * blocks +
// (its place among the blocks), and belongs to group j % groups.
template <typename T, int D, int NW, bool kApart, class Ring, class StateOk>
__device__ __forceinline__ void work_on_items(const StepArgs<T> &a, uint8_t *smem, int first, StateOk state_ok) {
    constexpr int kGroups = kStepWarps / NW;
    const int warp = threadIdx.x >> 5, group = warp / NW, blocks = (int)gridDim.x - a.first_item_block;
    float *mine = reinterpret_cast<float *>(smem + Ring::kTotal) + group * (kItemFloats + NW * 128);
    for (int j = group; ; j += kGroups) {
        const long long i = (int)blockIdx.x - a.first_item_block + (long long)j * blocks;
        if (i >= a.n_items) break;
        if (j >= first) linear_item<T, D, NW, kApart, Ring>(a, i, smem + warp * Ring::kWarp, mine, state_ok);
    }
}

// ---- bf16: the features of the block's first read-outs are formed by four warps of their own while the eight others work on the
// cache, so that these have nothing left to do for a read-out but to stream S.  (As a chain of q, W_q, phi(q) and S behind the
// cache pass a read-out took 7 of its 21 us before S came in at the rate of HBM.  us a step, then and now, d = 128, a quarter
// kept: 4 sequences of 32 heads x 2000 tokens 18.2 and 17.1, 8 x 4000 35.5 and 33.5, 32 x 8192 capped at 448 71.9 and 69.1; 64 of 16
// heads x 3000 82.7 and 81.4.)
constexpr int kMapWarps = 4, kMaxPhi = 14;   // features kept per block (a KB each beside the rings); read-outs beyond: work_on_items
// Shared memory behind the rings, in bytes: read-outs (kItemSmem), features, the map warps' q.
constexpr int kPhiAt = kItemSmem, kMapAt = kPhiAt + kMaxPhi * 256 * 4, kBesideSmem = kMapAt + kMapWarps * 128 * 4;
constexpr int kPhiBarrier = 15;   // (barriers 1 to 8: see group_sync)

// Features of the block's first read-outs, and their D_LA, by the map warps: f is the sum over rows in the order of linear_item
// by one warp.
template <int D>
__device__ __forceinline__ void map_items(const StepArgs<__nv_bfloat16> &a, uint8_t *beside) {
    using bf = __nv_bfloat16;
    const int mw = (threadIdx.x >> 5) - kStepWarps, lane = threadIdx.x & 31, df = a.df, dp = 2 * df, blocks = gridDim.x;
    float *qs = reinterpret_cast<float *>(beside + kMapAt) + mw * 128;
    const int lpr = df / 8, rpl = 32 / lpr, cg = lane % lpr;
    for (int j = mw; j < kMaxPhi; j += kMapWarps) {
        const long long bh = (int)blockIdx.x + (long long)j * blocks;
        if (bh >= a.n_items) break;
        const int h = (int)(bh % a.H);
        float *ph = reinterpret_cast<float *>(beside + kPhiAt) + j * 256;
        const bf *W = a.Wq + (long long)h * D * df + (lane / lpr) * df + cg * 8;
        float nx2 = 0.f;
        for (int i = lane; i < D; i += 32) {
            const float x = ld_f(a.q + bh * D + i);
            qs[i] = x;
            nx2 += x * x;
        }
        nx2 = warp_sum(nx2);
        __syncwarp();   // (q is read by other lanes than wrote it)
        float zv[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) zv[i] = lane + 32 * i < dp ? a.z[bh * dp + lane + 32 * i] : 0.f;
        float acc[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = 0.f;
        constexpr int kBatch = 8;   // rows of W_q requested together
        for (int r0 = 0; r0 < D; r0 += kBatch * rpl) {
            uint4 raw[kBatch];
#pragma unroll
            for (int k = 0; k < kBatch; ++k) raw[k] = *reinterpret_cast<const uint4 *>(W + (long long)(r0 + k * rpl) * df);
#pragma unroll
            for (int k = 0; k < kBatch; ++k) {
                const float x = qs[r0 + k * rpl + lane / lpr];
                const uint32_t w4[4] = {raw[k].x, raw[k].y, raw[k].z, raw[k].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    acc[2 * e] = fmaf(x, __uint_as_float(w4[e] << 16), acc[2 * e]);
                    acc[2 * e + 1] = fmaf(x, __uint_as_float(w4[e] & 0xffff0000u), acc[2 * e + 1]);
                }
            }
        }
        for (int o = lpr; o < 32; o <<= 1) {
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
        }
        __syncwarp();   // (every lane has read q)
        if (lane < lpr) {
#pragma unroll
            for (int e = 0; e < 8; ++e) qs[cg * 8 + e] = acc[e];
        }
        __syncwarp();
        float f[4];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) f[jj] = 32 * jj < df ? (a.bq ? ld_f(a.bq + (long long)h * df + lane + 32 * jj) : 0.f) + qs[lane + 32 * jj] : 0.f;
        features_of_row<bf>(f, nx2, df, ph);
        __syncwarp();
        float dz = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (lane + 32 * i < dp) dz = fmaf(ph[lane + 32 * i], zv[i], dz);
        dz = warp_sum(dz);
        if (lane == 0) a.part[(bh * kRecords + kLinRecord) * (D + 2) + 1] = dz;
    }
}

// The streams of S of the block's first read-outs, by groups of a.item_warps warps: request() is called when the warp's ring is
// free, run() when the features are there.
template <typename T, int D, class Ring>
struct StateStream {
    static constexpr int kStage = Ring::kStage, kStages = Ring::kStages, LPR = D / 4, RPW = 32 / LPR;
    const StepArgs<T> &a;
    uint8_t *ring;
    int group, in_group, groups;   // this warp's group, its place there; groups
    int s_bytes, n_s, total;       // this warp's slice of S, its stages; stages in all
    int requested = 0;
    __device__ __forceinline__ StateStream(const StepArgs<T> &args, uint8_t *smem)
        : a(args), ring(smem + (threadIdx.x >> 5) * Ring::kWarp) {
        group = (threadIdx.x >> 5) / a.item_warps;
        in_group = (threadIdx.x >> 5) % a.item_warps;
        groups = kStepWarps / a.item_warps;
        s_bytes = 2 * a.df * D * 4 / a.item_warps;
        n_s = (s_bytes + kStage - 1) / kStage;
        const int mine = (int)min((long long)kMaxPhi, (a.n_items - (int)blockIdx.x + (long long)gridDim.x - 1) / gridDim.x);   // of the block
        total = max(0, (mine - group + groups - 1) / groups) * n_s;
    }
    __device__ __forceinline__ long long item(int k) const {   // the group's k-th
        return (int)blockIdx.x + (long long)(group + k * groups) * gridDim.x;
    }
    __device__ __forceinline__ void issue() {
        if (requested < total) {
            const int k = requested / n_s, off = (requested - k * n_s) * kStage, bytes = min(kStage, s_bytes - off);
            const char *src = reinterpret_cast<const char *>(a.S + item(k) * 2 * a.df * D) + (long long)in_group * s_bytes + off;
            uint8_t *dst = ring + requested % kStages * kStage;
#pragma unroll 4
            for (int i = (threadIdx.x & 31) * 16; i < bytes; i += 512) cp_async16(dst + i, src + i, true);
        }
        ++requested;
        cp_async_commit();
    }
    __device__ __forceinline__ void request() {
#pragma unroll
        for (int c = 0; c < kStages; ++c) issue();
    }
    template <int NW>
    __device__ __forceinline__ void run(uint8_t *beside) {
        const int warp = in_group, lane = threadIdx.x & 31, tid = warp * 32 + lane;
        float *red = reinterpret_cast<float *>(beside) + group * NW * 128;
        for (int k = 0, c = 0; c < total; ++k) {
            const float *ph = reinterpret_cast<const float *>(beside + kPhiAt) + (group + k * groups) * 256 + warp * s_bytes / (D * 4) + lane / LPR;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int off = 0; off < s_bytes; off += kStage, ++c) {
                cp_async_wait<kStages - 1>();
                __syncwarp();
                const int rows = min(kStage, s_bytes - off) / (D * 4);
                const float *sr = reinterpret_cast<const float *>(ring + c % kStages * kStage) + lane * 4;
                const float *pr = ph + off / (D * 4);
#pragma unroll 4
                for (int r = 0; r < rows; r += RPW) {
                    const float4 x = *reinterpret_cast<const float4 *>(sr + r * D);
                    const float p = pr[r];
                    acc.x = fmaf(p, x.x, acc.x);
                    acc.y = fmaf(p, x.y, acc.y);
                    acc.z = fmaf(p, x.z, acc.z);
                    acc.w = fmaf(p, x.w, acc.w);
                }
                __syncwarp();
                issue();
            }
            if constexpr (RPW == 2) {
                acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 16);
                acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 16);
                acc.z += __shfl_xor_sync(0xffffffffu, acc.z, 16);
                acc.w += __shfl_xor_sync(0xffffffffu, acc.w, 16);
            }
            float *rec = a.part + (item(k) * kRecords + kLinRecord) * (D + 2) + 2;
            if constexpr (NW == 1) {
                if (lane < LPR) {
                    rec[lane * 4] = acc.x;       // (records are not 16-byte aligned)
                    rec[lane * 4 + 1] = acc.y;
                    rec[lane * 4 + 2] = acc.z;
                    rec[lane * 4 + 3] = acc.w;
                }
            } else {
                if (lane < LPR) *reinterpret_cast<float4 *>(red + warp * D + lane * 4) = acc;
                group_sync<NW, true>();
                for (int i = tid; i < D; i += NW * 32) {
                    float n = 0.f;
#pragma unroll
                    for (int w = 0; w < NW; ++w) n += red[w * D + i];
                    rec[i] = n;
                }
                group_sync<NW, true>();
            }
        }
        cp_async_wait<0>();
    }
};

// Rings of the cache pass.
template <typename T, int D>
struct StepRing : AttendPlan<D> {};
template <int D>
struct StepRing<float, D> : AttendPlanF32<D> {};
// What a block does beside its tiles: the read-outs apart have blocks of their own; or all share them, with map warps or without.
enum StepMode { kItemsApart, kItemsShared, kItemsMapped };
template <bool kMaps>
constexpr int kMainThreads = kStepThreads + (kMaps ? kMapWarps * 32 : 0);
// Shared memory of step_main_kernel: the rings, and what lies beside them.
template <typename T, int D, bool kMaps>
constexpr int step_main_smem() {
    return StepRing<T, D>::kTotal + (kMaps ? kBesideSmem : kItemSmem);
}
static_assert(step_main_smem<__nv_bfloat16, 128, true>() <= 232448 && step_main_smem<float, 128, false>() <= 232448, "shared memory of a step");

// One block per SM.  At large batches the bytes of K, V and S bound it (us a step, the merge included; in brackets the form
// with a launch each for append and score, routing, the cache pass in equal splits per group and the merge with its
// read-out, timed in turn on one box: B = 64, 32K prefix, every token 1302 (1657), 6.6 TB/s; B = 16, 16K, a quarter kept
// 148 (307); B = 32, 8K, capped at 448: 72 (203)), at one sequence the latency of a block's chain (one user, 2K prefix:
// 10.5 (72), of which the host needs 10).
template <typename T, int D, int NH, StepMode kMode>
__global__ void __launch_bounds__(kMode == kItemsMapped ? 512 : kStepThreads, 1)   // (512: 128 registers a thread, see below)
step_main_kernel(const __grid_constant__ StepArgs<T> a) {
    extern __shared__ __align__(128) uint8_t step_smem[];
    grid_dep_wait();
    grid_dep_launch();
    constexpr bool kMaps = kMode == kItemsMapped;
    using Ring = StepRing<T, D>;
    uint8_t *beside = step_smem + Ring::kTotal;
    // (a block with a read-out apart has no tiles, and compares the header itself)
    if (kMode != kItemsApart || (int)blockIdx.x < a.first_item_block) {   // the header against the call; on a mismatch nothing is written but the status word
        const int bad = state_mismatch(a.hdr, a.key);
        if (bad != 0) {
            if (blockIdx.x == 0 && threadIdx.x == 0 && bad != 4) report_status(a.hdr + 14, STILL_ERR_STATE_MISMATCH, bad);
            return;
        }
    }
    if constexpr (kMaps) {
        if (threadIdx.x >= kStepThreads) {
            reg_dec_step<64>();
            map_items<D>(a, beside);
            asm volatile("bar.arrive %0, %1;" ::"n"(kPhiBarrier), "n"(kMainThreads<kMaps>) : "memory");
            return;
        }
        // Per scheduler 2 x 160 + 64 registers, of the 3 x 128 that the block was launched with.  (The quarter of the register file
        // that is left over is what lets the blocks of the next kernel come in beside this one: with all of it taken a step was 4
        // us longer at 4 sequences, 12 at 32.)
        reg_inc_step<160>();
    }
    const int lo = min((int)blockIdx.x * a.per, a.total), hi = min(lo + a.per, a.total), rep = a.H / a.Hkv;
    [[maybe_unused]] StateStream<T, D, Ring> states(a, step_smem);
    constexpr bool kBeside = kMaps && NH == 4;   // (the sums of eight heads do not fit beside the rings)
    for (int x = lo; x < hi;) {
        const int u = x / a.unit_len;
        const int tile_lo = x - u * a.unit_len, tile_hi = min(a.tiles, hi - u * a.unit_len);
        x = min((u + 1) * a.unit_len, hi);
        if (tile_lo >= tile_hi) continue;
        const int row = u / a.units_per_group;               // batch * Hkv + KV head
        const int h0 = u % a.units_per_group * a.heads_per_unit;
        const long long bh = (long long)(row / a.Hkv) * a.H + row % a.Hkv * rep + h0;
        const int slot = (int)blockIdx.x - unit_first_block(a.per, a.unit_len, u);
        AttendView v = a.view;
        v.rep = min(a.heads_per_unit, rep - h0);
        const T *kh = a.kc + row * a.kvr * D, *vh = a.vc + row * a.kvr * D;   // (kvr is 64-bit)
        const uint32_t *mask = a.sel_mask + bh * v.n_chunk_cap * (v.C / 32);
        float *part = a.part + (bh * kRecords + slot) * (D + 2), *logits = a.part + (bh * kRecords + kLogitRecord) * (D + 2);
        if constexpr (sizeof(T) == 2)
            attend_segment<D, NH, kMaps, kBeside>(v, kh, vh, a.k + row * D, a.v + row * D, a.q + bh * D, mask, tile_lo, tile_hi, step_smem,
                                           reinterpret_cast<float *>(kBeside ? beside : step_smem), part, logits, kRecords * (D + 2), [&] {
                                               if constexpr (kBeside) {
                                                   if (x >= hi) states.request();   // (the block's last segment)
                                               }
                                           });
        else
            attend_segment_f32<D>(v, kh, vh, a.k + row * D, a.v + row * D, a.q + bh * D, mask, tile_lo, tile_hi,
                                  step_smem, part, logits, kRecords * (D + 2));
    }
    if constexpr (kMaps) {
        if (states.requested == 0) states.request();
        asm volatile("bar.sync %0, %1;" ::"n"(kPhiBarrier), "n"(kMainThreads<kMaps>) : "memory");
        if (a.item_warps == 1) states.template run<1>(beside);
        else if (a.item_warps == 2) states.template run<2>(beside);
        else states.template run<kStepWarps>(beside);
    }
    if ((int)blockIdx.x < a.first_item_block) return;
    if constexpr (kMode == kItemsApart) {
        work_on_items<T, D, kStepWarps, true, Ring>(a, step_smem, 0, [&] { return state_mismatch(a.hdr, a.key) == 0; });
        return;
    }
    // (beyond kMaxPhi a block only has more where a read-out is one warp's: the groups' places beside the rings do not meet)
    const int first = kMaps ? kMaxPhi : 0;
    if (a.item_warps == 1) work_on_items<T, D, 1, false, Ring>(a, step_smem, first, [] { return true; });
    else if (a.item_warps == 2) work_on_items<T, D, 2, false, Ring>(a, step_smem, first, [] { return true; });
    else work_on_items<T, D, kStepWarps, false, Ring>(a, step_smem, first, [] { return true; });
}

// grid (H, B), D + 64 threads: an output column each, then a warp that scores the new token and one that appends its K / V
// row.  For a few sequences its latency counts: everything it reads is requested before the first use (13 partials read
// four at a time, then the score, took 4 to 7 us).
template <typename T, int D>
__global__ void __launch_bounds__(D + 64)
step_merge_kernel(const __grid_constant__ StepArgs<T> a) {
    grid_dep_wait();
    grid_dep_launch();
    if (a.hdr[14] != 0) return;   // mismatch recorded by the step's first kernel: no output, token count unchanged
    const int h = blockIdx.x, b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, rep = a.H / a.Hkv;
    const long long bh = (long long)b * a.H + h;
    const float *pr = a.part + bh * kRecords * (D + 2);
    if (tid >= D + 32) {   // the new row of the K / V history (position p lives in ring row p % kvr)
        if (h % rep == 0) {
            const long long row = (long long)b * a.Hkv + h / rep, dst = (row * a.kvr + (uint32_t)a.t % (uint32_t)a.kvr) * D;
            constexpr int kVec = D * (int)sizeof(T) / 16;
            if (lane < kVec) {
                const uint4 kk = reinterpret_cast<const uint4 *>(a.k + row * D)[lane], vv = reinterpret_cast<const uint4 *>(a.v + row * D)[lane];
                reinterpret_cast<uint4 *>(a.kc + dst)[lane] = kk;
                reinterpret_cast<uint4 *>(a.vc + dst)[lane] = vv;
            }
        }
        return;
    }
    if (tid >= D) {        // Self-Saliency Score of the new token: its window's logits lie in the head's last records
        const int C = a.view.C;
        float l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int j = lane + 32 * i;
            l[i] = j < C && a.view.t - (C - 1) + j >= 0 ? pr[kLogitRecord * (D + 2) + j] : -INFINITY;
        }
        const float sc = window_score(l, lane, C >> 5, C, a.eps);
        if (lane == 0) a.score[bh * a.cap + a.t] = sc;
        if (h == 0 && b == 0 && lane == 0) {
            const long long nt = a.t + 1;
            a.hdr[12] = (int32_t)(nt & 0xffffffffll);
            a.hdr[13] = (int32_t)(nt >> 32);
        }
        return;
    }
    const int u = (b * a.Hkv + h / rep) * a.units_per_group + h % rep / a.heads_per_unit;
    const int n = unit_blocks(a.per, a.unit_len, a.tiles, u);    // at most kMaxSplits
    float nla = 0.f, dla = 0.f, gate = 1.f;
    if (a.la) {
        nla = pr[kLinRecord * (D + 2) + 2 + tid];
        dla = pr[kLinRecord * (D + 2) + 1];
        if (a.g) gate = ld_f(a.g + bh * D + tid);
    }
    const float ms = lane < n ? pr[lane * (D + 2)] : -INFINITY, ls = lane < n ? pr[lane * (D + 2) + 1] : 0.f;
    float x[16];
#pragma unroll
    for (int s = 0; s < 16; ++s) x[s] = s < n ? pr[s * (D + 2) + 2 + tid] : 0.f;
    // every warp forms the weights of the partials
    const float M = warp_max(ms);
    const float w = ms == -INFINITY ? 0.f : expf(ms - M);
    const float L = warp_sum(ms == -INFINITY ? 0.f : w * ls);
    float O = 0.f;
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        const float ws = __shfl_sync(0xffffffffu, w, s);
        if (ws != 0.f) O = fmaf(ws, x[s], O);
    }
    if (n > 16) {
#pragma unroll
        for (int s = 0; s < 16; ++s) x[s] = s + 16 < n ? pr[(s + 16) * (D + 2) + 2 + tid] : 0.f;
#pragma unroll
        for (int s = 0; s < 16; ++s) {
            const float ws = __shfl_sync(0xffffffffu, w, s + 16);
            if (ws != 0.f) O = fmaf(ws, x[s], O);
        }
    }
    nla *= gate;
    float fs = 1.f, fl = 0.f;
    if (dla > 0.f) {
        const float mm = fmaxf(M, 0.f);
        fs = expf(M - mm);
        fl = expf(-mm);
    }
    st_f(a.y + bh * D + tid, (O * fs + fl * nla) / (L * fs + fl * dla));
}

#define STILL_CUDA(expr)                               \
    do {                                               \
        cudaError_t e__ = (expr);                      \
        if (e__ != cudaSuccess) return STILL_ERR_CUDA; \
    } while (0)

template <typename T>
static int launch_route(const still_params_t *p, const StepArgs<T> &a, int32_t *sel, const T *Wk, const T *bk, long long cr,
                        int window, cudaStream_t st, int *launches) {
    const int C = p->chunk, d = p->d, df = p->d_f;
    T *wk = const_cast<T *>(Wk), *bkp = const_cast<T *>(bk);
    if constexpr (sizeof(T) == 2) {
        auto launch = [&](auto kernel, int smem, int max_smem) -> int {
            STILL_CUDA(ensure_dynamic_smem((const void *)kernel, max_smem));
            STILL_CUDA(launch_dependent(kernel, dim3(p->H, p->B), dim3(256), smem, st, a.kc, a.vc, a.score, sel, a.sel_mask, a.S, a.z,
                                        wk, bkp, a.hdr, a.key, p->H, p->Hkv, a.cap, a.kvr, df, C, p->topk, cr, window));
            return STILL_OK;
        };
        const int rc = d == 64 ? launch(step_route_mma_kernel<64>, RoutePlan<64>(C, df).total, RoutePlan<64>(128, 64).total)
                               : launch(step_route_mma_kernel<128>, RoutePlan<128>(C, df).total, RoutePlan<128>(128, 128).total);
        if (rc != STILL_OK) return rc;
    } else {
        size_t smem = ((size_t)C * 2 * df + (size_t)C * d + 8 * (size_t)d + C) * 4 + (size_t)C * 4;
        const int w_in_smem = smem + (size_t)d * df * sizeof(T) <= 200 * 1024 ? 1 : 0;
        if (w_in_smem) smem += (size_t)d * df * sizeof(T);
        STILL_CUDA(cudaFuncSetAttribute(step_route_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        STILL_CUDA(launch_dependent(step_route_kernel, dim3(p->H, p->B), dim3(256), smem, st, a.kc, a.vc, a.score, sel, a.sel_mask,
                                    a.S, a.z, wk, bkp, a.hdr, a.key, p->H, p->Hkv, a.cap, a.kvr, d, df, C, p->topk, cr, window,
                                    w_in_smem));
    }
    ++*launches;
    return STILL_OK;
}

// Map warps where the blocks have read-outs behind their tiles (bf16, up to eight heads a KV group: with 16 the cache pass
// needs the registers) and the tiles are not many: what the read-outs gain is a few us whatever the tiles, and the cache pass, in
// fewer registers and beside the loads of W_q, takes up to 2 % longer.  (us a step without and with them: 325 tiles a block
// 82.7 and 81.4, 865 tiles, 16 sequences x 16000 tokens, 141.2 and 142.5.)
constexpr int kMapTiles = 512;   // tiles of a block
// Nor where the map warps, four read-outs at a time, would be what the block waits for.  The fewest tiles of a block with which they
// are worth it, by read-outs a block (us a step without and with them; a quarter kept, 32 heads unless said):
//   two rounds and more: 70 tiles are as long as a round.  32 sequences x 8192 tokens capped at 448, 204 tiles and two rounds, 71.9
//     and 69.1; 64 x 1000, 215 and four, 104.9 and 109.9; 64 x 3000 capped at 128, 160 and four, 100.7 and 106.5.  Up to 4.5 a block the
//     second round is a few blocks' alone, and the others' eight warps have little to do: 20 sequences at 155 tiles 55.2 and
//     56.3, at 170 57.1 and 56.0; 22 (4.8 a block) at 127 52.2 and 53.0, at 141 54.8 and 54.0;
//   one round, d = d_f = 128: a map warp reads the 32 KB of W_q in eight batches.  One a block, which eight warps share otherwise:
//     4 sequences at 16 tiles 16.1 and 16.5, 3 at 11 15.2 and 16.2, at 21 16.54 and 16.65, at 24 16.98 and 16.87, 4 at 32 18.2 and 17.0.
//     Two or three: 9 of 20 heads at 5 tiles 18.5 and 18.8, 6 at 7 tiles 19.3 and 18.9, 12 at 13 23.5 and 21.9.  Nearly four, whose loads stand in each other's way: 15
//     (3.2 a block) at 16 tiles 25.2 and 24.8, 16 (3.5) at 17 25.8 and 26.7, 18 (3.9) at 20 24.9 and 28.6, at 49 36.1 and 37.5, at 62 36.9
//     and 35.0;
//   ... with narrower maps always: 3 sequences, d_f = 64, at 4 tiles 12.5 and 12.2, 18 at 20 20.0 and 17.5;
//   ... d = 64: three a block, four groups of two warps otherwise: 10 sequences at 10 tiles 15.2 and 15.8, at 34 (d_f = 32) 16.4 and
//     16.7, 12 at 44 18.25 and 18.18, at 82 22.2 and 22.1.  Else always: one 11.4 and 10.4, two 13.4 to 14.9 and 13.2 to 15.0, four 15.1 and 14.4.
static int least_map_tiles(long long n_items, long long blocks, int d, int df) {
    const long long rounds = (n_items + kMapWarps * blocks - 1) / (kMapWarps * blocks);
    if (rounds > 1) return 2 * n_items <= 9 * blocks ? 168 : (int)(70 * rounds);
    if (d == 64) return n_items > 2 * blocks && n_items <= 3 * blocks ? 48 : 0;
    if (df < 128) return 0;
    return n_items <= blocks ? 24 : 4 * n_items > 13 * blocks ? 60 : 6;
}
template <typename T, int D, int NH>
static int launch_main(const StepArgs<T> &a, unsigned grid, cudaStream_t st, int *launches) {
    auto launch = [&](auto mode) -> int {
        constexpr StepMode kMode = decltype(mode)::value;
        constexpr bool kMaps = kMode == kItemsMapped;
        constexpr int kSmem = step_main_smem<T, D, kMaps>();
        STILL_CUDA(ensure_dynamic_smem((const void *)step_main_kernel<T, D, NH, kMode>, kSmem));
        profile_mark_begin(st);
        STILL_CUDA(launch_dependent(step_main_kernel<T, D, NH, kMode>, dim3(grid), dim3(kMainThreads<kMaps>), kSmem, st, a));
        profile_mark_end(st);
        return STILL_OK;
    };
    const bool map = a.n_items > 0 && a.per <= kMapTiles && a.per >= least_map_tiles(a.n_items, grid, D, a.df);
    constexpr bool kCanMap = sizeof(T) == 2 && NH <= 8;
    int rc;
    if (a.n_items > 0 && a.first_item_block > 0) rc = launch(std::integral_constant<StepMode, kItemsApart>{});
    else if (kCanMap && map) rc = launch(std::integral_constant<StepMode, kCanMap ? kItemsMapped : kItemsShared>{});
    else rc = launch(std::integral_constant<StepMode, kItemsShared>{});
    if (rc != STILL_OK) return rc;
    STILL_CUDA(launch_dependent(step_merge_kernel<T, D>, dim3(a.H, a.B), dim3(D + 64), 0, st, a));
    *launches += 2;
    return STILL_OK;
}

template <typename T>
static int step_typed(const still_params_t *p, char *state, const still_state_layout_t *L, long long t,
                      const T *q, const T *k, const T *v, const T *g, const T *Wq, const T *bq,
                      const T *Wk, const T *bk, T *y, cudaStream_t st, int *launches) {
    const int C = p->chunk, d = p->d, df = p->d_f, lam = p->topk, rep = p->H / p->Hkv;
    const long long cap = L->capacity;
    const int window = lam > 0 ? (int)(p->max_salient / lam) : 0;   // chunks whose selections the salient cache holds
    constexpr bool kBf16 = sizeof(T) == 2;
    if (kBf16 && rep > 16) return STILL_ERR_UNSUPPORTED;            // the group's heads are two tiles of eight
    const long long c_cur = t / C;

    StepArgs<T> a{};
    a.kc = reinterpret_cast<T *>(state + L->k_cache);
    a.vc = reinterpret_cast<T *>(state + L->v_cache);
    a.score = reinterpret_cast<float *>(state + L->score);
    a.sel_mask = reinterpret_cast<uint32_t *>(state + L->sel_mask);
    a.S = reinterpret_cast<float *>(state + L->S);
    a.z = reinterpret_cast<float *>(state + L->z);
    a.part = reinterpret_cast<float *>(state + L->scratch);
    a.hdr = reinterpret_cast<int32_t *>(state + L->header);
    a.q = const_cast<T *>(q); a.k = const_cast<T *>(k); a.v = const_cast<T *>(v); a.g = const_cast<T *>(g);
    a.Wq = const_cast<T *>(Wq); a.bq = const_cast<T *>(bq); a.y = y;
    a.key = StateKey{p->B, p->H, p->Hkv, p->d, p->d_f, p->chunk, p->topk, p->dtype, cap, t};
    a.cap = cap;
    a.kvr = state_kv_rows(p, cap);
    a.t = t;
    a.B = p->B; a.H = p->H; a.Hkv = p->Hkv; a.df = df;
    a.la = lam < C || window > 0;
    a.eps = p->eps;
    AttendView &w = a.view;
    w.kvr = a.kvr;
    w.t = (int)t;
    w.loc0 = (int)(c_cur >= 1 ? (c_cur - 1) * C : 0);
    // routed chunks still cached: all, with a budget the last `window` before the local region, none when topk = 0
    w.first_pos = lam <= 0 ? w.loc0 : window > 0 ? (int)(std::max<long long>(0, c_cur - 1 - window) * C) : 0;
    w.C = C; w.lam = lam; w.rep = rep; w.n_chunk_cap = (int)(cap / C);
    w.scale = p->sm_scale;
    w.scale_log2 = p->sm_scale * 1.4426950408889634f;

    if (t % C == 0 && c_cur >= 2) {
        const int rc = launch_route<T>(p, a, reinterpret_cast<int32_t *>(state + L->sel_idx), Wk, bk, c_cur - 2, window, st, launches);
        if (rc != STILL_OK) return rc;
    }

    int n_sm = 0, dev = 0;
    STILL_CUDA(cudaGetDevice(&dev));
    STILL_CUDA(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
    constexpr int kKeys = kBf16 ? kTileKeys : kTileKeysF32;
    a.heads_per_unit = kBf16 ? rep : kUnitHeadsF32;
    a.units_per_group = (rep + a.heads_per_unit - 1) / a.heads_per_unit;
    a.tiles = (int)((t - w.first_pos) / kKeys) + 1;
    const long long units = (long long)p->B * p->Hkv * a.units_per_group;
    a.n_items = a.la ? p->B * p->H : 0;
    // Few read-outs (a sequence or two): a block each, beside the blocks of the cache pass.  More: every block takes its
    // share of the tiles and then of the read-outs.  (us a step, d = 128, a quarter kept, apart / together: 32 read-outs
    // 10.4 / 12.8 at 2000 tokens and 19.4 / 19.5 at 16000, 64: 11.4 / 13.9 and 35.0 / 29.9, 96: 17.2 / 15.1 and 73.9 / 39.5.)
    const bool apart = a.n_items <= n_sm / 2;
    const long long blocks = apart ? n_sm - a.n_items : n_sm;
    const long long least = (a.tiles + kMaxSplits - 2) / (kMaxSplits - 1);
    a.unit_len = a.tiles;
    a.per = (int)std::max<long long>({(units * a.tiles + blocks - 1) / blocks, least, 1});
    // Whole blocks per unit where a block's share is short: one with tiles of two units does two passes, one after the
    // other, and a pass of up to eight rounds of the warps is mostly latency.  (us a step, whole blocks / one line, every
    // token kept: 8 units of 31, 125 and 500 tiles 7.3 / 9.0, 8.8 / 10.4, 11.4 / 13.8, of 2000 (past the second limit)
    // 28.6 / 30.6; 32 units of 62 and 187 tiles 9.6 / 12.2, 13.2 / 14.7, of 1000 (past it) 46.1 / 48.9; 64 units (past the
    // first limit) of 62 and 250 tiles 11.9 / 14.2, 28.5 / 28.7; 128 units 15.7 / 17.2, 47.0 / 49.5.  The limits are on the safe
    // side: units just above half the SMs would leave nearly half of these without tiles, which was not timed.)
    const long long per_unit = blocks / units;
    if (per_unit >= 4 && a.tiles <= per_unit * 8 * kStepWarps) {
        a.per = (int)std::max<long long>((a.tiles + per_unit - 1) / per_unit, least);
        a.unit_len = (a.tiles + a.per - 1) / a.per * a.per;
    }
    a.total = (int)(units * a.unit_len);   // (a state of 2^31 tiles would be 8 TB)
    w.early_k = per_unit >= 4;
    const long long used = (a.total + a.per - 1) / a.per;           // blocks with tiles
    a.first_item_block = apart ? (int)used : 0;
    // The fewer warps share a read-out, the more run side by side and the longer one takes.  (us a step, d = 128, 2000 tokens,
    // by eight / two / one warps: 128 read-outs 16.5 / 18.3 / 23.1, 160: 23.1 / 21.4 / 26.4, 576: 49.5 / 42.4 / 44.7,
    // 640: 57.0 / 51.3 / 48.6, 2048: 147 / 120 / 120.)
    a.item_warps = a.n_items <= n_sm ? kStepWarps : a.n_items <= n_sm * (kStepWarps / 2) ? 2 : 1;
    const unsigned grid = (unsigned)(apart ? used + a.n_items : n_sm);
    auto launch = [&](auto head_dim) -> int {
        constexpr int D = decltype(head_dim)::value;
        if constexpr (kBf16) {
            if (rep <= 4) return launch_main<T, D, 4>(a, grid, st, launches);
            return rep <= 8 ? launch_main<T, D, 8>(a, grid, st, launches) : launch_main<T, D, 16>(a, grid, st, launches);
        } else {
            return launch_main<T, D, kUnitHeadsF32>(a, grid, st, launches);
        }
    };
    return d == 64 ? launch(std::integral_constant<int, 64>{}) : launch(std::integral_constant<int, 128>{});
}

int step_launch(const still_params_t *p, char *state, const still_state_layout_t *L, long long t_pos,
                const void *q, const void *k, const void *v, const void *g, const void *Wq,
                const void *bq, const void *Wk, const void *bk, void *y, cudaStream_t st,
                int *launches) {
    if (p->dtype == STILL_DTYPE_FP32)
        return step_typed<float>(p, state, L, t_pos, (const float *)q, (const float *)k, (const float *)v,
                                 (const float *)g, (const float *)Wq, (const float *)bq, (const float *)Wk,
                                 (const float *)bk, (float *)y, st, launches);
    using bf = __nv_bfloat16;
    return step_typed<bf>(p, state, L, t_pos, (const bf *)q, (const bf *)k, (const bf *)v, (const bf *)g,
                          (const bf *)Wq, (const bf *)bq, (const bf *)Wk, (const bf *)bk, (bf *)y, st,
                          launches);
}

}  // namespace still
