// Linear-attention branch of the prefill on tensor cores (bf16 inputs, sm_100a).
//
// npmap_tc_kernel -- Norm-Preserved Feature Map (Sec. 3.2, Eq. feature_map) of 128 rows of K per CTA,
//   fused into the load of the rows:  f = x W  on tcgen05 (x tile K-major from TMA, W MN-major from TMA,
//   accumulator in TMEM), then per row  u = (f + b) ||x|| / max(||f + b||, 1e-12),
//   phi = [softmax(u), softmax(-u)], stored as bf16 (the B operand of the bf16 state-update GEMM) once
//   per KV head, together with the column sums of every chunk.
//
// gather_kernel / z_scan_kernel -- the rows of the selected tokens in selection order, with the sums of their features,
//   and the normaliser z of Eq. cache_routing_sum after every routed chunk: column sums of the chunk minus the rows of
//   its selected tokens, as a running sum over chunks.
//
// la_fused_kernel -- Algorithm 1 "Linear Attention Branch" with the state of Eq. cache_routing_sum kept
//   in tensor memory and the query-side NP-Map computed on the fly (phi(Q) never reaches HBM).  One CTA
//   owns one (batch, query head) and one half of the feature dimension (the softmax(u) features or the
//   softmax(-u) features) and walks the chunks in order.  The state half is held transposed, S^T
//   [value columns x d_f features] fp32 in TMEM.
//     update   S^T += V_c^T phi_k(K_c)   for the chunk c that has just left the two-chunk local region:
//              bf16 UMMA, A = V tile (M-major, as TMA delivers it), B = phi(K) half tile (MN-major)
//              whose rows of the tokens selected for softmax attention were zeroed;
//     map      f = Q W_q for a block of 128 query rows (UMMA), then a thread per row: norm re-injection,
//              this CTA's softmax half, written unnormalised (e_j = 2^(+-u_j - max)) as an fp32 K-major
//              tile into shared memory; D_part = (e . z_half of the chunk two back) / sum e;
//     read-out N_part^T = S^T phi_q(Q_c)^T  for the chunk c being answered: TF32 UMMA with the fp32
//              state read straight from TMEM as the A operand (10-bit mantissa instead of the 7 bits a
//              bf16 copy of the state would keep), B = the phi(Q) tile.
//   Output: y_part = N_part / D_part = (e . S) / (e . z) (times the gate) as bf16 and D_part as fp32, per feature half; the
//   merge epilogue of the attention kernel forms N_LA = sum y_part D_part, D_LA = sum D_part.
//   The lag of two chunks between update and read-out is the delayed selection of Sec. 3.3.  Work is
//   tiled in 64-token sub-chunks, so C = 128 is two sub-chunks per chunk.
//
// Roles of la_fused_kernel (384 threads): warp 0 TMA producer, warp 1 MMA issuer, warps 2 and 3 take turns at zeroing the
// selected rows of the phi(K) tiles, warps 4-7 write the output, warps 8-11 the query-side map.  Every mbarrier
// wait is bounded; on expiry the kernel records STILL_ERR_DEVICE_TIMEOUT in the status word, all roles
// leave their loops and tensor memory is freed before the CTA exits.
#include "still_tc.h"

#include <algorithm>

#include "still_common.cuh"
#include "still_state.cuh"
#include "still_tc_ptx.cuh"

namespace still {

namespace {

using namespace ptx;

constexpr int kSms = 148;   // SMs that grids are planned for

// Instruction descriptor of kind::tf32 (fp32 accumulation, both operands TF32, B K-major).
__host__ __device__ constexpr uint32_t make_idesc_tf32(int M, int N) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ------------------------------------------------------------------------------------------
// NP-Map
// ------------------------------------------------------------------------------------------
// Shared memory of the NP-Map kernel: the x and W tiles, later reused as the staging space of the output
// (four warps x 32 padded rows); the region is the larger of the two.
template <int D, int DF, typename TOut>
struct NpmapSmem {
    static constexpr int kHalfChunks = 32 * (int)sizeof(TOut) / 16;   // 16-byte pieces of 32 features
    static constexpr int kStageRow = 2 * kHalfChunks * 16 + 16;       // padded: conflict-free 16-byte accesses
    static constexpr int kTiles = 128 * D * 2 + D * DF * 2;
    static constexpr int kStage = 4 * 32 * kStageRow;
    static constexpr int kRegion = ((kTiles > kStage ? kTiles : kStage) + 1023) / 1024 * 1024;
    static constexpr int kTotal = kRegion + 64;
};

template <int D, int DF, typename TOut>
__global__ void __launch_bounds__(192, 3)
npmap_tc_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                const __nv_bfloat16 *bias, TOut *phi, float *csum, int *status,
                int heads, int N, int C) {
    grid_dep_wait();
    grid_dep_launch();
    constexpr int kXBytes = 128 * D * 2, kWBytes = D * DF * 2;
    using Lay = NpmapSmem<D, DF, TOut>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *x_s = smem, *w_s = smem + kXBytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + Lay::kRegion);  // [0] loads done, [1] f done
    uint32_t *tmem_base_slot = reinterpret_cast<uint32_t *>(bars + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_base_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int hd = blockIdx.y, b = blockIdx.z, R0 = blockIdx.x * 128;
    const long long row0 = ((long long)b * heads + hd) * N + R0;
    if ((smem_u32(smem) & 1023u) != 0) {
        if (threadIdx.x == 0) report_status(status, STILL_ERR_DEVICE_TIMEOUT, 98);
        return;
    }
    if (threadIdx.x == 0) {
        mbar_init(bars, 1);
        mbar_init(bars + 1, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_base_slot, 128);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_base_slot;

    if (warp == 0 && lane == 0) {
        mbar_expect_tx(bars, kXBytes + kWBytes);
        for (int half = 0; half < D / 64; ++half)  // x rows: K-major, 64-element atoms 128 rows apart
            tma_load_2d(x_s + half * (128 * 128), &tm_x, bars, half * 64, (int)row0);
        for (int a = 0; a < DF / 64; ++a)          // W [d rows, d_f columns]: MN-major, 64-column atoms D rows apart
            tma_load_2d(w_s + a * (D * 128), &tm_w, bars, a * 64, hd * D);
    } else if (warp == 1 && lane == 0) {
        constexpr uint32_t idesc = make_idesc(128, DF, true);
        if (mbar_wait(bars, 0, abort_flag, status, 30)) {
            tc_fence_after();
#pragma unroll
            for (int k = 0; k < D / 16; ++k) {
                const uint32_t xa = smem_u32(x_s) + (k / 4) * (128 * 128) + (k % 4) * 32;
                const uint32_t wa = smem_u32(w_s) + k * (16 * 128);
                mma_ss(tmem_base, smem_desc(xa, 0), smem_desc(wa, D * 128), idesc, k > 0 ? 1u : 0u);
            }
            tc_commit(bars + 1);
        }
    } else if (warp >= 2) {
        const int wq = warp & 3, r = wq * 32 + lane;   // TMEM lane quarter of this warp; row of the tile
        const uint32_t taddr = tmem_base + ((uint32_t)(wq * 32) << 16);
        bool ok = mbar_wait(bars, 0, abort_flag, status, 31);   // x tile in shared memory
        ok = __all_sync(0xffffffffu, ok);
        float nx2 = 0.f;
        if (ok) {
#pragma unroll
            for (int a = 0; a < D / 64; ++a)
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint4 v = *reinterpret_cast<const uint4 *>(x_s + a * (128 * 128) + r * 128 + ((c ^ (r & 7)) << 4));
                    const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float lo = __uint_as_float(w4[e] << 16), hi = __uint_as_float(w4[e] & 0xffff0000u);
                        nx2 = fmaf(lo, lo, nx2);
                        nx2 = fmaf(hi, hi, nx2);
                    }
                }
        }
        // all four epilogue warps are done reading the x tile before any of them reuses it as staging space
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (ok) ok = mbar_wait(bars + 1, 0, abort_flag, status, 32);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
            tc_fence_after();
            // Three passes over the row of f in tensor memory, 32 columns at a time, so that the row is
            // never held in registers (several CTAs per SM then overlap their load / MMA / epilogue
            // phases): norms and extrema, the two softmax denominators, the features themselves.
            const __nv_bfloat16 *bh_ = bias != nullptr ? bias + (long long)hd * DF : nullptr;
            float nf2 = 0.f, fmax_ = -INFINITY, fmin_ = INFINITY;
#pragma unroll 1
            for (int q = 0; q < DF / 32; ++q) {
                uint32_t v[32];
                tmem_ld32(taddr + q * 32, v);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    float x = __uint_as_float(v[j]);
                    if (bh_ != nullptr) x += __bfloat162float(bh_[q * 32 + j]);
                    nf2 = fmaf(x, x, nf2);
                    fmax_ = fmaxf(fmax_, x);
                    fmin_ = fminf(fmin_, x);
                }
            }
            // u = f * ratio in the log2 domain; ratio > 0, so the extrema of u are those of f
            const float ratio = sqrtf(nx2) / fmaxf(sqrtf(nf2), 1e-12f) * 1.4426950408889634f;
            const float umax = fmax_ * ratio, umin = fmin_ * ratio;
            float zp = 0.f, zn = 0.f;
#pragma unroll 1
            for (int q = 0; q < DF / 32; ++q) {
                uint32_t v[32];
                tmem_ld32(taddr + q * 32, v);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    float x = __uint_as_float(v[j]);
                    if (bh_ != nullptr) x += __bfloat162float(bh_[q * 32 + j]);
                    const float u = x * ratio;
                    zp += ex2(u - umax);
                    zn += ex2(umin - u);
                }
            }
            const float ip = 1.f / zp, in = 1.f / zn;
            // The features leave through shared memory: a thread owns a row, but a store instruction in
            // which every lane writes to a different row touches 32 lines; staged, 8 (fp32) or 4 (bf16)
            // consecutive lanes write one 128- or 64-byte run of a row.  Each warp stages and writes its
            // own 32 rows (the x / W tiles are dead by now), 32 columns of both halves at a time.
            constexpr int kHalfChunks = Lay::kHalfChunks, kStageRow = Lay::kStageRow;
            uint8_t *stage = smem + wq * (32 * kStageRow);
            const int rows_live = min(32, N - (R0 + wq * 32));        // rows of this warp that exist
            float *csw = reinterpret_cast<float *>(smem + 4 * 32 * kStageRow) + wq * (2 * DF);   // this warp's column sums
#pragma unroll 1
            for (int q = 0; q < DF / 32; ++q) {
                uint32_t v[32];
                tmem_ld32(taddr + q * 32, v);
                tmem_wait_ld();
                uint8_t *mine = stage + lane * kStageRow;
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    float u[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float x = __uint_as_float(v[j + e]);
                        if (bh_ != nullptr) x += __bfloat162float(bh_[q * 32 + j + e]);
                        u[e] = x * ratio;
                    }
                    if constexpr (sizeof(TOut) == 4) {
                        *reinterpret_cast<float4 *>(mine + j * 4) =
                            make_float4(ex2(u[0] - umax) * ip, ex2(u[1] - umax) * ip, ex2(u[2] - umax) * ip, ex2(u[3] - umax) * ip);
                        *reinterpret_cast<float4 *>(mine + kHalfChunks * 16 + j * 4) =
                            make_float4(ex2(umin - u[0]) * in, ex2(umin - u[1]) * in, ex2(umin - u[2]) * in, ex2(umin - u[3]) * in);
                    } else {
                        *reinterpret_cast<uint2 *>(mine + j * 2) =
                            make_uint2(pack_bf16(ex2(u[0] - umax) * ip, ex2(u[1] - umax) * ip),
                                       pack_bf16(ex2(u[2] - umax) * ip, ex2(u[3] - umax) * ip));
                        *reinterpret_cast<uint2 *>(mine + kHalfChunks * 16 + j * 2) =
                            make_uint2(pack_bf16(ex2(umin - u[0]) * in, ex2(umin - u[1]) * in),
                                       pack_bf16(ex2(umin - u[2]) * in, ex2(umin - u[3]) * in));
                    }
                }
                __syncwarp();
                if constexpr (sizeof(TOut) == 2) {
                    // column sums of the stored (bf16-rounded) features over the warp's rows, in row order: lane l
                    // adds feature 32 q + l of both halves (what the normaliser z of the linear branch is made of)
                    if (csum != nullptr) {
                        float sp = 0.f, sn = 0.f;
                        for (int row = 0; row < rows_live; ++row) {
                            const uint8_t *src = stage + row * kStageRow + lane * 2;
                            sp += __uint_as_float((uint32_t)(*reinterpret_cast<const uint16_t *>(src)) << 16);
                            sn += __uint_as_float((uint32_t)(*reinterpret_cast<const uint16_t *>(src + kHalfChunks * 16)) << 16);
                        }
                        csw[q * 32 + lane] = sp;
                        csw[DF + q * 32 + lane] = sn;
                    }
                }
#pragma unroll
                for (int it = 0; it < 2 * kHalfChunks; ++it) {
                    const int id = it * 32 + lane, row = id / (2 * kHalfChunks), c = id % (2 * kHalfChunks);
                    if (row < rows_live) {
                        const uint4 val = *reinterpret_cast<const uint4 *>(stage + row * kStageRow + c * 16);
                        uint8_t *dst = reinterpret_cast<uint8_t *>(phi + (row0 + wq * 32 + row) * (2 * DF) +
                                                                   (c < kHalfChunks ? 0 : DF) + q * 32) +
                                       (c % kHalfChunks) * 16;
                        *reinterpret_cast<uint4 *>(dst) = val;
                    }
                }
                __syncwarp();
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (sizeof(TOut) == 2) {
        // per-chunk column sums: the warps of a chunk are added in warp order (fixed order: the sums are reproducible)
        if (csum != nullptr && warp >= 2 && !*abort_flag) {
            const float *csw_all = reinterpret_cast<const float *>(smem + 4 * 32 * NpmapSmem<D, DF, TOut>::kStageRow);
            const int Tn = (N + C - 1) / C, wpc = C / 32;             // warps (of 32 rows) per chunk: 2 or 4
            for (int i = threadIdx.x - 64; i < (128 / C) * 2 * DF; i += 128) {
                const int k = i / (2 * DF), f = i % (2 * DF), chunk = R0 / C + k;
                if (chunk < Tn) {
                    float acc = 0.f;
                    for (int w = 0; w < wpc; ++w)
                        if (R0 + (k * wpc + w) * 32 < N) acc += csw_all[(k * wpc + w) * (2 * DF) + f];
                    csum[(((long long)b * heads + hd) * Tn + chunk) * (2 * DF) + f] = acc;
                }
            }
        }
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 128);
    }
}

// ------------------------------------------------------------------------------------------
// Selected rows, and the normaliser z (Eq. cache_routing_sum): z after chunk c = sum over the chunks 0..c of the
// features of their unselected tokens = (column sums of phi(K) over the chunk) - (rows of its selected tokens).
// ------------------------------------------------------------------------------------------
// grid (T + 1, B*H; with the decode state: and as many rows as its blocks take), 256 threads: the lam selected tokens of a
// chunk of a query head, read once for everything
// that is made of them: their K and V rows in selection order (row j of a head is token sel_idx[j]; K_sel / V_sel, what
// the attention kernel tiles), with a salient-cache budget also their phi(K) rows (phi_sel, from which the tokens that
// leave the cache enter the state), and the sum of the phi(K) rows (selsum [B*H, n_routed, 2 DF], of the routed chunks).
// -1 entries and the rows of the padding (chunk T) are zero.  NULL outputs are not made.  Bound by the bytes written
// and the rows read: 32 heads x 131072 tokens, d = 128, 32 of 128 selected, with phi_sel: three kernels that each
// gathered for themselves (and one that summed a row after the other) took 1023 us, this one 305.
// A head begins with another chunk than the one before: else, where T + 1 is a multiple of 37, all paddings, which are the longest,
// lay on four SMs (32 heads x 2244 tokens, d = 64, with phi_sel: 15.2 us and 7.9; with five blocks an SM 10.8).
// kFew: at d = 64 up to 16 tokens of a chunk are one row a thread; eight blocks an SM instead of five keep as many rows in flight
// (128 heads x 4096 tokens, 16 of 64: 29.7 us and 23.7; with 32 of 64 a thread's two rows one after the other 6 us more).  Not with
// the decode state, whose copies do not fit 32 registers, nor 48 (92 and 16 bytes of a thread spilled; with 64 none: us a call of 128 heads x
// 300 tokens 69.4 and 66.9, 64 x 700 67.6 and 65.4, 32 x 1003 56.4 and 56.2).
template <int D, int DF, bool kFew, bool kState>
__global__ void __launch_bounds__(256, D == 128 || kState ? 4 : kFew ? 8 : 5)
gather_kernel(const __nv_bfloat16 *K, const __nv_bfloat16 *V, const __nv_bfloat16 *phiK,
              const int32_t *sel_idx, __nv_bfloat16 *Ksel, __nv_bfloat16 *Vsel,
              __nv_bfloat16 *phi_sel, float *selsum, int H, int Hkv, long long N, int lam,
              long long sel_rows, int n_routed, int BH, const __grid_constant__ StateParts state, const __grid_constant__ still_params_t p) {
    grid_dep_wait();
    grid_dep_launch();
    if (kState && (int)blockIdx.y >= BH) {   // the decode state (its blocks behind the others)
        const long long blk = (long long)((int)blockIdx.y - BH) * gridDim.x + blockIdx.x;
        if (blk < state.blocks) write_state_block(state, p, blk);
        return;
    }
    constexpr int kVec = D / 8, kPhiVec = 2 * DF / 8;       // 16-byte pieces of a row
    constexpr int kPer = 32 / kVec, kPhiPer = 32 / kPhiVec;  // rows that a warp moves at a time
    __shared__ __align__(16) float sums[8 * kPhiPer][2 * DF];   // (written 16 bytes at a time)
    const int bh = blockIdx.y, b = bh / H, h = bh % H, c = (int)((blockIdx.x + blockIdx.y) % gridDim.x), Tn = gridDim.x - 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long src0 = ((long long)b * Hkv + h / (H / Hkv)) * N, dst0 = (long long)bh * sel_rows + (long long)c * lam;
    if (c == Tn) {   // padding up to sel_rows
        const long long n = (sel_rows - (long long)Tn * lam) * kVec, n_phi = n / kVec * kPhiVec;
        const uint4 zero = make_uint4(0, 0, 0, 0);
        for (long long i = threadIdx.x; i < n; i += 256) {
            if (Ksel) reinterpret_cast<uint4 *>(Ksel + dst0 * D)[i] = zero;
            if (Vsel) reinterpret_cast<uint4 *>(Vsel + dst0 * D)[i] = zero;
        }
        if (phi_sel)
            for (long long i = threadIdx.x; i < n_phi; i += 256) reinterpret_cast<uint4 *>(phi_sel + dst0 * (2 * DF))[i] = zero;
        return;
    }
    const int32_t *pos = sel_idx + ((long long)bh * Tn + c) * lam;
    // K and V rows: K in even, V in odd groups of lanes.  A thread requests kBatch of these and of the phi(K) pieces before it
    // stores any: a store waits for its load, and the loads behind it would wait with it.
    const int piece = lane % kVec, which = (lane / kVec) & 1, piece_phi = lane % kPhiVec;
    const __nv_bfloat16 *src = which ? V : K;
    __nv_bfloat16 *dst = which ? Vsel : Ksel;
    const bool with_phi = phi_sel != nullptr || c < n_routed;
    constexpr int kStep = 8 * (kPer / 2), kPhiStep = 8 * kPhiPer, kBatch = D == 128 ? 4 : kFew ? 1 : 2;
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
    int r0 = dst ? warp * (kPer / 2) + lane / (2 * kVec) : lam, q0 = with_phi ? warp * kPhiPer + lane / kPhiVec : lam;
    for (; r0 < lam || q0 < lam; r0 += kBatch * kStep, q0 += kBatch * kPhiStep) {
        uint4 v[kBatch], f[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            const int r = r0 + i * kStep, q = q0 + i * kPhiStep, p = r < lam ? pos[r] : -1, pq = q < lam ? pos[q] : -1;
            v[i] = f[i] = make_uint4(0, 0, 0, 0);
            if (p >= 0) v[i] = reinterpret_cast<const uint4 *>(src + (src0 + p) * D)[piece];
            if (pq >= 0) f[i] = reinterpret_cast<const uint4 *>(phiK + (src0 + pq) * (2 * DF))[piece_phi];
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            const int r = r0 + i * kStep, q = q0 + i * kPhiStep;
            if (r < lam) reinterpret_cast<uint4 *>(dst + (dst0 + r) * D)[piece] = v[i];
            if (phi_sel && q < lam) reinterpret_cast<uint4 *>(phi_sel + (dst0 + q) * (2 * DF))[piece_phi] = f[i];
            const uint32_t w[4] = {f[i].x, f[i].y, f[i].z, f[i].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                acc[2 * e] += __uint_as_float(w[e] << 16);
                acc[2 * e + 1] += __uint_as_float(w[e] & 0xffff0000u);
            }
        }
    }
    if (c >= n_routed) return;
    float *mine = &sums[warp * kPhiPer + lane / kPhiVec][piece_phi * 8];
    *reinterpret_cast<float4 *>(mine) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    *reinterpret_cast<float4 *>(mine + 4) = make_float4(acc[4], acc[5], acc[6], acc[7]);
    __syncthreads();
    for (int f = threadIdx.x; f < 2 * DF; f += 256) {   // in a fixed order: the sums are reproducible
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < 8 * kPhiPer; ++w) s += sums[w][f];
        selsum[((long long)bh * n_routed + c) * (2 * DF) + f] = s;
    }
}
// grid (B*H, 2 d_f / 32), up to 1024 threads: z [B*H, n_routed, 2 d_f] after every routed chunk.  What chunk c adds: its column
// sums less its selected rows (nothing when lam = C), plus, with a salient-cache budget of `window` chunks, the selected
// rows of chunk c - window, which leave the cache for the state when chunk c is routed.  Two levels: each of the block's
// warps sums a part of the chunks, and adds them up again from the sum of the parts before.  (One thread per feature
// over all chunks took 132 us for 1022 chunks of 32 heads, a chain of loads; with eight chunks requested together 38 us.)
__global__ void __launch_bounds__(1024)
z_scan_kernel(const float *csum, const float *selsum, float *zpre, float *z_out,
              int H, int Hkv, int Tn, int n_routed, int all_selected, int window, int NF) {
    grid_dep_wait();
    grid_dep_launch();
    __shared__ float part[32][33];
    const int bh = blockIdx.x, b = bh / H, h = bh % H, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int f = blockIdx.y * 32 + lane;
    const float *cs = csum + ((long long)b * Hkv + h / (H / Hkv)) * Tn * NF + f;
    const float *ss = selsum + (long long)bh * n_routed * NF + f;
    float *z = zpre + (long long)bh * n_routed * NF + f;
    const float *leaving = all_selected ? cs : ss;
    constexpr int kAhead = 8;   // chunks whose sums are requested together
    auto deltas = [&](int c, int c1, float (&d)[kAhead]) {   // of chunks c .. (zero from c1 on)
        float a[kAhead], b[kAhead], w[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            a[i] = b[i] = w[i] = 0.f;
            const bool in = c + i < c1;
            if (in && !all_selected) {
                a[i] = cs[(long long)(c + i) * NF];
                b[i] = ss[(long long)(c + i) * NF];
            }
            if (in && window > 0 && c + i >= window) w[i] = leaving[(long long)(c + i - window) * NF];
        }
#pragma unroll
        for (int i = 0; i < kAhead; ++i) d[i] = (a[i] - b[i]) + w[i];
    };
    const int warps = blockDim.x >> 5, per = (n_routed + warps - 1) / warps, c0 = warp * per, c1 = min(c0 + per, n_routed);
    float acc = 0.f, d[kAhead];
    for (int c = c0; c < c1; c += kAhead) {
        deltas(c, c1, d);
#pragma unroll
        for (int i = 0; i < kAhead; ++i) acc += d[i];
    }
    part[warp][lane] = acc;
    __syncthreads();
    acc = 0.f;
    for (int w = 0; w < warp; ++w) acc += part[w][lane];
    for (int c = c0; c < c1; c += kAhead) {
        deltas(c, c1, d);
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            acc += d[i];
            if (c + i < c1) z[(long long)(c + i) * NF] = acc;
        }
    }
    if (z_out != nullptr && warp == warps - 1) z_out[(long long)bh * NF + f] = acc;
}

// ------------------------------------------------------------------------------------------
// State scan with the query-side NP-Map fused into its loads
// ------------------------------------------------------------------------------------------
// One CTA owns one (batch, query head) and one half of the feature dimension: the softmax(u) half or the
// softmax(-u) half of phi (each d_f features).  N_LA and D_LA are sums over features, so the two CTAs of a
// head produce two partial results that the merge epilogue of the attention kernel adds.
template <int D, int DF>
struct FusedPlan {
    static constexpr int kW = D * DF * 2;               // W_q, MN-major (as TMA delivers [d rows, d_f columns])
    static constexpr int kX = 128 * D * 2;              // raw Q rows of one block of 128 tokens
    static constexpr int kPhiQ = 64 * DF * 4;           // phi_q half of 64 tokens, fp32 (TF32 operand)
    static constexpr int kUTok = 32;                    // tokens per state-update tile
    static constexpr int kUStages = 4;                  // ring of update tiles (loads run this far ahead of the MMAs)
    // ... of the pass that only sums, whose ring takes the room of W_q, Q and phi(Q) too: it does nothing but wait for its loads
    // (with four stages 920 cycles a tile; 32768 tokens x 32 heads, d = 128: 136 us, with twelve 101).
    static constexpr int kMaxStages = 12;
    static constexpr int kPhiK = kUTok * DF * 2;        // phi_k half of an update tile, bf16
    static constexpr int kVt = kUTok * D * 2;           // V of an update tile
    static constexpr int kUStage = kPhiK + kVt;
    static constexpr int oW = 0;
    static constexpr int oX = oW + kW;
    static constexpr int oQ = oX + kX;                  // two slots
    static constexpr int oU = oQ + 2 * kPhiQ;           // kUStages stages
    static constexpr int oDinv = oU + kUStages * kUStage;      // [8][64] 1 / D_part of the tokens of the last sub-chunks
    static constexpr int oZ = oDinv + 8 * 64 * 4;       // [4 map warps][d_f] z half of the chunk two back
    static constexpr int oStage = oZ + 4 * DF * 4;      // [64 tokens][d] bf16: the output of a sub-chunk on its way out
    static constexpr int oBar = oStage + 64 * D * 2;
    static constexpr int kSumStages = (oDinv / kUStage) < kMaxStages ? oDinv / kUStage : kMaxStages;
    static constexpr int kNumBars = 18 + 3 * kMaxStages;
    static constexpr int oMisc = oBar + kNumBars * 8;
    static constexpr int kTotal = oMisc + 16;
};
static_assert(FusedPlan<128, 128>::kTotal <= 232448 && FusedPlan<128, 64>::kTotal <= 232448 && FusedPlan<64, 64>::kTotal <= 232448,
              "fused scan: the shared-memory plan exceeds what a CTA can have");
static_assert(FusedPlan<128, 128>::oStage % 1024 == 0 && FusedPlan<128, 64>::oStage % 1024 == 0 && FusedPlan<64, 64>::oStage % 1024 == 0,
              "fused scan: the staging tile is swizzle-aligned");

// What a launch of la_fused_kernel does (see there).  Folding again is a kernel of its own: beside the code for it the others
// took 1 to 2 % longer (128 heads x 4096 tokens, d = 64, a quarter kept: 512 -> 518 us a call).
enum LaMode { kFromSums, kSumsOnly, kFoldAll };

template <int D, int DF, bool kFoldAgain>
__global__ void __launch_bounds__(384, 1)
la_fused_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_wq,
                const __grid_constant__ CUtensorMap tm_phik, const __grid_constant__ CUtensorMap tm_v,
                const __grid_constant__ CUtensorMap tm_phiks, const __grid_constant__ CUtensorMap tm_vs,
                const __grid_constant__ CUtensorMap tm_y0, const __grid_constant__ CUtensorMap tm_y1,   // (a map per part: rows in 31 bits)
                const __nv_bfloat16 *bq, const __nv_bfloat16 *G,
                const int32_t *sel_idx, const float *zpre, __nv_bfloat16 *y_part,
                float *d_part, float *S_out, float *seg_sums, int *status, int H, int Hkv,
                int N, int C, int lam, int window, long long part_stride_y, long long part_stride_d, int seg_chunks, int n_seg,
                int sum_parts, int sums_pass, int sel_rows) {
    grid_dep_wait();
    grid_dep_launch();
    using P = FusedPlan<D, DF>;
    constexpr int NF = 2 * DF;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + P::oBar);
    uint64_t *w_full = bars, *x_full = bars + 1, *x_empty = bars + 2;
    uint64_t *f_done = bars + 15, *f_free = bars + 3;   // [2] each: f of even / odd blocks
    uint64_t *pq_full = bars + 5, *pq_empty = bars + 7, *r_done = bars + 9, *out_free = bars + 11, *fin = bars + 13;
    uint64_t *init_done = bars + 14, *u_full = bars + 18, *u_empty = u_full + P::kMaxStages, *u_masked = u_empty + P::kMaxStages;
    constexpr int kUTok = P::kUTok;
    const LaMode mode = kFoldAgain ? kFoldAll : sums_pass ? kSumsOnly : kFromSums;
    const bool sums_only = mode == kSumsOnly;
    const int n_stages = sums_only ? P::kSumStages : P::kUStages;
    uint8_t *ring = smem + (sums_only ? 0 : P::oU);
    // The ring stage of a tile, and the parity of its round; next: of the tile n further on (n <= n_stages).
    struct Slot {
        int stage, parity;
        __device__ __forceinline__ void next(int n, int n_stages) {
            stage += n;
            if (stage >= n_stages) {
                stage -= n_stages;
                parity ^= 1;
            }
        }
    };
    // Chunk of a tile and its number among the chunk's (counted up from tile to tile: a division by the tiles of a chunk costs
    // a single-thread role more than the tile's loads)
    struct Tile {
        int chunk, rt;
        __device__ __forceinline__ void next(int n, int per_chunk) {
            rt += n;
            if (rt >= per_chunk) {
                rt -= per_chunk;
                ++chunk;
            }
        }
    };
    uint32_t *tmem_base_slot = reinterpret_cast<uint32_t *>(smem + P::oMisc);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + P::oMisc + 8);
    float *dinv_ring = reinterpret_cast<float *>(smem + P::oDinv);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (known to be the same in all lanes)
    const int bh = blockIdx.x, b = bh / H, h = bh % H, kvh = h / (H / Hkv);
    const int half = blockIdx.y;                // 0: features softmax(u), 1: features softmax(-u)
    const int sc = C / 64;                      // 64-token sub-chunks per chunk
    const int Tn = (N + C - 1) / C;
    const int n_routed = Tn >= 3 ? Tn - 2 : 0;  // chunks whose tokens enter the state
    // The sequence is cut into n_seg segments of seg_chunks chunks (two-level scan): segment g answers the
    // sub-chunks [u_first, NU) and performs the updates that fall between them, starting from the sum of the
    // earlier segments' updates (kFromSums: seg_sums, produced by a first pass of this kernel, kSumsOnly), or folding
    // the chunks before it itself (kFoldAll, where they are few).
    // The first pass cuts every segment into sum_parts pieces, one CTA each (it has no scan to keep in order, and
    // the pieces fill the SMs that the n_seg - 1 summed segments alone would leave idle).  A segment that folds itself
    // forms the same pieces, one after the other, each from zero, and adds them up in fp32 as the other does: carried
    // through the accumulators, the state would take their rounding (with exact features and positive values S was 5 to 47 %
    // further from float64 than as the sum of the pieces: 2.05e-7 and 1.39e-7 for 16 heads x 2048 tokens, d = 128), and how a
    // call is launched would show in its results.
    const int seg = blockIdx.z;
    const int piece_chunks = seg_chunks / sum_parts;
    if (sums_only) seg_chunks = piece_chunks;
    const int NU_all = (N + 63) / 64;           // sub-chunks with query rows
    const int u_first = seg == 0 ? 2 * sc : seg * seg_chunks * sc;   // the first two chunks see an empty state
    const int NU = (!sums_only && seg == n_seg - 1) ? NU_all : min(NU_all, (seg + 1) * seg_chunks * sc);
    const int b_first = u_first / 2;            // blocks of 128 query rows: [b_first, NB)
    const int NB = sums_only ? b_first : (NU + 1) / 2;
    // Update tiles of kUTok tokens: per routed chunk its su tiles (selected rows zeroed) and, with a salient-cache
    // budget of `window` chunks, the su tiles of the chunk `window` back with everything but its selected rows
    // zeroed: those tokens leave the cache for the state when the chunk is routed.
    // With sel_rows > 0 the leaving tokens come from the gathered copies of their phi(K) and V rows (sel_rows rows
    // per head, lam per chunk): nl tiles per chunk instead of su, and only a last partial tile has rows to clear.
    const int su = C / kUTok;
    const int nl = sel_rows > 0 ? (lam + kUTok - 1) / kUTok : su;
    const int per_chunk = window > 0 ? su + nl : su;
    const int chunk0 = mode == kFoldAll ? 0 : u_first / sc - 2;   // first chunk that the segment folds
    const int n_upd = NU > u_first ? ((NU - 1) / sc - 1 - chunk0) * per_chunk : 0;
    const bool has_init = mode == kFromSums && seg > 0;
    // Pieces of what a segment folds before its own updates, one after the other (a pass of sums has one).  The sequence's first two chunks answer nothing, so the first
    // piece is two chunks shorter than the others: with pieces of two chunks it is empty and there is one less.
    const int n_pieces = sums_only ? 1 : mode == kFoldAll && n_upd > 0 ? seg * sum_parts - (seg > 0 && piece_chunks == 2 ? 1 : 0) : 0;
    __nv_bfloat16 *y_out = y_part + (long long)half * part_stride_y;
    float *d_out = d_part + (long long)half * part_stride_d;

    if ((smem_u32(smem) & 1023u) != 0) {
        if (threadIdx.x == 0) report_status(status, STILL_ERR_DEVICE_TIMEOUT, 97);
        return;
    }
    if (threadIdx.x == 0) *abort_flag = *reinterpret_cast<volatile int *>(status) != 0;
    __syncthreads();
    if (*abort_flag) return;
    __syncthreads();
    if (threadIdx.x == 0) {
        mbar_init(w_full, 1);
        mbar_init(x_full, 1);
        mbar_init(x_empty, 5);      // the f GEMM has read the rows (1) and so have the four map warps (4)
        for (int i = 0; i < 2; ++i) {
            mbar_init(f_done + i, 1);
            mbar_init(f_free + i, 4);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(pq_full + i, 2);   // the two map warps that own the slot's 64 rows
            mbar_init(pq_empty + i, 1);
            mbar_init(r_done + i, 1);
            mbar_init(out_free + i, 4);
        }
        for (int i = 0; i < P::kMaxStages; ++i) {
            mbar_init(u_full + i, 1);
            mbar_init(u_empty + i, 1);
            mbar_init(u_masked + i, 1);
        }
        mbar_init(fin, 1);
        mbar_init(init_done, 4);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_base_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_base_slot, 0);
    // TMEM columns: S^T half [value lanes x d_f features] fp32; f = x W_q of a block [128 rows x d_f]; two read-out
    // results [value lanes x 64 tokens]
    constexpr uint32_t col_state = 0, col_f = DF, col_out = 3 * DF;   // f: two buffers of DF columns
    // Pieces behind the first are formed where the second f and the read-outs will lie, by turns, and are handed to the
    // workers over the barriers of the read-outs: hand-over n (a piece or a read-out) uses r_done / out_free [n & 1].
    static_assert(DF <= 128, "fused scan: a piece's sum takes the columns of both read-outs");
    auto col_piece = [&](int n) -> uint32_t { return (n & 1) ? col_out : col_f + DF; };

    // Registers move from the first warpgroup (single-thread roles) to the map warps, whose threads hold a row of f
    // (per scheduler: 72 + 160 + 224 registers for its three warps, of the 3 x 168 the CTA was launched with).
    if (warp < 4) {
    reg_dec<72>();
    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            const int kv_row0 = (b * Hkv + kvh) * N, q_row0 = bh * N;
            const int n_blk = NB > b_first ? NB - b_first : 0;
            if (n_blk > 0) {
                mbar_expect_tx(w_full, P::kW);
                for (int a = 0; a < DF / 64; ++a) tma_load_2d(smem + P::oW + a * (D * 128), &tm_wq, w_full, a * 64, h * D);
            }
            int nu = 0, nx = 0, spins = 0;
            Slot us{0, 0};
            Tile ut{chunk0, 0};
            long long t0 = clock64();
            while (nu < n_upd || nx < n_blk) {
                bool progressed = false;
                if (nx < n_blk && mbar_try_wait(x_empty, (nx & 1) ^ 1)) {
                    mbar_expect_tx(x_full, P::kX);
                    for (int a = 0; a < D / 64; ++a)   // K-major, 64-element atoms 128 rows apart
                        tma_load_2d(smem + P::oX + a * (128 * 128), &tm_q, x_full, a * 64, q_row0 + (b_first + nx) * 128);
                    ++nx;
                    progressed = true;
                }
                if (nu < n_upd && mbar_try_wait(u_empty + us.stage, us.parity ^ 1)) {
                    uint8_t *stg = ring + us.stage * P::kUStage;
                    // a leaving-tile reads the chunk `window` back (before there is one, any valid tile: all its rows are zeroed)
                    const bool leaving = ut.rt >= su, gathered = leaving && sel_rows > 0;
                    const int src = leaving && ut.chunk >= window ? ut.chunk - window : ut.chunk, tile = leaving ? ut.rt - su : ut.rt;
                    // first row of the tile: in phi(K) / V of the KV head, or in the head's gathered rows
                    const int row = gathered ? bh * sel_rows + src * lam + tile * kUTok : kv_row0 + (src * su + tile) * kUTok;
                    const CUtensorMap *mp = gathered ? &tm_phiks : &tm_phik, *mv = gathered ? &tm_vs : &tm_v;
                    mbar_expect_tx(u_full + us.stage, P::kUStage);
                    for (int a = 0; a < DF / 64; ++a)  // phi(K) half: MN-major, 64-feature atoms kUTok rows apart
                        tma_load_2d(stg + a * (kUTok * 128), mp, u_full + us.stage, half * DF + a * 64, row);
                    for (int a = 0; a < D / 64; ++a)   // V: M-major A operand, 64-column atoms kUTok rows apart
                        tma_load_2d(stg + P::kPhiK + a * (kUTok * 128), mv, u_full + us.stage, a * 64, row);
                    us.next(1, n_stages);
                    ut.next(1, per_chunk);
                    ++nu;
                    progressed = true;
                }
                if (progressed) {
                    spins = 0;
                } else if ((++spins & 1023) == 0) {
                    if (spins == 1024) t0 = clock64();
                    if (*abort_flag) break;
                    if (clock64() - t0 > kWaitLimitCycles) {
                        *abort_flag = 1;
                        report_status(status, STILL_ERR_DEVICE_TIMEOUT, 60);
                        break;
                    }
                }
            }
            const long long t1 = clock64();
            if (n_blk > 0) mbar_wait_drain(w_full, 0, t1);
            mbar_drain_ring(x_full, 1, nx, t1);
            mbar_drain_ring(u_full, n_stages, nu, t1);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        // The whole warp walks the schedule and waits on the barriers; one elected lane issues (control flow and
        // descriptors stay the same in all lanes and can live in uniform registers, where the tensor-core
        // instructions take their operands from).  A failed wait does not leave the loops: it switches off the
        // remaining waits and instructions, and the loops run out.
        {
            const bool leader = elect_one();
            constexpr uint32_t idesc_f = make_idesc(128, DF, true);
            constexpr uint32_t idesc_upd = make_idesc(128, DF, true) | (1u << 15);  // A M-major, B MN-major
            constexpr uint32_t idesc_rd = make_idesc_tf32(128, 64);
            bool ok = true;
            int nu = 0, nq = 0, nx = 0;
            Slot us{0, 0};
            auto wait = [&](uint64_t *bar, int parity, int where) {
                if (ok) ok = mbar_wait(bar, (uint32_t)parity, abort_flag, status, where);
            };
            // descriptors as low words: a k-step adds a constant
            const uint32_t x_lo = desc_lo(smem_u32(smem + P::oX), 0), w_lo = desc_lo(smem_u32(smem + P::oW), D * 128);
            const uint32_t q_lo0 = desc_lo(smem_u32(smem + P::oQ), 0);
            const uint32_t pk_lo0 = desc_lo(smem_u32(ring), kUTok * 128);
            const uint32_t v_lo0 = desc_lo(smem_u32(ring + P::kPhiK), D == 128 ? kUTok * 128 : 0);
            // f = x W_q of block b_first + nx (the map warps have taken the previous f out of tensor memory)
            auto issue_f = [&]() {
                if (nx == 0) wait(w_full, 0, 61);
                wait(x_full, nx & 1, 62);
                wait(f_free + (nx & 1), ((nx >> 1) & 1) ^ 1, 63);
                tc_fence_after();
                if (leader && ok) {
#pragma unroll
                    for (int k = 0; k < D / 16; ++k) {
                        const uint32_t xo = ((k / 4) * (128 * 128) + (k % 4) * 32) >> 4, wo = (k * (16 * 128)) >> 4;
                        if (k == 0) mma_ss_lo<idesc_f, 0>(tmem_base + col_f + (nx & 1) * DF, x_lo + xo, w_lo + wo);
                        else mma_ss_lo<idesc_f, 1>(tmem_base + col_f + (nx & 1) * DF, x_lo + xo, w_lo + wo);
                    }
                    tc_commit(f_done + (nx & 1));
                    tc_commit(x_empty);
                }
                ++nx;
            };
            if (has_init) {   // the workers have put the sum of the earlier segments into tensor memory
                wait(init_done, 0, 73);
                tc_fence_after();
            }
            auto issue_update = [&](uint32_t col, bool add) {   // into, or over, the sum at these columns
                wait(u_masked + us.stage, us.parity, 64);
                tc_fence_after();
                const uint32_t so = (uint32_t)us.stage * (P::kUStage >> 4);
                if (leader && ok) {
                    mma_ss_lo_acc<idesc_upd>(tmem_base + col, v_lo0 + so, pk_lo0 + so, add ? 1u : 0u);
#pragma unroll
                    for (int k = 1; k < kUTok / 16; ++k)   // 16 tokens per step: 16 rows of 128 bytes in both operands
                        mma_ss_lo_acc<idesc_upd>(tmem_base + col, v_lo0 + so + k * (2048 >> 4), pk_lo0 + so + k * (2048 >> 4), 1u);
                    tc_commit(u_empty + us.stage);
                }
                us.next(1, n_stages);
                ++nu;
            };
            if (NB > b_first) issue_f();
            for (int g = 0; g < n_pieces; ++g) {
                const int tiles = sums_only ? n_upd : (g == 0 && piece_chunks > 2 ? piece_chunks - 2 : piece_chunks) * per_chunk;
                const uint32_t col = g == 0 ? col_state : col_piece(nq);
                if (g > 0) wait(out_free + (nq & 1), ((nq >> 1) & 1) ^ 1, 74);
                for (int i = 0; i < tiles; ++i) issue_update(col, i > 0);
                if (g > 0) {
                    if (leader && ok) tc_commit(r_done + (nq & 1));
                    ++nq;
                }
            }
            if (n_pieces > 1) wait(out_free + ((nq - 1) & 1), ((nq - 1) >> 1) & 1, 75);   // the last has been added
            for (int u = u_first; u < NU && !sums_only; ++u) {
                if (u % sc == 0) {
                    // the chunk that has just left the local region: sub-chunks of chunk u / sc - 2
                    for (int j = 0; j < per_chunk; ++j) issue_update(col_state, nu > 0 || has_init);
                }
                // The next block's f = x W_q goes out as soon as its rows have arrived and the map warps have taken the
                // current f out of tensor memory: it is then ready when they finish the current block.  (Issued after
                // this block's read-out, it made the map warps wait for a round trip through this warp per block.)
                if ((u & 1) == 0 && b_first + nx < NB) issue_f();
                wait(pq_full + (u & 1), ((u - u_first) >> 1) & 1, 65);   // (u_first is even)
                wait(out_free + (nq & 1), ((nq >> 1) & 1) ^ 1, 66);
                tc_fence_after();
                const uint32_t q_lo = q_lo0 + (uint32_t)(u & 1) * (P::kPhiQ >> 4), d_out_t = tmem_base + col_out + (nq & 1) * 64;
                if (leader && ok) {
#pragma unroll
                    for (int k = 0; k < DF / 8; ++k) {   // 8 features per step: 32 bytes within a 32-feature atom
                        const uint32_t qo = ((k / 4) * (64 * 128) + (k % 4) * 32) >> 4;
                        if (k == 0) mma_ts_tf32_lo<idesc_rd, 0>(d_out_t, tmem_base + col_state, q_lo + qo);
                        else mma_ts_tf32_lo<idesc_rd, 1>(d_out_t, tmem_base + col_state + k * 8, q_lo + qo);
                    }
                    tc_commit(r_done + (nq & 1));
                    tc_commit(pq_empty + (u & 1));
                }
                ++nq;
            }
            // state after the last update, for the decode state; after a failure, nothing issued may still run
            if (leader) tc_commit(fin);
            if (!__all_sync(0xffffffffu, ok) && leader) mbar_wait_drain(fin, 0);
        }
    } else {
        // ------------------------------------------------------------ mask warps (2 and 3: alternate tiles)
        // Zeroes, in every phi(K) tile, the rows of the tokens kept for softmax attention: only the others enter the
        // state.  The indices of a tile's chunk are requested one tile ahead (a round trip to L2 per tile would
        // otherwise pace the whole update path), and two warps take turns.
        bool ok = true;
        // positions of the selected tokens of a tile's chunk relative to the tile's first row (-1: none)
        auto fetch = [&](bool live, const Tile &ut, int (&r)[4]) {
            const bool leaving = ut.rt >= su;
            const int chunk = leaving ? ut.chunk - window : ut.chunk;   // (chunk < 0: nothing leaves yet, every row is zeroed)
            const int first = chunk * C + (leaving ? ut.rt - su : ut.rt) * kUTok;
            const bool need = live && chunk >= 0 && !(leaving && sel_rows > 0);   // (a gathered tile needs no indices)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = lane + 32 * q;
                r[q] = need && i < lam ? sel_idx[((long long)bh * Tn + chunk) * lam + i] - first : -1;
            }
        };
        auto process = [&](const Slot &us, const Tile &ut, const int (&sel)[4]) {
            const bool leaving = ut.rt >= su;                    // tile of the tokens that leave the salient cache
            // the selected rows of the tile as a 32-bit set
            uint32_t rows = 0u;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (sel[q] >= 0 && sel[q] < kUTok) rows |= 1u << sel[q];
            rows = __reduce_or_sync(0xffffffffu, rows);
            if (leaving) rows = ~rows;                           // rows to zero: the selected ones, or all the others
            if (leaving && sel_rows > 0) {
                // gathered tile: its first `valid` rows are the chunk's leaving tokens, the rest belong to the next chunk
                const int valid = ut.chunk < window ? 0 : min(kUTok, lam - (ut.rt - su) * kUTok);
                rows = valid >= 32 ? 0u : ~((1u << valid) - 1u);
            }
            if (ok) ok = mbar_wait(u_full + us.stage, us.parity, abort_flag, status, 67);
            ok = __all_sync(0xffffffffu, ok);
            if (ok) {
                // A row is 128 bytes in each 64-feature atom.  Eight lanes clear one such line (all 32 banks, no
                // conflict), so a store instruction clears the lines of four rows.
                uint8_t *tile = ring + us.stage * P::kUStage;
#pragma unroll
                for (int it = 0; it < kUTok / 4; ++it) {
                    const int rz = it * 4 + (lane >> 3);
                    if ((rows >> rz) & 1u) {
#pragma unroll
                        for (int a = 0; a < DF / 64; ++a)
                            *reinterpret_cast<uint4 *>(tile + a * (kUTok * 128) + rz * 128 + ((lane & 7) << 4)) = make_uint4(0, 0, 0, 0);
                    }
                }
                fence_proxy_async();
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(u_masked + us.stage);
        };
        // (two register sets that change roles: a copy from one to the other would wait for the loads)
        int sel_a[4], sel_b[4];
        Slot us{0, 0};
        Tile ut{chunk0, 0}, ft{chunk0, 0};   // of the next tile to process, and to fetch for
        if (warp == 3) {
            us.next(1, n_stages);
            ut.next(1, per_chunk);
            ft.next(1, per_chunk);
        }
        auto turn = [&](const int (&sel)[4]) {
            process(us, ut, sel);
            us.next(2, n_stages);
            ut.next(2, per_chunk);
        };
        fetch(warp - 2 < n_upd, ft, sel_a);
        for (int nu = warp - 2; nu < n_upd; nu += 4) {
            ft.next(2, per_chunk);
            fetch(nu + 2 < n_upd, ft, sel_b);
            turn(sel_a);
            ft.next(2, per_chunk);
            fetch(nu + 4 < n_upd, ft, sel_a);
            if (nu + 2 < n_upd) turn(sel_b);
        }
    }
    } else if (warp < 8) {
        reg_dec<160>();
        // ------------------------------------------------------------ workers: output
        const int wq = warp & 3;                     // TMEM lane quarter this warp may read
        const int e = wq * 32 + lane;                // value column (lane of S^T and of the read-out result)
        const uint32_t taddr = tmem_base + ((uint32_t)(wq * 32) << 16);
        const int tid = threadIdx.x - 128;           // 0..127
        bool ok = true;
        int nq = 0;
        for (int g = 1; g < n_pieces; ++g, ++nq) {
            if (ok) ok = mbar_wait(r_done + (nq & 1), (nq >> 1) & 1, abort_flag, status, 76);
            ok = __all_sync(0xffffffffu, ok);
            if (ok) {   // (the commit behind a piece's updates covers those of the pieces before it)
                tc_fence_after();
#pragma unroll 1
                for (int q = 0; q < DF / 32; ++q) {
                    uint32_t sum[32], add[32];
                    tmem_ld32(taddr + col_state + q * 32, sum);
                    tmem_ld32(taddr + col_piece(nq) + q * 32, add);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 32; ++j) sum[j] = __float_as_uint(__uint_as_float(sum[j]) + __uint_as_float(add[j]));
                    tmem_st32(taddr + col_state + q * 32, sum);
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(out_free + (nq & 1));
            }
        }
        // rows of the first two chunks see an empty state
        if (seg == 0 && !sums_only) {
            const int n0 = min(N, 2 * C);
            for (int i = tid; i < n0 * (D / 8); i += 128)
                reinterpret_cast<uint4 *>(y_out + (long long)bh * N * D)[i] = make_uint4(0, 0, 0, 0);
            for (int t = tid; t < n0; t += 128) d_out[(long long)bh * N + t] = 0.f;
        }
        if (has_init) {
            // S^T of this segment starts as the sum of the earlier segments' updates: lane e, column f <- sum_g P_g[f][e]
            const float *P0 = seg_sums + (((long long)bh * 2 + half) * ((n_seg - 1) * sum_parts)) * (DF * D);
            const int n_sums = seg * sum_parts;
#pragma unroll 1
            for (int q = 0; q < DF / 32; ++q) {
                // (a sum's 32 columns are requested together, two sums at a time: requested one value at a time, the
                // start of a segment took 90 us)
                uint32_t sreg[32];
                float acc[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) acc[j] = 0.f;
                if (e < D) {
                    const float *Pq = P0 + (q * 32) * D + e;
#pragma unroll 2
                    for (int g2 = 0; g2 < n_sums; ++g2)
#pragma unroll
                        for (int j = 0; j < 32; ++j) acc[j] += Pq[(long long)g2 * (DF * D) + j * D];
                }
#pragma unroll
                for (int j = 0; j < 32; ++j) sreg[j] = __float_as_uint(acc[j]);
                tmem_st32(taddr + col_state + q * 32, sreg);
            }
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(init_done);
        }
        constexpr int kPiecesPerRow = D / 8, kPieces = 64 * kPiecesPerRow / 128;   // 16-byte pieces per thread and sub-chunk
        for (int u = u_first; u < NU && !sums_only; ++u) {
            // the gate of the sub-chunk, requested before the wait (requested where it is used, a chain of round trips
            // to memory: the layer's 1003-token prompt spent 20 us of its scan on it)
            uint4 gate[kPieces];
            if (G != nullptr) {
#pragma unroll
                for (int it = 0; it < kPieces; ++it) {
                    const int id = it * 128 + tid, t = min(u * 64 + id / kPiecesPerRow, N - 1);
                    gate[it] = *reinterpret_cast<const uint4 *>(G + ((long long)bh * N + t) * D + (id % kPiecesPerRow) * 8);
                }
            }
            if (ok) ok = mbar_wait(r_done + (nq & 1), (nq >> 1) & 1, abort_flag, status, 68);
            ok = __all_sync(0xffffffffu, ok);
            // y_part[t][e] = N_part / D_part (times the gate): the read-out scaled by 1 / (e . z) of its token.  Tensor memory
            // holds it by value column, y_part is token-major.  Read as fragments of 8 x 8 (value columns g and g + 8 of 16,
            // tokens 8 i + 2 tig and + 1 in a thread), two tokens are a register of bf16, and stmatrix transposes on the way
            // to shared memory: 8 stores a thread for a sub-chunk where a thread per value column needs 64 of two bytes.  Rows
            // lie there as the tensor map has them (64 columns of 128 bytes, swizzled by the row), and one thread stores the
            // tile.  The workers, which were as busy as the map warps (3300 cycles a sub-chunk), now wait for half of the
            // time: 64 heads x 32768 tokens, a quarter kept, 6020 -> 5800 us a call.
            uint32_t out[2][16];
            uint8_t *stg = smem + P::oStage;
            const bool has_rows = wq * 32 < D;   // (at d = 64 the upper lanes of the product repeat the lower)
            if (ok) {
                tc_fence_after();
                const float *dinv = dinv_ring + (u & 7) * 64 + 2 * (lane & 3);
                if (has_rows) {
#pragma unroll
                    for (int h16 = 0; h16 < 2; ++h16) {
                        uint32_t o[32];
                        tmem_ld_frag64(taddr + col_out + (nq & 1) * 64 + ((uint32_t)(h16 * 16) << 16), o);
                        float2 sc2[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) sc2[i] = *reinterpret_cast<const float2 *>(dinv + 8 * i);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            out[h16][2 * i] = pack_bf16(__uint_as_float(o[4 * i]) * sc2[i].x, __uint_as_float(o[4 * i + 1]) * sc2[i].y);
                            out[h16][2 * i + 1] = pack_bf16(__uint_as_float(o[4 * i + 2]) * sc2[i].x, __uint_as_float(o[4 * i + 3]) * sc2[i].y);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(out_free + (nq & 1));
            }
            if (tid == 0) bulk_store_wait_read();            // the store of the sub-chunk before has read the staging tile
            asm volatile("bar.sync 2, 128;" ::: "memory");   // the four worker warps (always, whatever `ok`)
            if (ok && has_rows) {
#pragma unroll
                for (int h16 = 0; h16 < 2; ++h16)
#pragma unroll
                    for (int i = 0; i < 8; i += 2) {
                        // this lane's row of the four matrices: tokens 8 i .. + 7 and + 8 .. + 15, columns 0-7 and 8-15 of the 16
                        const int t = 8 * (i + (lane >> 4)) + (lane & 7), p = wq * 4 + h16 * 2 + ((lane >> 3) & 1);
                        stmatrix_x4_trans(stg + (p >> 3) * (64 * 128) + t * 128 + (((p & 7) ^ (t & 7)) << 4), out[h16][2 * i],
                                          out[h16][2 * i + 1], out[h16][2 * i + 2], out[h16][2 * i + 3]);
                    }
                fence_proxy_async();
            }
            asm volatile("bar.sync 2, 128;" ::: "memory");
            if (ok) {
                const int base = u * 64;
                if (G == nullptr && base + 64 <= N) {
                    if (tid == 0) {
#pragma unroll
                        for (int a = 0; a < D / 64; ++a) tma_store_2d(half ? &tm_y1 : &tm_y0, stg + a * (64 * 128), a * 64, bh * N + base);
                        bulk_store_commit();
                    }
                } else {   // with a gate, and the last rows of a sequence
#pragma unroll
                    for (int it = 0; it < kPieces; ++it) {
                        const int id = it * 128 + tid, t = id / kPiecesPerRow, c = id % kPiecesPerRow;
                        if (base + t < N) {
                            uint4 v = *reinterpret_cast<const uint4 *>(stg + (c >> 3) * (64 * 128) + t * 128 + (((c & 7) ^ (t & 7)) << 4));
                            if (G != nullptr) {
                                const uint4 gg = gate[it];
                                const uint32_t vw[4] = {v.x, v.y, v.z, v.w}, gw[4] = {gg.x, gg.y, gg.z, gg.w};
                                uint32_t rw[4];
#pragma unroll
                                for (int q = 0; q < 4; ++q)
                                    rw[q] = pack_bf16(__uint_as_float(vw[q] << 16) * __uint_as_float(gw[q] << 16),
                                                      __uint_as_float(vw[q] & 0xffff0000u) * __uint_as_float(gw[q] & 0xffff0000u));
                                v = make_uint4(rw[0], rw[1], rw[2], rw[3]);
                            }
                            *reinterpret_cast<uint4 *>(y_out + ((long long)bh * N + base + t) * D + c * 8) = v;
                        }
                    }
                }
            }
            ++nq;
        }
        if (tid == 0) bulk_store_wait();
        // the state after the segment's last update: the segment's own sum for the second pass (sums_only), or,
        // from the last segment, S [2 d_f, d] of the decode state (this CTA's features)
        float *S_dst = nullptr;
        if (sums_only) S_dst = seg_sums + (((long long)bh * 2 + half) * ((n_seg - 1) * sum_parts) + seg) * (DF * D);
        else if (S_out != nullptr && seg == n_seg - 1) S_dst = S_out + ((long long)bh * NF + half * DF) * D;
        if (S_dst != nullptr) {
            if (n_upd > 0 || has_init) {
                if (ok) ok = mbar_wait(fin, 0, abort_flag, status, 69);
                ok = __all_sync(0xffffffffu, ok);
                if (ok) {
                    tc_fence_after();
#pragma unroll 1
                    for (int q = 0; q < DF / 32; ++q) {
                        uint32_t sreg[32];
                        tmem_ld32(taddr + col_state + q * 32, sreg);
                        tmem_wait_ld();
                        if (e < D) {
#pragma unroll
                            for (int j = 0; j < 32; ++j) S_dst[(q * 32 + j) * D + e] = __uint_as_float(sreg[j]);
                        }
                    }
                }
            } else {
                for (int i = tid; i < DF * D; i += 128) S_dst[i] = 0.f;
            }
        }
    } else {
        reg_inc<224>();
        // ------------------------------------------------------------ map warps: phi_q of a block of 128 rows
        // A thread owns one row: u = (f + b) ||x|| / max(||f + b||, 1e-12); this CTA's half of phi is softmax(u) or
        // softmax(-u) over all d_f features.  The row goes to the slot of its 64-token sub-chunk as fp32, K-major
        // with the 128-byte swizzle the UMMA descriptor expects; D_part = phi_half . z_half of the chunk two back.
        const int wq = warp & 3, r = wq * 32 + lane;   // TMEM lane quarter; row of the block
        const uint32_t taddr = tmem_base + ((uint32_t)(wq * 32) << 16);
        const __nv_bfloat16 *bias = bq != nullptr ? bq + (long long)h * DF : nullptr;
        float *zs = reinterpret_cast<float *>(smem + P::oZ) + (warp - 8) * DF;   // this warp's copy of the z row
        bool ok = true;
        int nx = 0;
        // z half of the chunk two back (every row of the warp dots its features with it): requested a block ahead (a round
        // trip to memory otherwise stood in every block), placed in shared memory when its block begins
        auto request_z = [&](int blk) {
            const int chunk = min(((2 * blk + (r >> 6)) * 64) / C, Tn - 1);   // (a sub-chunk past the end of a ragged last block has no chunk)
            const float *zrow = zpre + ((long long)bh * n_routed + (chunk - 2)) * NF + half * DF;
            return lane < DF / 4 ? reinterpret_cast<const float4 *>(zrow)[lane] : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        float4 zreg = make_float4(0.f, 0.f, 0.f, 0.f);
        if (b_first < NB) zreg = request_z(b_first);
        for (int blk = b_first; blk < NB; ++blk, ++nx) {
            const int u = 2 * blk + (r >> 6);            // this row's sub-chunk; its slot is u & 1 = r >> 6
            const int slot = r >> 6, rr = r & 63;
            if (ok) ok = mbar_wait(x_full, nx & 1, abort_flag, status, 70);
            ok = __all_sync(0xffffffffu, ok);
            float nx2 = 0.f;
            if (ok) {
                float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int a = 0; a < D / 64; ++a)
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(smem + P::oX + a * (128 * 128) + r * 128 + ((c ^ (r & 7)) << 4));
                        const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float lo = __uint_as_float(w4[q] << 16), hi = __uint_as_float(w4[q] & 0xffff0000u);
                            s4[q] = fmaf(lo, lo, s4[q]);
                            s4[q] = fmaf(hi, hi, s4[q]);
                        }
                    }
                nx2 = (s4[0] + s4[1]) + (s4[2] + s4[3]);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(x_empty);
            if (lane < DF / 4) reinterpret_cast<float4 *>(zs)[lane] = zreg;
            if (blk + 1 < NB) zreg = request_z(blk + 1);
            // f of this block is read from tensor memory twice, 32 columns at a time, in loops that stay rolled: the
            // warp's instruction stream per block is then a few kilobytes.  (With the row held in 128 registers and
            // everything unrolled, instruction fetch was the first stall reason of the kernel.)  f has a buffer per
            // block parity, so the next block's GEMM does not wait for this second reading.
            const uint32_t faddr = taddr + col_f + (nx & 1) * DF;
            if (ok) ok = mbar_wait(f_done + (nx & 1), (nx >> 1) & 1, abort_flag, status, 71);
            ok = __all_sync(0xffffffffu, ok);
            float sgn = 0.f, shift = 0.f;
            if (ok) {
                tc_fence_after();
                // (packed arithmetic and four independent chains each; this CTA's half needs only one extremum:
                // max f for softmax(u), min f for softmax(-u))
                float2 n2[4];
                float ex[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    n2[q] = make_float2(0.f, 0.f);
                    ex[q] = half == 0 ? -INFINITY : INFINITY;
                }
#pragma unroll 1
                for (int q = 0; q < DF / 32; ++q) {
                    float fv[32];
                    tmem_ld32(faddr + q * 32, reinterpret_cast<uint32_t *>(fv));
                    tmem_wait_ld();
                    if (bias != nullptr) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) fv[j] += __bfloat162float(bias[q * 32 + j]);
                    }
#pragma unroll
                    for (int j = 0; j < 32; j += 8) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const float2 v = make_float2(fv[j + 2 * c], fv[j + 2 * c + 1]);
                            n2[c] = __ffma2_rn(v, v, n2[c]);
                            ex[c] = half == 0 ? max3(ex[c], v.x, v.y) : min3(ex[c], v.x, v.y);
                        }
                    }
                }
                const float nf2 = ((n2[0].x + n2[0].y) + (n2[1].x + n2[1].y)) + ((n2[2].x + n2[2].y) + (n2[3].x + n2[3].y));
                const float unit = half == 0 ? 1.f : -1.f;
                const float extreme = half == 0 ? fmaxf(fmaxf(ex[0], ex[1]), fmaxf(ex[2], ex[3]))
                                                : -fminf(fminf(ex[0], ex[1]), fminf(ex[2], ex[3]));   // max of +-f
                // u = f * ratio in the log2 domain; the exponent of this half is +-u - max(+-u) <= 0
                const float ratio = sqrtf(nx2) / fmaxf(sqrtf(nf2), 1e-12f) * 1.4426950408889634f;
                sgn = unit * ratio;
                shift = -extreme * ratio;
            }
            // the slot is written only after the read-out that used it last has completed (every block fills both
            // slots once)
            if (ok) ok = mbar_wait(pq_empty + slot, (nx & 1) ^ 1, abort_flag, status, 72);
            ok = __all_sync(0xffffffffu, ok);
            if (ok) {
                // The features go into the tile unnormalised, e_j = 2^(+-u_j - max): with D_part = (e . z) / sum e and
                // N_part = (e . S) / sum e the output N_part / D_part = (e . S) / (e . z) does not need the sum, so the
                // row is written as it is computed.  The z values of a block of 32 features are loaded before the
                // block's stores (shared-memory loads are kept behind earlier stores).
                uint8_t *tile = smem + P::oQ + slot * P::kPhiQ;
                float2 zs2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, ds2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                const float2 sgn2 = make_float2(sgn, sgn), shift2 = make_float2(shift, shift);
#pragma unroll 1
                for (int q = 0; q < DF / 32; ++q) {          // 32 features: one swizzle atom of the tile
                    float fv[32];
                    tmem_ld32(faddr + q * 32, reinterpret_cast<uint32_t *>(fv));
                    float4 zc[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) zc[i] = *reinterpret_cast<const float4 *>(zs + 32 * q + 4 * i);
                    tmem_wait_ld();
                    if (bias != nullptr) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) fv[j] += __bfloat162float(bias[q * 32 + j]);
                    }
                    uint8_t *row = tile + q * (64 * 128) + rr * 128;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int j = 4 * i;
                        const float2 a0 = __ffma2_rn(make_float2(fv[j], fv[j + 1]), sgn2, shift2);
                        const float2 a1 = __ffma2_rn(make_float2(fv[j + 2], fv[j + 3]), sgn2, shift2);
                        float4 ev;
                        ev.x = ex2(a0.x);
                        ev.y = ex2(a0.y);
                        ev.z = ex2(a1.x);
                        ev.w = ex2(a1.y);
                        zs2[0] = __fadd2_rn(zs2[0], make_float2(ev.x, ev.y));
                        zs2[1] = __fadd2_rn(zs2[1], make_float2(ev.z, ev.w));
                        ds2[0] = __ffma2_rn(make_float2(ev.x, ev.y), make_float2(zc[i].x, zc[i].y), ds2[0]);
                        ds2[1] = __ffma2_rn(make_float2(ev.z, ev.w), make_float2(zc[i].z, zc[i].w), ds2[1]);
                        // features 4 i .. 4 i + 3 of the atom: 16-byte piece i, swizzled by the row
                        *reinterpret_cast<float4 *>(row + ((i ^ (rr & 7)) << 4)) = ev;
                    }
                }
                tc_fence_before();
                const float zsum = (zs2[0].x + zs2[0].y) + (zs2[1].x + zs2[1].y), draw = (ds2[0].x + ds2[0].y) + (ds2[1].x + ds2[1].y);
                const int t = u * 64 + rr;
                if (t < N) d_out[(long long)bh * N + t] = draw / zsum;     // D_part
                dinv_ring[(u & 7) * 64 + rr] = draw > 0.f ? 1.f / draw : 0.f;
                fence_proxy_async();
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(f_free + (nx & 1));
            __syncwarp();
            if (lane == 0) mbar_arrive(pq_full + slot);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ------------------------------------------------------------------------------------------ host side

template <int D, int DF, typename TOut>
int launch_npmap(const void *X, const void *W, const void *bias, void *phi, float *csum, int B, int heads, long long N,
                 int C, int *status, cudaStream_t st, int *launches) {
    CUtensorMap tx, tw;
    if (!make_map_2d(&tx, X, (unsigned long long)B * heads * N, D, 128, false) ||
        !make_map_2d(&tw, W, (unsigned long long)heads * D, DF, D, false))
        return STILL_ERR_CUDA;
    constexpr int kSmem = NpmapSmem<D, DF, TOut>::kTotal;
    if (ensure_dynamic_smem((const void *)npmap_tc_kernel<D, DF, TOut>, kSmem) != cudaSuccess) return STILL_ERR_CUDA;
    dim3 grid((unsigned)((N + 127) / 128), (unsigned)heads, (unsigned)B);
    ++*launches;
    return launch_dependent(npmap_tc_kernel<D, DF, TOut>, grid, dim3(192), kSmem, st, tx, tw, (const __nv_bfloat16 *)bias, (TOut *)phi,
                            csum, status, heads, (int)N, C) == cudaSuccess ? STILL_OK : STILL_ERR_CUDA;
}

template <int D, int DF>
int launch_gather(const still_params_t *p, long long N, const void *K, const void *V, const void *phiK, const int32_t *sel_idx,
                  void *k_sel, void *v_sel, void *phiK_sel, float *selsum, long long sel_rows, int n_routed, const StateParts *state,
                  cudaStream_t st, int *launches) {
    using bf = __nv_bfloat16;
    const long long Tn = (N + p->chunk - 1) / p->chunk;
    ++*launches;
    const long long BH = (long long)p->B * p->H, rows = state != nullptr ? (state->blocks + Tn) / (Tn + 1) : 0;
    const bool few = D == 64 && p->topk <= 16;
    return launch_dependent(state != nullptr ? gather_kernel<D, DF, false, true> : few ? gather_kernel<D, DF, D == 64, false> : gather_kernel<D, DF, false, false>,
                            dim3((unsigned)(Tn + 1), (unsigned)(BH + rows)), dim3(256), 0, st, (const bf *)K, (const bf *)V,
                            (const bf *)phiK, sel_idx, (bf *)k_sel, (bf *)v_sel, (bf *)phiK_sel, selsum, p->H, p->Hkv, N, p->topk, sel_rows,
                            n_routed, (int)BH, state != nullptr ? *state : StateParts{}, *p) == cudaSuccess ? STILL_OK : STILL_ERR_CUDA;
}

// Whether every segment of the scan folds the chunks before it itself, rather than starting from a pass of sums: up to a
// number of update tiles before the last segment, 64 where the pass has more CTAs than SMs; fewer where they run at once,
// its time then being that of one piece.  (Gain of folding in % of a call, C = 64, a quarter kept.  One wave, d = 64: 1 to 4
// heads 16 tiles 4 to 8, 24 2 to 4, 48 -5 to -6, 72 -11 to -13, 96 -18; d = 128: 16 10 to 11, 24 5 to 6, 48 1 to 3, 72 -5 to -8,
// 96 -12 to -15; C = 128: 32 tiles 1 to 5, 48 -4 to 2.  Two waves, 8 heads: 48 tiles 1 at d = 64, 7 at 128, 72 -6 and -1, 96 -12
// and -6; 32 heads: 16 tiles 15 and 17, 32 9 and 11, 64 2 and 3, 96 -1 and 0, 128 -3 and -2.  Three, 16 heads: 48 tiles 8 and 17,
// 72 1 and 9, 96 -3 and 3, 144 -8 and -5.)
bool fold_again(const still_params_t *p, int n_seg, int seg_chunks, int parts, int tiles_per_chunk) {
    const long long pass_ctas = 2ll * p->B * p->H * (n_seg - 1) * parts, tiles = (long long)(n_seg - 1) * seg_chunks * tiles_per_chunk;
    return n_seg > 1 && tiles <= (pass_ctas > kSms ? 64 : p->d == 64 ? 40 : 48);
}

template <int D, int DF>
int launch_fused(const still_params_t *p, long long N, const void *Q, const void *V, const void *G, const void *Wq,
                 const void *bq, const int32_t *sel_idx, const void *phiK, const float *zpre, void *y_part, float *d_part,
                 float *S_out, float *seg_sums, void *phiK_sel, void *v_sel, long long sel_rows, int *status, cudaStream_t st,
                 int *launches) {
    using bf = __nv_bfloat16;
    CUtensorMap tq, tw, tk, tv, tks, tvs, ty0, ty1;
    const unsigned long long BH = (unsigned long long)p->B * p->H, BHkv = (unsigned long long)p->B * p->Hkv;
    if (!make_map_2d(&tq, Q, BH * N, D, 128, false) || !make_map_2d(&tw, Wq, (unsigned long long)p->H * D, DF, D, false) ||
        !make_map_2d(&tk, phiK, BHkv * N, 2 * DF, FusedPlan<D, DF>::kUTok, false) ||
        !make_map_2d(&tv, V, BHkv * N, D, FusedPlan<D, DF>::kUTok, false) || !make_map_2d(&ty0, y_part, BH * N, D, 64, false) ||
        !make_map_2d(&ty1, (bf *)y_part + BH * N * D, BH * N, D, 64, false))
        return STILL_ERR_CUDA;
    // With a salient-cache budget and topk < chunk the leaving tokens are read from gathered copies of their rows
    // (otherwise every token of a chunk is selected and the chunk's own tiles are the leaving tiles).
    const bool gathered = p->max_salient > 0 && p->topk < p->chunk && phiK_sel != nullptr && v_sel != nullptr;
    tks = tk;
    tvs = tv;
    if (gathered) {
        if (BH * (unsigned long long)sel_rows >= (1ull << 31)) return STILL_ERR_UNSUPPORTED;   // TMA row coordinate
        if (!make_map_2d(&tks, phiK_sel, BH * (unsigned long long)sel_rows, 2 * DF, FusedPlan<D, DF>::kUTok, false) ||
            !make_map_2d(&tvs, v_sel, BH * (unsigned long long)sel_rows, D, FusedPlan<D, DF>::kUTok, false))
            return STILL_ERR_CUDA;
    }
    using Plan = FusedPlan<D, DF>;
    int seg_chunks = 0;
    const int n_seg = tc_la_segments(p, N, &seg_chunks), parts = tc_la_sum_parts(seg_chunks);
    // (tiles of a chunk, and of the tokens that leave a capped cache with it: see the kernel)
    const int su = p->chunk / Plan::kUTok, nl = gathered ? (p->topk + Plan::kUTok - 1) / Plan::kUTok : su;
    const bool again = fold_again(p, n_seg, seg_chunks, parts, p->max_salient > 0 ? su + nl : su);
    const auto kernel = again ? la_fused_kernel<D, DF, true> : la_fused_kernel<D, DF, false>;
    if (ensure_dynamic_smem((const void *)kernel, Plan::kTotal) != cudaSuccess) return STILL_ERR_CUDA;
    for (int pass = n_seg > 1 && !again ? 0 : 1; pass < 2; ++pass) {
        // pass 0 (only with several segments): the sum of every segment's own updates; pass 1: the scan proper
        dim3 grid((unsigned)BH, 2, (unsigned)(pass == 0 ? (n_seg - 1) * parts : n_seg));   // head, feature half, segment (piece)
        const cudaError_t e = launch_dependent(kernel, grid, dim3(384), Plan::kTotal, st, tq, tw, tk, tv, tks, tvs, ty0, ty1, (const bf *)bq, (const bf *)G, sel_idx, zpre,
                                                               (bf *)y_part, d_part, S_out, seg_sums, status, p->H, p->Hkv, (int)N,
                                                               p->chunk, p->topk, p->topk > 0 ? (int)(p->max_salient / p->topk) : 0,
                                                               (long long)BH * N * D, (long long)BH * N,
                                                               seg_chunks, n_seg, parts, pass == 0 ? 1 : 0, gathered ? (int)sel_rows : 0);
        if (e != cudaSuccess) return STILL_ERR_CUDA;
        ++*launches;
    }
    return STILL_OK;
}

}  // namespace

bool tc_la_supported(const still_params_t *p) {
    return tc_supported(p) && (p->d_f == 64 || p->d_f == 128) && p->d_f <= p->d;
}

// Two-level scan: with few (batch, head) units the sequence is cut into segments that run side by side, each
// starting from the sum of the earlier segments' state updates.  Segments are whole, even numbers of chunks, at
// least eight of them, and as many as fill the SMs once (two CTAs per head and segment).
int tc_la_segments(const still_params_t *p, long long N, int *seg_chunks) {
    const long long Tn = (N + p->chunk - 1) / p->chunk, ctas = 2ll * p->B * p->H;
    int n_seg = 1;
    while (n_seg < 4 && ctas * (n_seg * 2) <= kSms && Tn / (n_seg * 2) >= 8) n_seg *= 2;
    long long sc = (Tn + n_seg - 1) / n_seg;
    sc += sc & 1;
    if (seg_chunks) *seg_chunks = (int)sc;
    return n_seg;
}

// Pieces per segment in the first pass of the two-level scan (each at least two chunks long).
int tc_la_sum_parts(int seg_chunks) {
    return (seg_chunks % 4 == 0 && seg_chunks >= 8) ? 4 : (seg_chunks % 2 == 0 && seg_chunks >= 4) ? 2 : 1;
}

int tc_la_branch(const still_params_t *p, long long N, const void *Q, const void *K, const void *V, const void *G,
                 const void *Wq, const void *bq, const void *Wk, const void *bk, const int32_t *sel_idx, void *phiK,
                 float *csum, float *zpre, void *y_part, float *d_part, float *seg_sums, float *S_out, float *z_out,
                 void *phiK_sel, void *k_sel, void *v_sel, long long sel_rows, const StateParts *state_parts, bool *state_written,
                 int *status_words, cudaStream_t st, int *launches) {
    using bf = __nv_bfloat16;
    if ((long long)p->B * p->H * N >= (1ll << 31)) return STILL_ERR_UNSUPPORTED;  // TMA row coordinate
    const int NF = 2 * p->d_f, C = p->chunk;
    const long long Tn = (N + C - 1) / C, BH = (long long)p->B * p->H;
    const int n_routed = Tn >= 3 ? (int)(Tn - 2) : 0;
    // phi(K) once per KV head (bf16; the B operand of the state update), with the column sums of every chunk
    int rc;
    if (p->d == 64 && p->d_f == 64)
        rc = launch_npmap<64, 64, bf>(K, Wk, bk, phiK, csum, p->B, p->Hkv, N, C, status_words, st, launches);
    else if (p->d == 128 && p->d_f == 64)
        rc = launch_npmap<128, 64, bf>(K, Wk, bk, phiK, csum, p->B, p->Hkv, N, C, status_words, st, launches);
    else
        rc = launch_npmap<128, 128, bf>(K, Wk, bk, phiK, csum, p->B, p->Hkv, N, C, status_words, st, launches);
    if (rc != STILL_OK) return rc;
    // selected rows of K, V (and phi(K)), then z after every routed chunk (per query head: the selection is per query
    // head).  The sums of the selected rows lie where the branch's output will: the scan has taken them by then.
    float *selsum = reinterpret_cast<float *>(y_part);
    const int window = p->topk > 0 ? (int)(p->max_salient / p->topk) : 0;
    if (p->topk < C) {
        // The decode state rides along up to 512 blocks, where a launch is longer than what it does.  (32 heads, d = 128, gated, 1003
        // tokens, 350 blocks: 82.9 us a call with a launch of its own, 80.7 like this; 4000 tokens, 1250 blocks: 215 and 224, the rows'
        // copies stand in the gather's way.)
        if (state_parts != nullptr && (state_parts->blocks > 512 || BH > 32768)) state_parts = nullptr;   // (BH: rows of a grid)
        if (p->d == 64 && p->d_f == 64)
            rc = launch_gather<64, 64>(p, N, K, V, phiK, sel_idx, k_sel, v_sel, phiK_sel, selsum, sel_rows, n_routed, state_parts, st, launches);
        else if (p->d == 128 && p->d_f == 64)
            rc = launch_gather<128, 64>(p, N, K, V, phiK, sel_idx, k_sel, v_sel, phiK_sel, selsum, sel_rows, n_routed, state_parts, st, launches);
        else
            rc = launch_gather<128, 128>(p, N, K, V, phiK, sel_idx, k_sel, v_sel, phiK_sel, selsum, sel_rows, n_routed, state_parts, st, launches);
        if (rc != STILL_OK) return rc;
        *state_written = state_parts != nullptr;
    }
    if (n_routed > 0 || z_out != nullptr) {
        // a warp per eight chunks, whose loads are in flight together; at most 32
        const int warps = std::max(1, std::min(32, (n_routed + 7) / 8));
        if (launch_dependent(z_scan_kernel, dim3((unsigned)BH, NF / 32), dim3(32 * warps), 0, st, csum, selsum, zpre, z_out, p->H, p->Hkv,
                             (int)Tn, n_routed, p->topk >= C ? 1 : 0, window, NF) != cudaSuccess)
            return STILL_ERR_CUDA;
        ++*launches;
    }
    if (p->d == 64 && p->d_f == 64)
        return launch_fused<64, 64>(p, N, Q, V, G, Wq, bq, sel_idx, phiK, zpre, y_part, d_part, S_out, seg_sums, phiK_sel, v_sel, sel_rows,
                                   status_words, st, launches);
    if (p->d == 128 && p->d_f == 64)
        return launch_fused<128, 64>(p, N, Q, V, G, Wq, bq, sel_idx, phiK, zpre, y_part, d_part, S_out, seg_sums, phiK_sel, v_sel, sel_rows,
                                   status_words, st, launches);
    return launch_fused<128, 128>(p, N, Q, V, G, Wq, bq, sel_idx, phiK, zpre, y_part, d_part, S_out, seg_sums, phiK_sel, v_sel, sel_rows,
                                   status_words, st, launches);
}

}  // namespace still
