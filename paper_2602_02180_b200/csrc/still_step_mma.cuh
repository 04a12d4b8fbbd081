// Split-KV pass of the decode step for bf16 (Sec. 3.3: N_SA, D_SA over the salient cache h_t).
//
// HBM-bound: every step reads the K and V history once, for all query heads of a KV group together.  The history of
// a group is cut into tiles of 16 positions; a warp takes every eighth tile of its block's range through a ring of
// 16-byte cp.async stages (no padding: the 16-byte pieces of a row are XOR-swizzled by the row, so that the copies and
// the ldmatrix reads are free of bank conflicts).  Keys are the rows of the tensor-core tiles and the group's query
// heads their columns -- S^T = K Q^T, then O^T += V^T P^T -- because a group has at most 16 heads and usually four:
// as rows of an m16n8k16 they would fill a quarter of the tile, as columns they fill half.  P^T changes from an
// accumulator to an operand fragment by one movmatrix per eight keys, without shared memory.
//
// Which rows a query head sees is a per-head membership mask: for a position in a routed chunk, whether the head's
// selection (the sel_mask words of the decode state) contains it; for the two-chunk local region, every position up
// to the new token.  A row is read from memory only if some head of the group selected it; with topk = chunk that is
// every row.  A tile without a new maximum (most of them, past the first few) costs one vote instead of a reduction and
// a rescaling of O.
//
// The weights P enter the second product as two bf16 parts, the upper 8 bits of the significand and the rest: rounded
// to bf16 once they would be the largest error of a step, and one that depends on how the history is cut (a weight is
// exact where it is its partial's maximum): relative error of y against 64 bits 1.84e-3 to 2.25e-3, with both parts
// 1.66e-3, which is y's own rounding.  A group of up to four heads takes no further product for it: the four columns
// that it leaves idle carry the second part (16 x 16000 tokens, a quarter kept: 148 us a step, rounded once 145.5).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace still {

__device__ __forceinline__ void cp_async16(void *dst_smem, const void *src, bool valid) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst_smem));
    const int bytes = valid ? 16 : 0;  // 0 source bytes: the 16 destination bytes are zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory"); }

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], const void *p) {
    const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p));
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], const void *p) {
    const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p));
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
// D (16x8, fp32) += A (16x16, bf16, row) * B (16x8, bf16, col)
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Transpose of an 8x8 matrix of 16-bit elements held one row per four lanes.
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
    uint32_t r;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(a));
    return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack2_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// Two weights (>= 0) as bf16 parts: their upper halves, and what these leave off.  The rest of a weight that is not
// zero is never zero, so that an infinite value stays infinite under both parts.
__device__ __forceinline__ uint32_t weight_hi2(float a, float b) { return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632); }
__device__ __forceinline__ uint32_t weight_lo2(float a, float b) {
    const float ra = a - __uint_as_float(__float_as_uint(a) & 0xffff0000u), rb = b - __uint_as_float(__float_as_uint(b) & 0xffff0000u);
    return pack2_bf16(fmaxf(ra, a * 0x1p-24f), fmaxf(rb, b * 0x1p-24f));
}

// Geometry of a decode step's cache pass (see step_main_kernel).
struct AttendView {
    long long kvr;       // ring rows per KV head
    int first_pos, t;    // first position read, position of the new token
    int loc0;            // first position of the local region
    int C, lam, rep, n_chunk_cap;
    float scale, scale_log2;
    int early_k;         // request K rows before it is known which of them are needed (see load_tile)
};

constexpr int kStepWarps = 8;
constexpr int kTileKeys = 16;

template <int D>
struct AttendPlan {
    static constexpr int kRow = D * 2;                     // bytes of a row
    static constexpr int kPieces = D / 8;                  // 16-byte pieces of a row
    static constexpr int kTile = kTileKeys * kRow;         // K or V rows of a tile
    static constexpr int kStage = 2 * kTile;
    static constexpr int kStages = D == 128 ? 3 : 4;       // per warp: 24 KB / 16 KB, 196 KB / 131 KB a block
    static constexpr int kWarp = kStages * kStage;
    static constexpr int kTotal = kStepWarps * kWarp;
};

// The barrier of the eight warps of the cache pass; kOthers: the block has other warps too.
template <bool kOthers>
__device__ __forceinline__ void step_sync() {
    if constexpr (kOthers) asm volatile("bar.sync 0, %0;" ::"n"(kStepWarps * 32) : "memory");
    else __syncthreads();
}

// Tiles [tile_lo, tile_hi) of one KV head by 8 warps.  kh, vh: the head's rows; k_new, v_new: the new
// token's (position t is read from the call's inputs, not from the row that another block is writing); qh: the
// group's queries; mask: sel_mask of the group's first head.  Leaves one record per head (maximum in natural-log
// units, sum, numerator [D]) at part + head * part_stride, and the new token's logits against the last C positions,
// oldest first, at logits + head * part_stride.  NH: room for heads, 4, 8 or 16 (tiles of 8 columns; with 4 the second
// half of the tile repeats the heads and takes the second part of their weights).  The warps' sums are merged through
// `staging`: the rings, or (kBeside) a place of its own, so that what after() requests into the rings is on its way meanwhile.
template <int D, int NH, bool kOthers, bool kBeside, class After>
__device__ __forceinline__ void attend_segment(const AttendView &v, const __nv_bfloat16 *kh, const __nv_bfloat16 *vh,
                                               const __nv_bfloat16 *k_new, const __nv_bfloat16 *v_new,
                                               const __nv_bfloat16 *qh, const uint32_t *mask, int tile_lo, int tile_hi,
                                               uint8_t *smem, float *staging, float *part, float *logits, long long part_stride,
                                               After after) {
    using P = AttendPlan<D>;
    constexpr int NT = NH == 16 ? 2 : 1;
    constexpr bool kRepeat = NH == 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tig = lane & 3;
    uint8_t *my = smem + warp * P::kWarp;
    auto head_of = [](int column) { return kRepeat ? column & 3 : column; };

    // Q^T as B fragments: columns are heads (head >= rep: zero)
    uint32_t qb[NT][D / 16][2];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
            const int h = head_of(nt * 8 + g), col = ks * 16 + tig * 2;
            qb[nt][ks][0] = h < v.rep ? *reinterpret_cast<const uint32_t *>(qh + h * D + col) : 0u;
            qb[nt][ks][1] = h < v.rep ? *reinterpret_cast<const uint32_t *>(qh + h * D + col + 8) : 0u;
        }
    float o[NT][D / 16][4];
    float m_run[NT][2], l_run[NT][2];   // of heads 8 nt + 2 tig and + 1, log2 domain; l: this thread's keys only
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
        for (int i = 0; i < D / 16; ++i) o[nt][i][0] = o[nt][i][1] = o[nt][i][2] = o[nt][i][3] = 0.f;
        m_run[nt][0] = m_run[nt][1] = -INFINITY;
        l_run[nt][0] = l_run[nt][1] = 0.f;
    }

    // Membership of tile j's 16 positions (bits 0-15) for the head in this lane (lanes >= group size: 0).
    auto member_word = [&](int j) -> uint32_t {
        if (j >= tile_hi || lane >= v.rep) return 0u;
        const int p0 = v.first_pos + j * kTileKeys;
        if (p0 >= v.loc0) {
            const int last = v.t - p0;   // positions up to the new token
            return last >= 15 ? 0xffffu : ((1u << (last + 1)) - 1u);
        }
        if (v.lam >= v.C) return 0xffffu;
        // (chunk sizes are multiples of 32: words run on from chunk to chunk)
        return mask[(long long)lane * v.n_chunk_cap * (v.C / 32) + (p0 >> 5)] >> (p0 & 16) & 0xffffu;
    };
    const int c_piece = lane % P::kPieces, c_row = lane / P::kPieces;   // this lane's piece and first row of a copy
    constexpr int kRowsPerIt = 32 / P::kPieces;
    // With few sequences a step is a chain of latencies: K is then read without waiting for the membership words (all rows
    // up to the new token; a masked logit is never used), V as soon as they are there.  (One user, 2000 tokens: 10.5 us a
    // step, waiting 10.6; at 2 to 4 sequences waiting is 0.1 to 0.5 us faster, from 6 on 0.2 to 0.6.)
    auto load_tile = [&](int j, int stage, uint32_t rows, bool with_k, bool with_v) {
        uint8_t *ks = my + stage * P::kStage, *vs = ks + P::kTile;
        const int p0 = v.first_pos + j * kTileKeys;
        // position p lives in ring row p % kvr; kvr is a multiple of the chunk size, so a tile never straddles the end
        const long long r0 = (uint32_t)p0 % (uint32_t)v.kvr;
        const __nv_bfloat16 *kp = kh + (r0 + c_row) * D + c_piece * 8, *vp = vh + (r0 + c_row) * D + c_piece * 8;
        const int t_row = v.t - p0;   // row of the new token if it lies in this tile
#pragma unroll
        for (int it = 0; it < kTileKeys / kRowsPerIt; ++it) {
            const int row = it * kRowsPerIt + c_row;
            const int dst = row * P::kRow + ((c_piece ^ (row & 7)) << 4);
            const bool valid = (rows >> row) & 1u;
            const bool is_new = row == t_row;
            if (with_k) cp_async16(ks + dst, is_new ? k_new + c_piece * 8 : kp + it * kRowsPerIt * D, valid);
            if (with_v) cp_async16(vs + dst, is_new ? v_new + c_piece * 8 : vp + it * kRowsPerIt * D, valid);
        }
    };
    auto rows_so_far = [&](int j) -> uint32_t {   // rows of tile j up to the new token
        const int last = v.t - (v.first_pos + j * kTileKeys);
        return last >= 15 ? 0xffffu : ((1u << (last + 1)) - 1u);
    };

    // ring: kStages - 1 tiles in flight; membership words run one tile ahead of the copies they steer
    constexpr int kAhead = P::kStages - 1;
    uint32_t words[kAhead + 1];   // words[i]: tile (current + i) of this warp
    const int first = tile_lo + warp;
#pragma unroll
    for (int i = 0; i <= kAhead; ++i) words[i] = member_word(first + kStepWarps * i);
    if (v.early_k) {
#pragma unroll
        for (int i = 0; i < kAhead; ++i)
            if (first + kStepWarps * i < tile_hi) load_tile(first + kStepWarps * i, i, rows_so_far(first + kStepWarps * i), true, false);
    }
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
        if (first + kStepWarps * i < tile_hi)
            load_tile(first + kStepWarps * i, i, __reduce_or_sync(0xffffffffu, words[i]), !v.early_k, true);
        cp_async_commit();
    }
    int stage = 0;
    for (int j = first; j < tile_hi; j += kStepWarps) {
        const uint32_t after = member_word(j + kStepWarps * (kAhead + 1));
        {
            int ps = stage + kAhead;
            if (ps >= P::kStages) ps -= P::kStages;
            const int jn = j + kStepWarps * kAhead;
            if (jn < tile_hi) load_tile(jn, ps, __reduce_or_sync(0xffffffffu, words[kAhead]), true, true);
            cp_async_commit();
        }
        const uint32_t word = words[0];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) words[i] = words[i + 1];
        words[kAhead] = after;
        cp_async_wait<kAhead>();
        __syncwarp();
        const uint8_t *ks = my + stage * P::kStage, *vs = ks + P::kTile;

        // S^T = K Q^T: rows are keys g and g + 8, columns heads 2 tig and 2 tig + 1.  Two chains of products, of even and
        // odd k-steps: half the latency, and fewer roundings in a row.
        float s[NT][4], s_odd[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[nt][e] = s_odd[nt][e] = 0.f;
#pragma unroll
        for (int k16 = 0; k16 < D / 16; ++k16) {
            uint32_t a[4];
            const int row = ((lane >> 3) & 1) * 8 + (lane & 7), piece = k16 * 2 + (lane >> 4);
            ldmatrix_x4(a, ks + row * P::kRow + ((piece ^ (row & 7)) << 4));
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) mma_16816(k16 & 1 ? s_odd[nt] : s[nt], a, qb[nt][k16][0], qb[nt][k16][1]);
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[nt][e] += s_odd[nt][e];
        const int slot0 = v.first_pos + j * kTileKeys - (v.t - (v.C - 1));   // slot of the tile's first key in the window
        if (slot0 > -kTileKeys) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int h = nt * 8 + tig * 2 + (e & 1), sl = slot0 + g + (e >> 1) * 8;
                    if (h < v.rep && sl >= 0 && sl < v.C) logits[h * part_stride + sl] = s[nt][e] * v.scale;
                }
        }
        bool grow = false;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const uint32_t vis = __shfl_sync(0xffffffffu, word, head_of(nt * 8 + tig * 2 + hh));
                s[nt][hh] = (vis >> g) & 1u ? s[nt][hh] * v.scale_log2 : -INFINITY;
                s[nt][2 + hh] = (vis >> (g + 8)) & 1u ? s[nt][2 + hh] * v.scale_log2 : -INFINITY;
                grow |= !(max_nan(s[nt][hh], s[nt][2 + hh]) <= m_run[nt][hh]);
            }
        }
        if (__any_sync(0xffffffffu, grow)) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                float alpha[2];
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    float mx = max_nan(s[nt][hh], s[nt][2 + hh]);
                    mx = max_nan(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
                    mx = max_nan(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
                    mx = max_nan(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
                    const float mn = max_nan(m_run[nt][hh], mx);
                    alpha[hh] = (mn == -INFINITY) ? 1.f : ex2_approx(m_run[nt][hh] - mn);
                    m_run[nt][hh] = mn;
                    l_run[nt][hh] *= alpha[hh];
                }
#pragma unroll
                for (int i = 0; i < D / 16; ++i) {
                    o[nt][i][0] *= alpha[0];
                    o[nt][i][1] *= alpha[1];
                    o[nt][i][2] *= alpha[0];
                    o[nt][i][3] *= alpha[1];
                }
            }
        }
        uint32_t pb[NT][2], pr[NT][2];   // P^T as B fragments: first part (repeated heads: the column's part), second part
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            float pv[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float m = m_run[nt][e & 1];
                pv[e] = (m == -INFINITY) ? 0.f : ex2_approx(s[nt][e] - m);
            }
            l_run[nt][0] += pv[0] + pv[2];
            l_run[nt][1] += pv[1] + pv[3];
            const uint32_t h0 = weight_hi2(pv[0], pv[1]), h1 = weight_hi2(pv[2], pv[3]);
            const uint32_t l0 = weight_lo2(pv[0], pv[1]), l1 = weight_lo2(pv[2], pv[3]);
            pb[nt][0] = movmatrix_trans(kRepeat && tig >= 2 ? l0 : h0);
            pb[nt][1] = movmatrix_trans(kRepeat && tig >= 2 ? l1 : h1);
            if constexpr (!kRepeat) {
                pr[nt][0] = movmatrix_trans(l0);
                pr[nt][1] = movmatrix_trans(l1);
            }
        }
        // O^T += V^T P^T: rows are value columns
#pragma unroll
        for (int dt = 0; dt < D / 16; ++dt) {
            uint32_t a[4];
            const int row = (lane >> 4) * 8 + (lane & 7), piece = dt * 2 + ((lane >> 3) & 1);
            ldmatrix_x4_trans(a, vs + row * P::kRow + ((piece ^ (row & 7)) << 4));
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                mma_16816(o[nt][dt], a, pb[nt][0], pb[nt][1]);
                if constexpr (!kRepeat) mma_16816(o[nt][dt], a, pr[nt][0], pr[nt][1]);
            }
        }
        __syncwarp();   // the stage may be overwritten
        if (++stage == P::kStages) stage = 0;
    }
    if constexpr (kBeside) {
        after();
    } else {
        cp_async_wait<0>();
        step_sync<kOthers>();
    }

    // merge the eight warps: [8 warps][rep][D + 2] in shared memory
    float *mg = staging;
    constexpr int kStride = D + 2;
    const int rep = v.rep;
    if constexpr (kRepeat) {   // both parts of a head's sums
#pragma unroll
        for (int dt = 0; dt < D / 16; ++dt)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[0][dt][e] += __shfl_xor_sync(0xffffffffu, o[0][dt][e], 2);
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int h = nt * 8 + tig * 2 + hh;
            float l = l_run[nt][hh];
            l += __shfl_xor_sync(0xffffffffu, l, 4);
            l += __shfl_xor_sync(0xffffffffu, l, 8);
            l += __shfl_xor_sync(0xffffffffu, l, 16);
            if (h < rep) {
                float *dst = mg + (warp * rep + h) * kStride;
                if (g == 0) {
                    dst[0] = m_run[nt][hh];
                    dst[1] = l;
                }
#pragma unroll
                for (int dt = 0; dt < D / 16; ++dt) {
                    dst[2 + dt * 16 + g] = o[nt][dt][hh];
                    dst[2 + dt * 16 + g + 8] = o[nt][dt][2 + hh];
                }
            }
        }
    }
    step_sync<kOthers>();
    for (int idx = threadIdx.x; idx < rep * kStride; idx += kStepWarps * 32) {
        const int h = idx / kStride, col = idx % kStride;
        float mw[kStepWarps], M = -INFINITY;
#pragma unroll
        for (int w = 0; w < kStepWarps; ++w) {
            mw[w] = mg[(w * rep + h) * kStride];
            M = max_nan(M, mw[w]);
        }
        float acc = 0.f;
        if (col == 0) {
            acc = M * 0.6931471805599453f;   // the merge kernel works in natural-log units
        } else {
#pragma unroll
            for (int w = 0; w < kStepWarps; ++w)
                if (mw[w] != -INFINITY) acc += ex2_approx(mw[w] - M) * mg[(w * rep + h) * kStride + col];
        }
        part[h * part_stride + col] = acc;
    }
    step_sync<kOthers>();   // the staging space is the next segment's
}

}  // namespace still
