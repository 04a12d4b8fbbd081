// Split-KV pass of the decode step for fp32 states: the structure of still_step_mma.cuh (tiles of the history through
// a per-warp cp.async ring, one read of a K / V row for up to four query heads) with fp32 arithmetic throughout.
// A tile is 8 positions, so that a lane owns one (position, head) pair of the logits and its dot product runs over
// shared memory: the K row's 16-byte pieces are swizzled (8 rows, 8 bank groups) and the query is a broadcast.  For
// P V a lane owns D / 32 value columns of all four heads and the probabilities come by shuffle.
// Groups of more than four query heads are cut into units of four.
#pragma once
#include "still_step_mma.cuh"

namespace still {

constexpr int kTileKeysF32 = 8;
constexpr int kUnitHeadsF32 = 4;

template <int D>
struct AttendPlanF32 {
    static constexpr int kRow = D * 4;
    static constexpr int kPieces = D / 4;
    static constexpr int kTile = kTileKeysF32 * kRow;
    static constexpr int kStage = 2 * kTile;
    static constexpr int kStages = D == 128 ? 3 : 4;
    static constexpr int kWarp = kStages * kStage;
    static constexpr int kQ = kStepWarps * kWarp;                       // the unit's queries [4][D]
    static constexpr int kTotal = kQ + kUnitHeadsF32 * kRow;
};

// Arguments as attend_segment; v.rep is the unit's number of heads (at most four).
template <int D>
__device__ __forceinline__ void attend_segment_f32(const AttendView &v, const float *kh, const float *vh, const float *k_new,
                                                   const float *v_new, const float *qh, const uint32_t *mask, int tile_lo,
                                                   int tile_hi, uint8_t *smem, float *part, float *logits, long long part_stride) {
    using P = AttendPlanF32<D>;
    constexpr int NH = kUnitHeadsF32, kKeys = kTileKeysF32, DPL = D / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t *my = smem + warp * P::kWarp;
    float *qs = reinterpret_cast<float *>(smem + P::kQ);
    for (int i = threadIdx.x; i < NH * D; i += kStepWarps * 32) qs[i] = i < v.rep * D ? qh[i] : 0.f;
    __syncthreads();

    const int key = lane & 7, hd = lane >> 3;
    float o[NH][DPL];
#pragma unroll
    for (int h = 0; h < NH; ++h)
#pragma unroll
        for (int x = 0; x < DPL; ++x) o[h][x] = 0.f;
    float m_run = -INFINITY, l_run = 0.f;   // of head hd; l: this lane's positions only

    auto member_word = [&](int j) -> uint32_t {   // bits 0-7, for the head in this lane
        if (j >= tile_hi || lane >= v.rep) return 0u;
        const int p0 = v.first_pos + j * kKeys;
        if (p0 >= v.loc0) {
            const int last = v.t - p0;
            return last >= 7 ? 0xffu : ((1u << (last + 1)) - 1u);
        }
        if (v.lam >= v.C) return 0xffu;
        return mask[(long long)lane * v.n_chunk_cap * (v.C / 32) + (p0 >> 5)] >> (p0 & 24) & 0xffu;
    };
    auto load_tile = [&](int j, int stage, uint32_t rows) {
        uint8_t *ks = my + stage * P::kStage, *vs = ks + P::kTile;
        const int p0 = v.first_pos + j * kKeys, t_row = v.t - p0;
        const long long r0 = (uint32_t)p0 % (uint32_t)v.kvr;
#pragma unroll
        for (int i = lane; i < kKeys * P::kPieces; i += 32) {
            const int row = i / P::kPieces, piece = i % P::kPieces;
            const int dst = row * P::kRow + ((piece ^ (row & 7)) << 4);
            const bool valid = (rows >> row) & 1u, is_new = row == t_row;
            cp_async16(ks + dst, is_new ? k_new + piece * 4 : kh + (r0 + row) * D + piece * 4, valid);
            cp_async16(vs + dst, is_new ? v_new + piece * 4 : vh + (r0 + row) * D + piece * 4, valid);
        }
    };
    constexpr int kAhead = P::kStages - 1;
    uint32_t words[kAhead + 1];
    const int first = tile_lo + warp;
#pragma unroll
    for (int i = 0; i <= kAhead; ++i) words[i] = member_word(first + kStepWarps * i);
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
        if (first + kStepWarps * i < tile_hi) load_tile(first + kStepWarps * i, i, __reduce_or_sync(0xffffffffu, words[i]));
        cp_async_commit();
    }
    int stage = 0;
    for (int j = first; j < tile_hi; j += kStepWarps) {
        const uint32_t after = member_word(j + kStepWarps * (kAhead + 1));
        {
            int ps = stage + kAhead;
            if (ps >= P::kStages) ps -= P::kStages;
            const int jn = j + kStepWarps * kAhead;
            if (jn < tile_hi) load_tile(jn, ps, __reduce_or_sync(0xffffffffu, words[kAhead]));
            cp_async_commit();
        }
        const uint32_t word = words[0];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) words[i] = words[i + 1];
        words[kAhead] = after;
        cp_async_wait<kAhead>();
        __syncwarp();
        const uint8_t *ks = my + stage * P::kStage;
        const float *vs = reinterpret_cast<const float *>(ks + P::kTile);

        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll 8
        for (int piece = 0; piece < P::kPieces; ++piece) {
            const float4 kk = *reinterpret_cast<const float4 *>(ks + key * P::kRow + ((piece ^ key) << 4));
            const float4 qq = *reinterpret_cast<const float4 *>(qs + hd * D + piece * 4);
            a0 = fmaf(qq.x, kk.x, a0);
            a1 = fmaf(qq.y, kk.y, a1);
            a2 = fmaf(qq.z, kk.z, a2);
            a3 = fmaf(qq.w, kk.w, a3);
        }
        const uint32_t vis = __shfl_sync(0xffffffffu, word, hd);
        const bool on = (vis >> key) & 1u;
        const float dot = ((a0 + a1) + (a2 + a3)) * v.scale;
        const float s = on ? dot : -INFINITY;
        const int slot = v.first_pos + j * kKeys + key - (v.t - (v.C - 1));   // of this lane's key in the new token's window
        if (slot >= 0 && slot < v.C && hd < v.rep) logits[hd * part_stride + slot] = dot;
        float mx = s;
        mx = max_nan(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = max_nan(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        mx = max_nan(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
        const float mn = max_nan(m_run, mx);
        const float alpha = (mn == -INFINITY) ? 1.f : expf(m_run - mn);
        const float p = (on && mn != -INFINITY) ? expf(s - mn) : 0.f;
        m_run = mn;
        l_run = l_run * alpha + p;
        if (__any_sync(0xffffffffu, alpha != 1.f)) {
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                const float ah = __shfl_sync(0xffffffffu, alpha, h * 8);
#pragma unroll
                for (int x = 0; x < DPL; ++x) o[h][x] *= ah;
            }
        }
#pragma unroll
        for (int jj = 0; jj < kKeys; ++jj) {
            float vv[DPL];
            if constexpr (DPL == 4) {
                const float4 f = *reinterpret_cast<const float4 *>(vs + jj * D + ((lane ^ jj) << 2));
                vv[0] = f.x; vv[1] = f.y; vv[2] = f.z; vv[3] = f.w;
            } else {
                const float2 f = *reinterpret_cast<const float2 *>(vs + jj * D + (((lane >> 1) ^ jj) << 2) + (lane & 1) * 2);
                vv[0] = f.x; vv[1] = f.y;
            }
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                const float ph = __shfl_sync(0xffffffffu, p, h * 8 + jj);
#pragma unroll
                for (int x = 0; x < DPL; ++x) o[h][x] = fmaf(ph, vv[x], o[h][x]);
            }
        }
        __syncwarp();
        if (++stage == P::kStages) stage = 0;
    }
    cp_async_wait<0>();
    __syncthreads();

    float *mg = reinterpret_cast<float *>(smem);   // [8 warps][4][D + 2]
    constexpr int kStride = D + 2;
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 4);
    if (key == 0) {
        mg[(warp * NH + hd) * kStride] = m_run;
        mg[(warp * NH + hd) * kStride + 1] = l_run;
    }
#pragma unroll
    for (int h = 0; h < NH; ++h)
#pragma unroll
        for (int x = 0; x < DPL; ++x) mg[(warp * NH + h) * kStride + 2 + lane * DPL + x] = o[h][x];
    __syncthreads();
    for (int idx = threadIdx.x; idx < v.rep * kStride; idx += kStepWarps * 32) {
        const int h = idx / kStride, col = idx % kStride;
        float mw[kStepWarps], M = -INFINITY;
#pragma unroll
        for (int w = 0; w < kStepWarps; ++w) {
            mw[w] = mg[(w * NH + h) * kStride];
            M = max_nan(M, mw[w]);
        }
        float acc = 0.f;
        if (col == 0) {
            acc = M;
        } else {
#pragma unroll
            for (int w = 0; w < kStepWarps; ++w)
                if (mw[w] != -INFINITY) acc += expf(mw[w] - M) * mg[(w * NH + h) * kStride + col];
        }
        part[h * part_stride + col] = acc;
    }
    __syncthreads();
}

}  // namespace still
