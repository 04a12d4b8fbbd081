// What a prefill writes of the decode state beside S and z: the K / V rows, the scores, the selection and the header.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/still.h"

namespace still {

__device__ __forceinline__ void write_header(int32_t *hdr, const still_params_t &p, long long cap, long long t) {
    hdr[0] = 0x5354494c;  // "STIL"
    hdr[1] = 1;
    hdr[2] = p.B; hdr[3] = p.H; hdr[4] = p.Hkv; hdr[5] = p.d; hdr[6] = p.d_f;
    hdr[7] = p.chunk; hdr[8] = p.topk; hdr[9] = p.dtype;
    hdr[10] = (int32_t)(cap & 0xffffffffll); hdr[11] = (int32_t)(cap >> 32);
    hdr[12] = (int32_t)(t & 0xffffffffll); hdr[13] = (int32_t)(t >> 32);
    hdr[14] = 0; hdr[15] = 0;
}

// Everything of the decode state that a prefill only has to put in its place, by blocks of 256 threads, in one launch
// (as four strided copies and two kernels it was 27 us of a 1003-token prompt, nearly all of it launches), or among the blocks of
// gather_kernel, where there is one (the launch of its own is 4.4 us of such a prompt):
//   kv_blocks per (K or V, batch, KV head): the rows [first, N) of the sequence into their ring rows (position q in row
//     q % kvr; first > 0 only with a salient-cache budget), 16 bytes a thread and step;
//   score_blocks per (batch, query head): the scores;
//   then a warp per (batch, query head, chunk): the selected positions, also as bit masks -- bit j of word w is set when
//     position chunk * C + 32 w + j is among them;
//   the last block: the header.
struct StateParts {
    const char *K, *V;
    char *k_cache, *v_cache;
    const float *scores;
    float *score_out;
    const int32_t *sel;
    int32_t *sel_out, *hdr;
    uint32_t *mask_out;
    long long N, first, kvr, cap, T, capT;
    int BH, BHkv, row_bytes, C, lam, kv_blocks, score_blocks, sel_blocks;
    long long blocks;
};
constexpr int kStateSteps = 4;   // pieces (K / V) or scores per thread
__device__ __forceinline__ void write_state_block(const StateParts &s, const still_params_t &p, long long blk) {
    const long long n_kv = 2ll * s.BHkv * s.kv_blocks, n_sc = (long long)s.BH * s.score_blocks;
    if (blk < n_kv) {
        const long long unit = blk / s.kv_blocks, head = unit >> 1;
        const int ppr = s.row_bytes / 16;
        const long long n = (s.N - s.first) * ppr, i0 = (blk - unit * s.kv_blocks) * (256 * kStateSteps) + threadIdx.x;
        const uint4 *src = reinterpret_cast<const uint4 *>((unit & 1 ? s.V : s.K) + (head * s.N + s.first) * s.row_bytes);
        uint4 *dst = reinterpret_cast<uint4 *>((unit & 1 ? s.v_cache : s.k_cache) + head * s.kvr * s.row_bytes);
        uint4 v[kStateSteps];
#pragma unroll
        for (int k = 0; k < kStateSteps; ++k)
            if (i0 + 256 * k < n) v[k] = src[i0 + 256 * k];
#pragma unroll
        for (int k = 0; k < kStateSteps; ++k) {
            const long long i = i0 + 256 * k;
            if (i < n) {
                const uint32_t q = (uint32_t)(i / ppr + s.first), r = q < s.kvr ? q : q % (uint32_t)s.kvr;
                dst[(long long)r * ppr + i % ppr] = v[k];
            }
        }
        return;
    }
    blk -= n_kv;
    if (blk < n_sc) {
        const long long bh = blk / s.score_blocks, i0 = (blk - bh * s.score_blocks) * (256 * kStateSteps) + threadIdx.x;
#pragma unroll
        for (int k = 0; k < kStateSteps; ++k)
            if (i0 + 256 * k < s.N) s.score_out[bh * s.cap + i0 + 256 * k] = s.scores[bh * s.N + i0 + 256 * k];
        return;
    }
    blk -= n_sc;
    if (blk < s.sel_blocks) {
        const long long wid = blk * 8 + (threadIdx.x >> 5);
        if (wid >= (long long)s.BH * s.T) return;
        const int lane = threadIdx.x & 31;
        const long long bh = wid / s.T, c = wid % s.T;
        const int32_t *si = s.sel + (bh * s.T + c) * s.lam;
        int32_t *so = s.sel_out + (bh * s.capT + c) * s.lam;
        int pos[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            pos[i] = lane + 32 * i < s.lam ? si[lane + 32 * i] : -1;
            if (lane + 32 * i < s.lam) so[lane + 32 * i] = pos[i];
        }
        for (int w = 0; w < s.C / 32; ++w) {
            const long long p0 = c * s.C + 32ll * w;
            uint32_t bits = 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (pos[i] >= p0 && pos[i] < p0 + 32) bits |= 1u << (int)(pos[i] - p0);
            bits = __reduce_or_sync(0xffffffffu, bits);
            if (lane == 0) s.mask_out[(bh * s.capT + c) * (s.C / 32) + w] = bits;
        }
        return;
    }
    if (threadIdx.x == 0) write_header(s.hdr, p, s.cap, s.N);
}

}  // namespace still
