// Tensor-core prefill path for bf16 (sm_100a): salient K/V compaction and the
// softmax-attention + merge kernel on tcgen05 / TMEM / TMA.
//
// Softmax Attention Branch of Algorithm 1 + the merge equation of Sec. 3.3.
// For a query in chunk c the keys are: the selected tokens of chunks 0..c-2, all
// of chunk c-1, and chunk c up to the query itself.  The selected rows of every
// chunk are first compacted per query head into K_sel / V_sel ([B*H, sel_rows, d],
// ascending position), so that "selected tokens of chunks 0..c-2" is the prefix
// [0, (c-1)*lambda) of a contiguous array that TMA can tile.
//
// One CTA owns 256 consecutive query rows of one (batch, head), a pair of CTAs 512: two query tiles A and B of 128
// (256) rows.  Their keys come as a stream of 128-key tiles: SEL tiles j (rows [128j, 128j+128) of K_sel / V_sel), and
// the LOC tiles around the rows (rows of K / V at positions [128m, 128m+128)).  First the SEL tiles that both query
// tiles see (before them what has already left the window of B), then what only one of them sees, by turns.  Which
// columns of a tile a query row sees is a per-row column interval, applied as a mask in the softmax.
//
// Warp roles (384 threads):
//   warps 0-7  softmax, four warps per query tile, one thread per query row (tcgen05.ld of the S row): online softmax in
//              the log2 domain with lazy rescaling of O, P to TMEM as bf16; then the epilogue: O / l merged with the
//              linear branch (N_LA, D_LA) under one denominator and stored as bf16
//   warp 8     TMA producer: Q tiles once, then K and V tiles through mbarrier rings
//   warp 9     MMA issuer (one elected thread): S = Q_X K^T (operands in shared memory, SWIZZLE_128B K-major),
//              O_X += P_X V (P_X read from TMEM, V in shared memory MN-major)
//   (warps 10, 11 only give up their registers)
//
// Every mbarrier wait is bounded: on expiry the kernel records
// STILL_ERR_DEVICE_TIMEOUT in the status word, all roles leave their loops, and
// tensor memory is freed before the CTA exits.
#include "still_tc.h"

#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>

#include "still_common.cuh"
#include "still_tc_ptx.cuh"

namespace still {

namespace {

constexpr int kBlockM = 128;   // query rows per tile and CTA
constexpr int kBlockN = 128;   // keys per tile
constexpr int kThreads = 384, kProducerWarp = 8, kMmaWarp = 9;
constexpr int kMaxDynamicSmem = 232448;   // 227 KiB: the most a CTA can be given on sm_100
using namespace ptx;

// ----------------------------------------------------------------- shared memory plan

// In a CTA pair every CTA holds half of each key tile: 64 of the 128 keys of K, half of the value columns of V.
template <int D, bool kPair>
struct AttnPlan {
    static constexpr int kQTile = kBlockM * D * 2;             // one Q tile of this CTA
    static constexpr int kKRows = kPair ? kBlockN / 2 : kBlockN;
    static constexpr int kVCols = kPair ? D / 2 : D;
    static constexpr int kKTile = kKRows * D * 2;
    static constexpr int kVTile = kBlockN * kVCols * 2;
    static constexpr int kStages = 5;                          // of the ring: a K and a V tile each
    static constexpr int kQ = 0;
    static constexpr int kK = kQ + 2 * kQTile;
    static constexpr int kV = kK + kStages * kKTile;
    static constexpr int kBar = kV + kStages * kVTile;         // mbarriers
    static constexpr int kNumBars = 1 + 2 * kStages + 2 + 2 + 2 + 2 + 1;
    static constexpr int kMisc = kBar + kNumBars * 8;          // tmem base, abort flag, "a CTA has failed before"
    static constexpr int kTotal = kMisc + 16;
    static constexpr int kAlloc = kTotal + 1024;               // slack to align the base to 1024
    static_assert(kAlloc <= kMaxDynamicSmem, "attention kernel: the shared-memory plan exceeds what a CTA can have");
    static_assert(kMisc % 8 == 0 && kKTile % 1024 == 0 && kVTile % 1024 == 0, "attention kernel: operand tiles are swizzle-aligned");
};

struct AttnBars {
    uint64_t *q_full;
    uint64_t *kv_full, *kv_empty;   // [kStages]
    uint64_t *s_full;    // [2] S of query tile x is in tensor memory
    uint64_t *s_free;    // [2] ... and has been read
    uint64_t *p_full;    // [2] P_x is in tensor memory
    uint64_t *pv_done;   // [2] O_x includes the tile's product (and P_x may be overwritten)
    uint64_t *drain;     // MMA warp: everything issued has completed (failure path)
    template <class P>
    __device__ __forceinline__ static AttnBars at(uint8_t *smem, P) {
        AttnBars b;
        b.q_full = reinterpret_cast<uint64_t *>(smem + P::kBar);
        b.kv_full = b.q_full + 1;
        b.kv_empty = b.kv_full + P::kStages;
        b.s_full = b.kv_empty + P::kStages;
        b.s_free = b.s_full + 2;
        b.p_full = b.s_free + 2;
        b.pv_done = b.p_full + 2;
        b.drain = b.pv_done + 2;
        return b;
    }
};

// A stage of the ring and the parity of its round.
struct RingPos {
    int stage, parity;
    __device__ __forceinline__ void next(int n_stages) {
        if (++stage == n_stages) {
            stage = 0;
            parity ^= 1;
        }
    }
};

// Tensor memory (512 columns): S_A, S_B, O_A, O_B and, beside them, P_A and P_B (64 columns each: 128 bf16).  P has a place
// of its own so that S_x of the next tile can be formed while the softmax warps still work on this one, which they hold
// in registers.  At D = 128 that leaves 128 columns for S: S_A and S_B share them, one after the other.
template <int D>
struct TmemPlan {
    static constexpr bool kOneS = D == 128;
    __device__ __forceinline__ static uint32_t s(int x) { return kOneS ? 0u : (uint32_t)x * 128u; }
    __device__ __forceinline__ static uint32_t p(int x) { return (kOneS ? 128u : 384u) + (uint32_t)x * 64u; }
    __device__ __forceinline__ static uint32_t o(int x) { return 256u + (uint32_t)x * (uint32_t)D; }
};

// The key stream of a CTA (or CTA pair).  Query tile x takes its SEL tiles in the order of their positions, then its LOC
// tiles; that order is the one in which a row's weights are rounded and summed, and it does not depend on where the query
// tiles lie.  Entries: n_lead SEL tiles that only A sees (the oldest of its window, with a salient-cache budget), n_shared
// that both use, then what is left of either, A and B by turns until one has no more.  (With an entry's query tiles one
// after the other at the end, A waited for B there and B for A.  The n_lead tiles, at most two, wait for nobody: taken
// behind the shared ones and by turns with B's, 32 heads x 131072 tokens capped at 896 took 7908 us a call, like this 7992.)
struct Stream {
    int n_lead, n_shared;
    int sel_a, n_sel_a, loc_a, n_a;  // A's first SEL tile, SEL tiles, first LOC tile, and its entries behind the shared ones
    int sel_b, n_sel_b, loc_b, n_b;
    __device__ __forceinline__ int first_own(int x) const { return n_shared + (x ? 0 : n_lead); }   // (x's tiles before those)
    __device__ __forceinline__ int entries() const { return n_lead + n_shared + n_a + n_b; }
    __device__ __forceinline__ int entries_of(int x) const { return first_own(x) + (x ? n_b : n_a); }
    __device__ __forceinline__ bool shared(int e) const { return e >= n_lead && e < n_lead + n_shared; }
    // k-th tile of query tile x: a SEL tile, or a LOC tile?  Returns its number.
    __device__ __forceinline__ int tile_of(int x, int k, bool &sel) const {
        const int n = x ? n_sel_b : n_sel_a;
        sel = k < n;
        return k + (sel ? (x ? sel_b : sel_a) : (x ? loc_b : loc_a) - n);
    }
    // ... and its entry
    __device__ __forceinline__ int entry(int x, int k) const {
        const int i = k - first_own(x), turns = min(n_a, n_b);
        return i < 0 ? k + (x ? n_lead : 0) : n_lead + n_shared + (i < turns ? 2 * i + x : i + turns);
    }
    // the tile of entry e
    __device__ __forceinline__ int tile(int e, bool &sel) const {
        const int s = e - n_lead - n_shared, turns = min(n_a, n_b);
        if (s < 0) return tile_of(0, e, sel);
        const int x = s < 2 * turns ? s & 1 : (n_a > n_b ? 0 : 1);
        return tile_of(x, first_own(x) + (s < 2 * turns ? s >> 1 : s - turns), sel);
    }
};

// Which row block of which (batch, head) the i-th CTA (or CTA pair) works on.  The row blocks of the heads are launched
// in the order of their length, longest first, so that the last wave holds the short ones; with the heads one after the
// other it held whole heads (128 heads x 4096 tokens, d = 64, on 148 SMs: 592 us a call, in this order 551; with a
// quarter of the tokens kept 612 and 582).  Heads whose K / V do not fit the L2 cache together are taken in sets that do,
// about half the cache, one set after the other.
__device__ __forceinline__ void row_block(int i, int n_blocks, int n_heads, int set_heads, int &block, int &bh) {
    int bh0 = 0, heads = n_heads;
    if (set_heads < n_heads) {
        const int set = i / (n_blocks * set_heads);
        i -= set * n_blocks * set_heads;
        bh0 = set * set_heads;
        heads = min(set_heads, n_heads - bh0);
    }
    const int q = i / heads;
    block = n_blocks - 1 - q;
    bh = bh0 + (i - q * heads);
}

__device__ __forceinline__ int sel_limit(long long pos, int C, int lam) {  // end of the visible range of K_sel
    long long c = pos / C;
    return c >= 2 ? (int)((c - 1) * lam) : 0;
}
// Start of the visible range: 0, or with a salient-cache budget of `budget` tokens per head (a multiple of lam;
// the oldest cached tokens have left for the linear state) the last `budget` entries before the end.
__device__ __forceinline__ int sel_start(int limit, int budget) { return budget > 0 ? max(limit - budget, 0) : 0; }

// The key stream of the query tiles that start at rows R0 and R0 + rows, of `rows` (a multiple of 128) rows each.
__device__ __forceinline__ Stream make_stream(int R0, int rows, int N, int C, int lam, int budget) {
    Stream st;
    const int last_m = (N - 1) / kBlockN, m_a = R0 / kBlockN, m_b = m_a + rows / kBlockN;
    const int last_a = min(R0 + rows, N) - 1, last_b = min(R0 + 2 * rows, N) - 1;
    // SEL tiles [a0, a1) and [b0, b1): a tile's first row sees the oldest entries, its last row the newest
    const int a0 = sel_start(sel_limit(R0, C, lam), budget) / kBlockN, a1 = (sel_limit(last_a, C, lam) + kBlockN - 1) / kBlockN;
    st.sel_a = a0;
    st.n_sel_a = max(a1 - a0, 0);
    st.loc_a = max(m_a - 1, 0);
    st.n_lead = st.n_shared = st.sel_b = st.n_sel_b = st.loc_b = st.n_b = 0;
    if (R0 + rows < N) {
        const int b0 = sel_start(sel_limit(R0 + rows, C, lam), budget) / kBlockN, b1 = (sel_limit(last_b, C, lam) + kBlockN - 1) / kBlockN;
        st.n_shared = max(a1 - b0, 0);                    // (a0 <= b0 and a1 <= b1)
        st.n_lead = st.n_shared > 0 ? b0 - a0 : 0;
        st.sel_b = b0;
        st.n_sel_b = max(b1 - b0, 0);
        st.loc_b = m_b - 1;
        st.n_b = st.n_sel_b - st.n_shared + min(m_b + rows / kBlockN - 1, last_m) - st.loc_b + 1;
    }
    st.n_a = st.n_sel_a - st.n_lead - st.n_shared + min(m_b - 1, last_m) - st.loc_a + 1;
    return st;
}

// ---------------------------------------------------------------------------
// Softmax warps of the attention kernels (one warpgroup per query tile, a thread per query row) and the merge epilogue.
// x is the query tile (0: A, 1: B), tile_row0 the position of the tile's first row, stage_tile the tile's Q region in
// shared memory (the epilogue's staging space).  The barriers are this CTA's, except that in a CTA pair what the issuing
// warp waits for is announced on the first CTA's.
// ---------------------------------------------------------------------------
template <int D, bool kPair>
__device__ __forceinline__ void softmax_role(const Stream &st, const AttnBars &bar, const int x, const int tile_row0,
                                             const uint32_t tmem_base, volatile int *abort_flag, int *status,
                                             uint8_t *stage_tile, const __nv_bfloat16 *y_part,
                                             const float *d_part, const int n_parts, const long long part_stride_y,
                                             const long long part_stride_d, __nv_bfloat16 *Y, const int bh,
                                             const int N, const int C, const int lam, const int budget,
                                             const float scale_log2) {
    constexpr int kStages = AttnPlan<D, kPair>::kStages;
    // The MUFU unit (one warp instruction per eight cycles) would need 1024 cycles for a query tile's exponentials, which is as
    // long as the tensor pipe needs for the tile's two products; so one of kPolyEvery column pairs takes 2^x from the FMA
    // pipes instead (see exp2_fma2), interleaved with the others so that both units work at the same time.  The same share
    // on both head dims: equal logits then get equal weights, bit for bit.  (4096 tokens, d = 64: none 536 us, one of 8 515,
    // of 4 512, 5 of 16 517; 32768 tokens, d = 128, every token kept, in turn on one box: one of 8 15.17 ms, of 4 15.28.)
    constexpr int kPolyEvery = 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto arrive_first = [&](uint64_t *b) {   // on the barrier of the CTA whose warp issues the products
        if constexpr (kPair) mbar_arrive_cluster(mapa(smem_u32(b), 0));
        else mbar_arrive(b);
    };
    const int row_in_tile = ((warp & 3) << 5) | lane;
    const int t = tile_row0 + row_in_tile;         // this thread's query position
    const int n_mine = st.entries_of(x);
    if (n_mine > 0) {                              // (in a pair also where none of this CTA's rows are below N)
        const uint32_t lane_addr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
        const uint32_t s_addr = lane_addr + TmemPlan<D>::s(x), p_addr = lane_addr + TmemPlan<D>::p(x), o_addr = lane_addr + TmemPlan<D>::o(x);
        const int tq = min(t, N - 1);              // rows past N mimic the last row (never stored)
        const int c = tq / C;
        const int lim_sel = c >= 2 ? (c - 1) * lam : 0, lo_sel = sel_start(lim_sel, budget);
        const int loc_lo = c >= 1 ? (c - 1) * C : 0;
        float m_used = -INFINITY, l_sum = 0.f;     // log2 domain
        bool ok = true;
        // A wait can end in one lane and run out in another, and the warp has to stay together for the instructions that take
        // it whole.  So no wait is left by a branch: the loop runs out with whatever has been read (a wait gives up at once
        // where a role has given up before), and the warp votes behind it.  (A vote behind every wait took 0.6 % longer at
        // 64 heads x 32768 tokens, d = 128, one a tile 0.5 % at 128 x 4096, d = 64; skipping the waits after a failure 2 %.)
        auto wait = [&](uint64_t *b, int parity, int where) {
            ok = mbar_wait(b, (uint32_t)parity, abort_flag, status, where) && ok;
        };
        // one thread of a query tile releases the stage of its last product: its share of two, or both where the entry is
        // the tile's alone
        auto release = [&](int e) {
            if (row_in_tile != 0 || !ok) return;
            mbar_arrive(bar.kv_empty + e % kStages);
            if (!st.shared(e)) mbar_arrive(bar.kv_empty + e % kStages);
        };
        for (int k = 0; k < n_mine; ++k) {
            // visible column interval [lo, hi] of this row in the stream tile
            bool sel;
            const int p0 = st.tile_of(x, k, sel) * kBlockN;
            const int lo = max((sel ? lo_sel : loc_lo) - p0, 0), hi = min((sel ? lim_sel - 1 : tq) - p0, kBlockN - 1);
            const bool need_mask = __any_sync(0xffffffffu, lo > 0 || hi < kBlockN - 1);
            const bool none = need_mask && !__any_sync(0xffffffffu, lo <= hi);   // (a warp whose rows see none of it skips the arithmetic)
            wait(bar.s_full + x, k & 1, 8);
            tc_fence_after();
            if (none) {
                __syncwarp();   // (no lane still looks for this phase)
                if (lane == 0) arrive_first(bar.s_free + x);
                uint32_t masked[32];   // the weights of masked columns: 0, and 2^-126 from the cubic
#pragma unroll
                for (int j = 0; j < 32; ++j) masked[j] = j % kPolyEvery == 0 ? 0x00800080u : 0u;
                if (k > 0) {
                    wait(bar.pv_done + x, (k - 1) & 1, 11);
                    release(st.entry(x, k - 1));
                    tc_fence_after();
                }
                __syncwarp();
                tmem_st32(p_addr, masked);
                tmem_st32(p_addr + 32, masked);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) arrive_first(bar.p_full + x);
                continue;
            }
            uint32_t sr[128];
            tmem_ld32(s_addr, sr);
            tmem_ld32(s_addr + 32, sr + 32);
            tmem_ld32(s_addr + 64, sr + 64);
            tmem_ld32(s_addr + 96, sr + 96);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_first(bar.s_free + x);
            float *s = reinterpret_cast<float *>(sr);
            if (need_mask) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    // columns of this block of 32 that the row sees, as a bit set
                    const int l = min(max(lo - 32 * q, 0), 32), n = min(max(hi - 32 * q + 1, 0), 32);
                    const uint32_t seen = n > l ? (0xffffffffu >> (32 - n)) & (0xffffffffu << l) : 0u;
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (!((seen >> j) & 1u)) s[q * 32 + j] = -INFINITY;
                }
            }
            float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
            for (int j = 0; j < 128; j += 8) {
                mx0 = max3_nan(mx0, s[j], s[j + 1]);
                mx1 = max3_nan(mx1, s[j + 2], s[j + 3]);
                mx2 = max3_nan(mx2, s[j + 4], s[j + 5]);
                mx3 = max3_nan(mx3, s[j + 6], s[j + 7]);
            }
            const float mt = max_nan(max_nan(mx0, mx1), max_nan(mx2, mx3)) * scale_log2;
            // lazy rescale: keep the old reference unless the new maximum exceeds it by 2^8.  A NaN or +inf logit makes the
            // reference NaN, and with it every weight that is not a cubic's: those would lose it in the clamp.
            const bool grow = !(mt <= m_used + 8.f);
            float alpha = 1.f;
            if (grow) {
                const float m_new = mt < INFINITY ? mt : NAN;
                alpha = (m_used == -INFINITY) ? 0.f : ex2(m_used - m_new);
                m_used = m_new;
            }
            // the previous product is in O, has read P and is done with its stage (asked for as late as P is written: the
            // issuing warp takes it up behind a product of the other query tile)
            auto previous_done = [&]() { wait(bar.pv_done + x, (k - 1) & 1, 11); };
            if (k > 0 && __any_sync(0xffffffffu, grow)) {
                previous_done();
                tc_fence_after();
                {
#pragma unroll
                    for (int q = 0; q < D / 32; ++q) {
                        uint32_t orow[32];
                        tmem_ld32(o_addr + q * 32, orow);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 32; ++j) orow[j] = __float_as_uint(__uint_as_float(orow[j]) * alpha);
                        tmem_st32(o_addr + q * 32, orow);
                    }
                }
            }
            l_sum *= alpha;
            const float neg_m = (m_used == -INFINITY) ? 0.f : -m_used;
            const float2 scale2 = make_float2(scale_log2, scale_log2), negm2 = make_float2(neg_m, neg_m);
            float2 acc = make_float2(0.f, 0.f);
            // P = 2^(s * scale - m) as bf16
            uint32_t pk[2][32];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const float2 sv = make_float2(s[q * 64 + 2 * j], s[q * 64 + 2 * j + 1]);
                    const float2 xv = __ffma2_rn(sv, scale2, negm2);
                    const float2 pr = j % kPolyEvery == 0 ? exp2_fma2(xv) : make_float2(ex2(xv.x), ex2(xv.y));
                    acc = __fadd2_rn(acc, pr);
                    pk[q][j] = pack_bf16(pr.x, pr.y);
                }
            }
            if (k > 0) {
                previous_done();
                tc_fence_after();
                release(st.entry(x, k - 1));
                __syncwarp();
            }
            tmem_st32(p_addr, pk[0]);
            tmem_st32(p_addr + 32, pk[1]);
            l_sum += acc.x + acc.y;
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_first(bar.p_full + x);
        }
        // ---- epilogue: y = (O e^{m-ms} + e^{-ms} N_LA) / (l e^{m-ms} + e^{-ms} D_LA), ms = max(m, 0)
        // The linear branch arrives as up to two partial results (one per feature half): y_p = N_p / D_p as bf16
        // and D_p, so N_LA = sum y_p D_p and D_LA = sum D_p.  A thread owns a row, but loads / stores in which
        // every lane touches a different row cost a memory instruction per 16 bytes and row; so the y_p come in
        // and Y goes out through shared memory with 16 consecutive lanes per row.  The staging space is this
        // warp's 32 rows of the tile's Q region (one row = D bf16 = 2 D bytes: D / 2 columns of both parts), free
        // once the tile's last Q K^T has completed; 16-byte pieces are swizzled by the row so that row-wise and
        // piece-wise accesses avoid bank conflicts.
        wait(bar.pv_done + x, (n_mine - 1) & 1, 9);   // (every query tile has a LOC tile)
        if (__all_sync(0xffffffffu, ok)) {
            tc_fence_after();
            release(st.entry(x, n_mine - 1));   // (the other query tile may have entries left)
            constexpr int kRowBytes = D * 2, kPieces = kRowBytes / 16;   // pieces of 16 bytes per staged row
            constexpr int kPartPieces = kPieces / 2;                     // pieces of one part (D / 2 columns)
            uint8_t *stg = stage_tile + (warp & 3) * 32 * kRowBytes;
            const int t0 = tile_row0 + (warp & 3) * 32;                    // first row of this warp
            float fs = 1.f, fa = 0.f, fb = 0.f, dla = 0.f;
            if (n_parts > 0 && t < N) {
                const float da = d_part[(long long)bh * N + t];
                const float db = n_parts > 1 ? d_part[part_stride_d + (long long)bh * N + t] : 0.f;
                dla = da + db;
                if (dla > 0.f) {
                    const float m_nat = m_used * 0.6931471805599453f;
                    const float ms = fmaxf(m_nat, 0.f);
                    fs = __expf(m_nat - ms);
                    const float fl = __expf(-ms);
                    fa = fl * da;
                    fb = fl * db;
                }
            }
            const float inv = 1.f / (l_sum * fs + fa + fb);
            const bool with_la = (n_parts > 0) && __any_sync(0xffffffffu, dla > 0.f);
            uint32_t out[D / 2];   // the row as packed bf16
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {   // halves of D / 2 columns
                if (with_la) {
                    __syncwarp();
                    uint4 v[kPieces];   // (all requested before the first is stored: one round trip to memory, not kPieces)
#pragma unroll
                    for (int it = 0; it < kPieces; ++it) {
                        const int id = it * 32 + lane, row = id / kPieces, c = id % kPieces;
                        const int part = c / kPartPieces, cc = c % kPartPieces;
                        v[it] = make_uint4(0, 0, 0, 0);
                        if (t0 + row < N && part < n_parts)
                            v[it] = *reinterpret_cast<const uint4 *>(y_part + part * part_stride_y + ((long long)bh * N + t0 + row) * D +
                                                                     hh * (D / 2) + cc * 8);
                    }
#pragma unroll
                    for (int it = 0; it < kPieces; ++it) {
                        const int id = it * 32 + lane, row = id / kPieces, c = id % kPieces;
                        *reinterpret_cast<uint4 *>(stg + row * kRowBytes + ((c ^ (row & (kPieces - 1))) << 4)) = v[it];
                    }
                    __syncwarp();
                }
#pragma unroll
                for (int q = 0; q < D / 64; ++q) {
                    uint32_t orow[32];
                    tmem_ld32(o_addr + hh * (D / 2) + q * 32, orow);
                    tmem_wait_ld();
#pragma unroll
                    for (int j8 = 0; j8 < 4; ++j8) {
                        uint4 pa = make_uint4(0, 0, 0, 0), pb = pa;
                        if (with_la) {
                            const int ca = q * 4 + j8, cb = kPartPieces + ca;
                            pa = *reinterpret_cast<const uint4 *>(stg + lane * kRowBytes + ((ca ^ (lane & (kPieces - 1))) << 4));
                            pb = *reinterpret_cast<const uint4 *>(stg + lane * kRowBytes + ((cb ^ (lane & (kPieces - 1))) << 4));
                        }
                        const uint32_t wa[4] = {pa.x, pa.y, pa.z, pa.w}, wb[4] = {pb.x, pb.y, pb.z, pb.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {   // two columns per 32-bit word
                            const float la0 = fmaf(fa, __uint_as_float(wa[e] << 16), fb * __uint_as_float(wb[e] << 16));
                            const float la1 = fmaf(fa, __uint_as_float(wa[e] & 0xffff0000u), fb * __uint_as_float(wb[e] & 0xffff0000u));
                            const float a0 = fmaf(__uint_as_float(orow[8 * j8 + 2 * e]), fs, la0);
                            const float a1 = fmaf(__uint_as_float(orow[8 * j8 + 2 * e + 1]), fs, la1);
                            out[hh * (D / 4) + q * 16 + 4 * j8 + e] = pack_bf16(a0 * inv, a1 * inv);
                        }
                    }
                }
            }
            // Y: own row into the staging space, then the warp writes its 32 rows piece-wise
            __syncwarp();
#pragma unroll
            for (int c = 0; c < kPieces; ++c)
                *reinterpret_cast<uint4 *>(stg + lane * kRowBytes + ((c ^ (lane & (kPieces - 1))) << 4)) =
                    make_uint4(out[4 * c], out[4 * c + 1], out[4 * c + 2], out[4 * c + 3]);
            __syncwarp();
#pragma unroll
            for (int it = 0; it < kPieces; ++it) {
                const int id = it * 32 + lane, row = id / kPieces, c = id % kPieces;
                if (t0 + row < N)
                    *reinterpret_cast<uint4 *>(Y + ((long long)bh * N + t0 + row) * D + c * 8) =
                        *reinterpret_cast<const uint4 *>(stg + row * kRowBytes + ((c ^ (row & (kPieces - 1))) << 4));
            }
        }
    }
}

// TMA producer (one thread): the Q tiles, then the K and V tiles of the stream, as far ahead as the ring has free stages.  In a
// pair every CTA loads its halves; their byte counts complete on the first CTA's barriers.
template <int D, bool kPair, class TellPeer>
__device__ __forceinline__ void producer_role(const Stream &st, const AttnBars &bar, uint8_t *smem, const uint32_t rank,
                                              const CUtensorMap &tm_q, const CUtensorMap &tm_k, const CUtensorMap &tm_v,
                                              const CUtensorMap &tm_ksel, const CUtensorMap &tm_vsel, const int q_row,
                                              const int kv_row0, const int sel_row0, volatile int *abort_flag, int *status,
                                              TellPeer tell_peer) {
    using P = AttnPlan<D, kPair>;
    constexpr int kCtas = kPair ? 2 : 1, kStages = P::kStages;
    const uint32_t q_full0 = mapa(smem_u32(bar.q_full), 0), kv_full0 = mapa(smem_u32(bar.kv_full), 0);
    auto load = [&](uint8_t *dst, const CUtensorMap &map, uint64_t *b, uint32_t b0, int col, int row) {
        if constexpr (kPair) tma_load_2d_pair(dst, &map, b0, col, row);
        else tma_load_2d(dst, &map, b, col, row);
    };
    const int n_q = st.n_b > 0 ? 2 : 1, n = st.entries();   // (every query tile has a LOC tile)
    if (rank == 0) mbar_expect_tx(bar.q_full, kCtas * n_q * P::kQTile);
    for (int x = 0; x < n_q; ++x)
        for (int half = 0; half < D / 64; ++half)
            load(smem + P::kQ + x * P::kQTile + half * (kBlockM * 128), tm_q, bar.q_full, q_full0, half * 64,
                 q_row + ((int)rank + x * kCtas) * kBlockM);
    bool ok = true;
    int armed = 0;
    RingPos pos{0, 0};
    for (; armed < n; ++armed) {
        ok = mbar_wait(bar.kv_empty + pos.stage, pos.parity ^ 1, abort_flag, status, 1);
        if (!ok) break;
        bool sel;
        const int tile = st.tile(armed, sel), row = (sel ? sel_row0 : kv_row0) + tile * kBlockN;
        if (rank == 0) mbar_expect_tx(bar.kv_full + pos.stage, kCtas * (P::kKTile + P::kVTile));
        for (int half = 0; half < D / 64; ++half)   // (of a pair: this CTA's 64 keys)
            load(smem + P::kK + pos.stage * P::kKTile + half * (P::kKRows * 128), sel ? tm_ksel : tm_k, bar.kv_full + pos.stage,
                 kv_full0 + pos.stage * 8, half * 64, row + (int)rank * P::kKRows);
        for (int q = 0; q < P::kVCols / 64; ++q)    // this CTA's value columns, 64 at a time
            load(smem + P::kV + pos.stage * P::kVTile + q * (kBlockN * 128), sel ? tm_vsel : tm_v, bar.kv_full + pos.stage,
                 kv_full0 + pos.stage * 8, (int)rank * P::kVCols + q * 64, row);
        pos.next(kStages);
    }
    // leave no copy in flight behind.  In a pair the first CTA's barriers count both CTAs' bytes; the second, where it has
    // given up and the first may not know of its last copies, waits out a fixed stretch that is long against a tile load.
    const long long t0 = clock64();
    if constexpr (kPair) {
        if (!ok) tell_peer();
    }
    if (rank == 0) {
        mbar_wait_drain(bar.q_full, 0, t0);
        mbar_drain_ring(bar.kv_full, kStages, armed, t0);
    } else if (!ok) {
        while (clock64() - t0 < 200000) {}
    }
}

// MMA issuer (in a pair: of the first CTA).  The whole warp walks the items and waits on the barriers; one elected lane
// issues.  Kept this way, control flow and every descriptor are the same in all lanes, which lets them live in the
// warp's uniform registers, where the tensor-core instructions take their operands from.  (With a single lane in a
// divergent branch each instruction cost that lane 55 - 80 cycles of operand marshalling, whatever the instruction's
// size, and the tensor pipe starved behind it.)  A failed wait does not leave the loop: it switches off the remaining
// waits and instructions, and the loop runs out.
//
// Q K^T runs three items ahead of P V: P_A V, Q_B K^T of B's next tile, P_B V, Q_A K^T of A's next but one, and so on.
// S of A's next tile is then complete when its softmax warps come back for it, and where S_A and S_B share their place
// the warps of A have read theirs by the time B's is to be formed.  What bounds the kernel is then the softmax warps'
// arithmetic, two of them per scheduler (32768 tokens, d = 128: issue slots 52 %, special-function unit 51 %, tensor pipe 69 %;
// 4096 tokens, d = 64: 50, 45 and 30 %), and for short streams the start and the end of a CTA.  With P over S, S of a tile
// waited for the softmax warps of the tile before and these for it (us a call, then and now, in turn on one box: 64 heads x 32768
// tokens, d = 128, every token kept 15887 and 15154, a quarter 6665 and 6208; 32 x 131072, capped at 896, 8697 and 7809; 128 x
// 4096, d = 64, every token 551 and 502, a quarter 585 and 515; the scan and the score kernel have a part in the quarters and in
// the capped call).  Two threads per row instead of one (16 softmax warps) were slower by 10 %: the stream's bookkeeping doubles.
template <int D, bool kPair, class TellPeer>
__device__ __forceinline__ void mma_role(const Stream &st, const AttnBars &bar, uint8_t *smem, const uint32_t tmem_base,
                                         volatile int *abort_flag, int *status, TellPeer tell_peer) {
    using P = AttnPlan<D, kPair>;
    using TM = TmemPlan<D>;
    constexpr int kM = kPair ? 2 * kBlockM : kBlockM, kStages = P::kStages, kAhead = 3;
    constexpr uint32_t idesc_qk = make_idesc(kM, kBlockN, false);
    constexpr uint32_t idesc_pv = make_idesc(kM, D, true);
    const bool leader = elect_one();
    bool ok = mbar_wait(bar.q_full, 0, abort_flag, status, 4);
    tc_fence_after();
    // descriptors as low words: a k-step adds a constant
    const uint32_t q_lo0 = desc_lo(smem_u32(smem + P::kQ), 0);
    const uint32_t k_lo0 = desc_lo(smem_u32(smem + P::kK), 0);
    const uint32_t v_lo0 = desc_lo(smem_u32(smem + P::kV), kBlockN * 128);
    auto wait = [&](uint64_t *b, int parity, int where) {
        if (ok) ok = mbar_wait(b, (uint32_t)parity, abort_flag, status, where);
    };
    auto commit = [&](uint64_t *b) {
        if constexpr (kPair) tc_commit_pair(b, 3);
        else tc_commit(b);
    };
    // A place in the order of the products: query tile x, its k-th tile, and the ring stage of that.
    const int n_own0 = st.n_lead + 2 * st.n_shared, n_items = n_own0 + st.n_a + st.n_b;
    const int turns = min(st.n_a, st.n_b), x_last = st.n_a > st.n_b ? 0 : 1;
    struct Item {
        int m, x, k;
        RingPos pos;
    };
    auto advance = [&](Item &it) {
        ++it.m;
        if (it.m <= st.n_lead && it.m < n_own0) {
            ++it.k;
        } else if (it.m < n_own0) {
            it.x ^= 1;
            if (it.x == 1) {   // (both query tiles use the entry)
                it.k -= st.n_lead;
                return;
            }
            it.k += st.n_lead + 1;
        } else {
            const int s = it.m - n_own0;
            it.x = s < 2 * turns ? s & 1 : x_last;
            it.k = st.first_own(it.x) + (s < 2 * turns ? s >> 1 : s - turns);
        }
        it.pos.next(kStages);
    };
    Item qk{0, 0, 0, {0, 0}}, pv{0, 0, 0, {0, 0}};
    int x_prev = 0, k_prev = 0;   // of the item whose S was formed last
    auto issue_qk = [&]() {
        // K and V of the entry have arrived (B follows A on the entries that they share)
        if (qk.m >= n_own0 || qk.x == 0) wait(bar.kv_full + qk.pos.stage, qk.pos.parity, 7);
        // the place of S is free: its last tile has been read
        if constexpr (TM::kOneS) {
            if (qk.m > 0) wait(bar.s_free + x_prev, k_prev & 1, 3);
        } else {
            if (qk.k > 0) wait(bar.s_free + qk.x, (qk.k - 1) & 1, 3);
        }
        tc_fence_after();
        const uint32_t q_lo = q_lo0 + qk.x * (P::kQTile >> 4), k_lo = k_lo0 + qk.pos.stage * (P::kKTile >> 4), d_s = tmem_base + TM::s(qk.x);
        if (leader && ok) {
#pragma unroll
            for (int j = 0; j < D / 16; ++j) {
                // k-step of 16 elements: 32 bytes within a 64-element swizzle atom; atoms are 128 rows apart in a Q
                // tile, and in a K tile as many as the CTA holds
                const uint32_t off_q = ((j / 4) * (kBlockM * 128) + (j % 4) * 32) >> 4;
                const uint32_t off_k = ((j / 4) * (P::kKRows * 128) + (j % 4) * 32) >> 4;
                if constexpr (kPair) {
                    if (j == 0) mma_ss_lo_pair<idesc_qk, 0>(d_s, q_lo, k_lo);
                    else mma_ss_lo_pair<idesc_qk, 1>(d_s, q_lo + off_q, k_lo + off_k);
                } else {
                    if (j == 0) mma_ss_lo<idesc_qk, 0>(d_s, q_lo, k_lo);
                    else mma_ss_lo<idesc_qk, 1>(d_s, q_lo + off_q, k_lo + off_k);
                }
            }
            commit(bar.s_full + qk.x);
        }
        x_prev = qk.x;
        k_prev = qk.k;
        advance(qk);
    };
    auto issue_pv = [&]() {
        const uint32_t v_lo = v_lo0 + pv.pos.stage * (P::kVTile >> 4), d_o = tmem_base + TM::o(pv.x), a_p = tmem_base + TM::p(pv.x);
        const uint32_t acc0 = pv.k > 0 ? 1u : 0u;
        wait(bar.p_full + pv.x, pv.k & 1, 5);
        tc_fence_after();
        if (leader && ok) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {   // 16 keys a step
                if constexpr (kPair) mma_ts_lo_pair<idesc_pv>(d_o, a_p + j * 8, v_lo + j * (16 * 128 >> 4), j == 0 ? acc0 : 1u);
                else mma_ts_lo<idesc_pv>(d_o, a_p + j * 8, v_lo + j * (16 * 128 >> 4), j == 0 ? acc0 : 1u);
            }
            commit(bar.pv_done + pv.x);
        }
        advance(pv);
    };
    for (int m = 0; m < min(kAhead, n_items); ++m) issue_qk();
    while (pv.m < n_items) {
        issue_pv();
        if (qk.m < n_items) issue_qk();
    }
    if (!__all_sync(0xffffffffu, ok) && leader) {  // no MMA may still be running when tensor memory is freed
        if constexpr (kPair) {
            tell_peer();
            tc_commit_pair_local(bar.drain);
        } else {
            tc_commit(bar.drain);
        }
        mbar_wait_drain(bar.drain, 0);
    }
}

// Softmax-attention branch and merge for rows [R0, R0 + 256) (a pair: 512) of one (batch, head).
template <int D, bool kPair>
__device__ __forceinline__ void attention_body(const CUtensorMap &tm_q, const CUtensorMap &tm_k, const CUtensorMap &tm_v,
                                               const CUtensorMap &tm_ksel, const CUtensorMap &tm_vsel, const __nv_bfloat16 *y_part,
                                               const float *d_part, int n_parts, __nv_bfloat16 *Y, int *status, int H, int Hkv, int N,
                                               int C, int lam, int budget, int sel_rows, int sel_identity, float scale_log2,
                                               int n_blocks, int n_heads, int set_heads) {
    using P = AttnPlan<D, kPair>;
    constexpr int kCtas = kPair ? 2 : 1, kRows = kCtas * kBlockM;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const AttnBars bar = AttnBars::at(smem, P{});
    uint32_t *tmem_base_slot = reinterpret_cast<uint32_t *>(smem + P::kMisc);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + P::kMisc + 4);
    volatile int *failed_before = reinterpret_cast<volatile int *>(smem + P::kMisc + 8);

    // (warp index and cluster rank through a shuffle / from the block index: values the compiler knows to be
    // the same in all lanes)
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const uint32_t rank = kPair ? blockIdx.x & 1u : 0u, peer = rank ^ 1u;
    int rb, bh;
    row_block(kPair ? blockIdx.x >> 1 : blockIdx.x, n_blocks, n_heads, set_heads, rb, bh);
    const int b = bh / H, h = bh % H, kvh = h / (H / Hkv);
    const int R0 = rb * 2 * kRows;
    const Stream st = make_stream(R0, kRows, N, C, lam, budget);
    auto sync_all = [&]() {
        if constexpr (kPair) cluster_sync_all();
        else __syncthreads();
    };

    if (threadIdx.x == 0) {
        mbar_init(bar.q_full, 1);
        for (int i = 0; i < P::kStages; ++i) {
            mbar_init(bar.kv_full + i, 1);
            mbar_init(bar.kv_empty + i, 2);   // one share per query tile
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar.s_full + i, 1);
            mbar_init(bar.s_free + i, kCtas * 4);   // one arrival per softmax warp of the query tile
            mbar_init(bar.p_full + i, kCtas * 4);
            mbar_init(bar.pv_done + i, 1);
        }
        mbar_init(bar.drain, 1);
        *abort_flag = 0;
        // A CTA that starts after another one has reported a failure does nothing; in a pair the first decides for both.
        if (!kPair || rank == 0) *failed_before = *reinterpret_cast<volatile int *>(status) != 0;
        fence_barrier_init();
    }
    // The peer's barriers exist and its shared memory may be written from here on.
    sync_all();
    if constexpr (kPair) {
        if (threadIdx.x == 0 && rank == 0)
            st_cluster_u32(mapa(smem_u32(const_cast<int *>(failed_before)), 1), (uint32_t)*failed_before);
        cluster_sync_all();
    }
    if (*failed_before) return;
    if (warp == kMmaWarp) {
        if constexpr (kPair) {
            tmem_alloc_pair(tmem_base_slot, 512);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(tmem_base_slot, 512);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    sync_all();   // (both CTAs of a pair hold their tensor memory before its first instruction)
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_base_slot, 0);
    // a role that gives up tells the other CTA, whose waits would otherwise run to their own limit
    auto tell_peer = [&]() { st_cluster_u32(mapa(smem_u32(const_cast<int *>(abort_flag)), peer), 1u); };

    // Registers move from the last four warps to the softmax warps, whose threads hold a row of S (per scheduler: 2 x 208 + 88
    // registers for its three warps, of the 3 x 168 that the CTA was launched with).
    if (warp >= kProducerWarp) {
        reg_dec<88>();
        if (warp == kProducerWarp) {
            // With topk = chunk every token is selected and the compacted arrays would be copies of K / V: the salient
            // prefix is then read from K / V themselves (tm_ksel / tm_vsel alias tm_k / tm_v).
            const int kv_row0 = (b * Hkv + kvh) * N;
            if (lane == 0)
                producer_role<D, kPair>(st, bar, smem, rank, tm_q, tm_k, tm_v, tm_ksel, tm_vsel, bh * N + R0, kv_row0,
                                        sel_identity ? kv_row0 : bh * sel_rows, abort_flag, status, tell_peer);
        } else if (warp == kMmaWarp && rank == 0) {
            mma_role<D, kPair>(st, bar, smem, tmem_base, abort_flag, status, tell_peer);
        }
    } else {
        reg_inc<208>();
        const int x = warp >> 2;                       // 0: tile A, 1: tile B
        softmax_role<D, kPair>(st, bar, x, R0 + (x * kCtas + (int)rank) * kBlockM, tmem_base, abort_flag, status,
                                               smem + P::kQ + x * P::kQTile, y_part, d_part, n_parts, (long long)n_heads * N * D, (long long)n_heads * N, Y, bh, N,
                                               C, lam, budget, scale_log2);
        if constexpr (kPair) {
            if (*abort_flag) tell_peer();
        }
    }
    // (Of a pair nobody touches the peer's shared memory or tensor memory after this point.)
    tc_fence_before();
    sync_all();
    if (warp == kMmaWarp) {
        tc_fence_after();
        if constexpr (kPair) tmem_dealloc_pair(tmem_base, 512);
        else tmem_dealloc(tmem_base, 512);
    }
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
sa_merge_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                   const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_ksel,
                   const __grid_constant__ CUtensorMap tm_vsel, const __nv_bfloat16 *y_part, const float *d_part, int n_parts,
                   __nv_bfloat16 *Y, int *status, int H, int Hkv, int N, int C, int lam, int budget, int sel_rows, int sel_identity,
                   float scale_log2, int n_blocks, int n_heads, int set_heads) {
    grid_dep_wait();
    grid_dep_launch();
    attention_body<D, false>(tm_q, tm_k, tm_v, tm_ksel, tm_vsel, y_part, d_part, n_parts, Y, status, H, Hkv, N, C, lam, budget, sel_rows,
                             sel_identity, scale_log2, n_blocks, n_heads, set_heads);
}

// The same branch on CTA pairs (head dim 128): two CTAs of a cluster work on 512 consecutive query rows of
// one (batch, head) with UMMAs of the cta_group::2 form.  Query tile X of the pair is 256 rows -- rows
// [R0 + 256 X + 128 r, + 128) belong to the CTA of cluster rank r -- and one instruction, issued by a thread
// of rank 0, computes S_X = Q_X K^T (or O_X += P_X V) for both CTAs.  Each CTA keeps only its half of every
// key tile in shared memory: 64 of the 128 keys of K (the B operand of Q K^T is split along N) and 64 of the
// 128 value columns of V (likewise for P V); the tensor cores of both SMs read both halves.  Per FLOP a CTA
// therefore pulls half the K / V bytes from L2 and reads a quarter less shared memory than a CTA working
// alone.
//
// Who signals whom.  K / V / Q tiles: every CTA loads its halves into its own shared memory with plain TMA
// loads (no multicast) whose byte counts complete on the full-barriers of rank 0, where the issuing thread
// waits.  S_X ready, P_X V done: one tcgen05.commit arrives on the barrier of both CTAs.  S_X read, P_X written: the
// softmax warps of both CTAs arrive on rank 0's barriers.  Ring stages are released locally: what a CTA's softmax
// warps see completed has completed in both CTAs.
template <int D>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
sa_merge_pair_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                     const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_ksel,
                     const __grid_constant__ CUtensorMap tm_vsel, const __nv_bfloat16 *y_part, const float *d_part, int n_parts,
                     __nv_bfloat16 *Y, int *status, int H, int Hkv, int N, int C, int lam, int budget, int sel_rows, int sel_identity,
                     float scale_log2, int n_blocks, int n_heads, int set_heads) {
    grid_dep_wait();
    grid_dep_launch();
    attention_body<D, true>(tm_q, tm_k, tm_v, tm_ksel, tm_vsel, y_part, d_part, n_parts, Y, status, H, Hkv, N, C, lam, budget, sel_rows,
                            sel_identity, scale_log2, n_blocks, n_heads, set_heads);
}

// ---------------------------------------------------------------------------
// Self-Saliency Score (Sec. 3.1; Algorithm 1 "Compute Self-Saliency Score") and
// per-chunk top-k (Sec. 3.3, delayed selection) on tensor cores.
// One CTA scores 128 consecutive query rows of one (batch, head): one UMMA of
// shape 128 x 256 x d gives the logits of those rows against the 256 keys at
// positions [R0-128, R0+128) -- s_prev and s_in of Algorithm 1 side by side.  A
// thread owns one row; its window is the last C keys up to itself, i.e. the
// elements j in [lane+1, lane+C] of the C+32 columns its warp reads from TMEM
// (element lane+C is the token itself).  With e_j = exp(l_j - max), Z = sum e_j,
// Z' = sum_{j != t} e_j:  a_diag_j = e_j / Z,  a_nodiag_j = e_j / Z' (0 at j = t),
// Score = sum_j a_diag_j log((a_diag_j + eps) / (a_nodiag_j + eps)).
// The kernel is persistent: a CTA (one per SM) walks over tiles n = blockIdx.x, blockIdx.x + gridDim.x, ...
// (tile n = head n / n_row_blocks, rows 128 (n % n_row_blocks) ...) with two stages of shared memory and two
// TMEM accumulators, so that the loads of tile n+1 and its UMMA run under the row epilogue of tile n.
// The row's epilogue bounds it: three special-function instructions per window element (one 2^x, two logarithms) against
// six or seven others, by eight warps an SM, two tiles at a time (d = 128, C = 64: special-function unit 53 % busy, issue slots
// 38 %, DRAM 38 %; C = 128: 61, 37 and 24 %).  2 x 32 heads x 32768 tokens, d = 128, C = 64: 199 us, 4 x 32 x 4096, d = 64: 51 us,
// 32 x 131072, d = 128, C = 128: 650 us (with a threshold per token in the ranking, see below: 223, 58 and 825; with scalar
// arithmetic, logarithms for subnormal arguments, and for C = 128 a second set of exponentials as well: 325 to 368, 83 and 1030).
// Warps: 0 TMA producer, 1 MMA issuer, 2-5 score group 0 (even tiles of the CTA), 6-9 score group 1 (odd
// tiles); TMEM lane quarter = warp % 4.
// ---------------------------------------------------------------------------
template <int D>
struct ScoreSmem {
    static constexpr int kQBytes = kBlockM * D * 2, kKBytes = 2 * kBlockN * D * 2;
    static constexpr int kStage = kQBytes + kKBytes;
    static constexpr int kBar = 2 * kStage;          // full[2], mma_done[2], smem_free[2], tmem_free[2]
    static constexpr int kMisc = kBar + 8 * 8;       // tmem base, abort flag
    static constexpr int kSc = kMisc + 16;           // [2][128] ranking keys of the group's tile (16-byte aligned)
    static constexpr int kBallot = kSc + 2 * kBlockM * 4;   // [2][4]
    static constexpr int kTotal = kBallot + 2 * 4 * 4;
    static constexpr int kAlloc = kTotal + 1024;     // slack to align the base to 1024
};

static_assert(ScoreSmem<64>::kAlloc <= kMaxDynamicSmem && ScoreSmem<128>::kAlloc <= kMaxDynamicSmem,
              "score kernel: two stages must fit one CTA's shared memory");

// log2 of a positive number.  The general form costs four instructions more to scale subnormal arguments; they cannot
// occur when eps, which every argument contains, is a normal number.
template <bool kTiny>
__device__ __forceinline__ float log2_of(float x) {
    if constexpr (kTiny) return __log2f(x);
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int D, int C, bool kTinyEps>
__global__ void __launch_bounds__(320, 1)
score_select_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                       float *scores, int32_t *sel_idx, int *status, int H, int Hkv,
                       int N, int lam, float scale_log2, float eps, int n_row_blocks, int n_tiles) {
    grid_dep_wait();
    grid_dep_launch();
    clear_status(status);
    using P = ScoreSmem<D>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + P::kBar);
    uint64_t *mma_done = full + 2, *smem_free = full + 4, *tmem_free = full + 6;
    uint32_t *tmem_base_slot = reinterpret_cast<uint32_t *>(smem + P::kMisc);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + P::kMisc + 8);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int Tn = (N + C - 1) / C;

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(full + s, 1);
            mbar_init(mma_done + s, 1);
            mbar_init(smem_free + s, 1);
            mbar_init(tmem_free + s, 4);   // one arrival per warp of the score group
        }
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
    const uint32_t tmem_base = *tmem_base_slot;

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            for (int n = blockIdx.x; n < n_tiles; n += gridDim.x, ++it) {
                const int s = it & 1, ph = (it >> 1) & 1;
                if (!mbar_wait(smem_free + s, ph ^ 1, abort_flag, status, 22)) break;
                const int bh = n / n_row_blocks, R0 = (n - bh * n_row_blocks) * kBlockM;
                const int b = bh / H, h = bh - b * H, kvh = h / (H / Hkv);
                uint8_t *q_s = smem + s * P::kStage, *k_s = q_s + P::kQBytes;
                mbar_expect_tx(full + s, P::kQBytes + P::kKBytes);
                // rows before the start of K or of the previous head are masked by position in the epilogue
                const int k_row = (b * Hkv + kvh) * N + R0 - kBlockN;
                for (int half = 0; half < D / 64; ++half) {
                    tma_load_2d(q_s + half * (kBlockM * 128), &tm_q, full + s, half * 64, bh * N + R0);
                    // K-major operand of 256 rows: per 64-column half, rows 0..255 contiguous
                    tma_load_2d(k_s + half * (2 * kBlockN * 128), &tm_k, full + s, half * 64, k_row);
                    tma_load_2d(k_s + half * (2 * kBlockN * 128) + kBlockN * 128, &tm_k, full + s, half * 64, k_row + kBlockN);
                }
            }
            mbar_drain_ring(full, 2, it, clock64());
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = make_idesc(kBlockM, 2 * kBlockN, false);
            int it = 0;
            bool ok = true;
            for (int n = blockIdx.x; n < n_tiles; n += gridDim.x, ++it) {
                const int s = it & 1, ph = (it >> 1) & 1;
                ok = mbar_wait(full + s, ph, abort_flag, status, 20) &&
                     mbar_wait(tmem_free + s, ph ^ 1, abort_flag, status, 23);
                if (!ok) break;
                tc_fence_after();
                const uint32_t q_a = smem_u32(smem + s * P::kStage), k_a = q_a + P::kQBytes;
#pragma unroll
                for (int k = 0; k < D / 16; ++k) {
                    const uint32_t qa = q_a + (k / 4) * (kBlockM * 128) + (k % 4) * 32;
                    const uint32_t ka = k_a + (k / 4) * (2 * kBlockN * 128) + (k % 4) * 32;
                    mma_ss(tmem_base + s * 256, smem_desc(qa, 0), smem_desc(ka, 0), idesc, k > 0 ? 1u : 0u);
                }
                tc_commit(mma_done + s);
            }
            // no MMA may still be running when tensor memory is freed: after a failure wait (bounded) for the
            // last group issued (its commit covers everything before it)
            if (!ok && it > 0) mbar_wait_drain(mma_done + ((it - 1) & 1), ((it - 1) >> 1) & 1);
        }
    } else {
        const int g = (warp - 2) >> 2;                 // score group = stage = TMEM accumulator
        const int wq = warp & 3;                       // TMEM lane quarter this warp may read
        const int r = wq * 32 + lane;                  // row of the tile owned by this thread
        int *keys = reinterpret_cast<int *>(smem + P::kSc) + g * kBlockM;
        uint32_t *ballots = reinterpret_cast<uint32_t *>(smem + P::kBallot) + g * 4;
        const uint32_t taddr = tmem_base + g * 256 + ((uint32_t)(wq * 32) << 16) + (uint32_t)(wq * 32 + kBlockN - C);
        const int group_bar = 1 + g;
        int it = g, j = 0;
        for (int n = blockIdx.x + g * gridDim.x; n < n_tiles; n += 2 * gridDim.x, it += 2, ++j) {
            const int ph = j & 1;
            const int bh = n / n_row_blocks, R0 = (n - bh * n_row_blocks) * kBlockM;
            const int t = R0 + r;
            bool ok = mbar_wait(mma_done + g, ph, abort_flag, status, 21);
            // the group leaves the loop together
            {
                uint32_t all_ok;
                asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 p, %1, 0;\nbarrier.cta.red.and.pred q, %2, 128, p;\nselp.b32 %0, 1, 0, q;\n}"
                             : "=r"(all_ok) : "r"((uint32_t)ok), "r"(group_bar) : "memory");
                ok = all_ok != 0;
            }
            if (!ok) break;
            tc_fence_after();
            if (r == 0) mbar_arrive(smem_free + g);    // the logits are complete: the stage's operands are free
            float score = 0.f;
            {
                // Element j of the warp's C+32 columns is the key at position R0 + 32 wq - C + j, and the window of
                // the row in lane l is j in [l+1, l+C].  Columns [32, C) lie in every lane's window; of columns jj
                // and C + jj (jj < 32) exactly one does (the first if jj > l).  So the first and the last block of
                // 32 columns fold into one, and a row becomes C values without gaps: block 0 is the folded one (the
                // token itself sits at jj = l), blocks 1 .. C/32-1 are columns [32 q, 32 q + 32).  Keys at negative
                // positions (first tile of a sequence only) are set to -inf, which the exponential turns into 0.
                constexpr int kBlocks = C / 32;
                const bool first_tile = R0 == 0;
                auto load_block = [&](int q, uint32_t (&v)[32]) {
                    tmem_ld32(taddr + q * 32, v);
                    if (q == 0) {
                        uint32_t w[32];
                        tmem_ld32(taddr + C, w);
                        tmem_wait_ld();
#pragma unroll
                        for (int jj = 0; jj < 32; ++jj) v[jj] = (jj > lane) ? v[jj] : w[jj];
                    } else {
                        tmem_wait_ld();
                    }
                    if (first_tile) {
                        const int n_neg = C - wq * 32;   // columns below n_neg are before the start of the sequence
#pragma unroll
                        for (int jj = 0; jj < 32; ++jj)
                            if (q * 32 + jj < n_neg && (q > 0 || jj > lane)) v[jj] = 0xff800000u;
                    }
                };
                auto tmem_read_done = [&]() {   // the accumulator may be overwritten by the UMMA of the tile after next
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tmem_free + g);
                };
                // The row is held in registers (C values; at C = 128 some 50 bytes of a thread's spill): one read of tensor
                // memory, exponentials kept in place.
                uint32_t v[kBlocks][32];
#pragma unroll
                for (int q = 0; q < kBlocks; ++q) load_block(q, v[q]);
                tmem_read_done();
                float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                for (int q = 0; q < kBlocks; ++q)
#pragma unroll
                    for (int jj = 0; jj < 32; jj += 2)
                        mx[(jj >> 1) & 3] = max3(mx[(jj >> 1) & 3], __uint_as_float(v[q][jj]), __uint_as_float(v[q][jj + 1]));
                const float neg_m = -fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * scale_log2;
                const float2 scale2 = make_float2(scale_log2, scale_log2), negm2 = make_float2(neg_m, neg_m);
                // e_j; the token's own (jj = lane of block 0) is taken out of the row, so that the sum without it is formed
                // directly and the terms below need no case for it
                float2 z2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                float e_self = 0.f;
#pragma unroll
                for (int q = 0; q < kBlocks; ++q)
#pragma unroll
                    for (int jj = 0; jj < 32; jj += 2) {
                        const float2 x = __ffma2_rn(make_float2(__uint_as_float(v[q][jj]), __uint_as_float(v[q][jj + 1])), scale2, negm2);
                        float2 e = make_float2(ex2(x.x), ex2(x.y));
                        if (q == 0) {
                            if (jj == lane) { e_self = e.x; e.x = 0.f; }
                            if (jj + 1 == lane) { e_self = e.y; e.y = 0.f; }
                        }
                        z2[(jj >> 1) & 1] = __fadd2_rn(z2[(jj >> 1) & 1], e);
                        v[q][jj] = __float_as_uint(e.x);
                        v[q][jj + 1] = __float_as_uint(e.y);
                    }
                const float z_nd = (z2[0].x + z2[0].y) + (z2[1].x + z2[1].y), z_all = z_nd + e_self;
                const float inv_all = 1.f / z_all, inv_nd = z_nd > 0.f ? 1.f / z_nd : 0.f;
                const float2 ia2 = make_float2(inv_all, inv_all), in2 = make_float2(inv_nd, inv_nd), eps2 = make_float2(eps, eps);
                const float2 minus2 = make_float2(-1.f, -1.f);
                float2 s2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
                for (int q = 0; q < kBlocks; ++q)
#pragma unroll
                    for (int jj = 0; jj < 32; jj += 2) {
                        // a log2((a + eps) / (b + eps)) without the factor 1 / Z; a masked key has e = 0 and adds nothing
                        const float2 e = make_float2(__uint_as_float(v[q][jj]), __uint_as_float(v[q][jj + 1]));
                        const float2 a = __ffma2_rn(e, ia2, eps2), bb = __ffma2_rn(e, in2, eps2);
                        const float2 la = make_float2(log2_of<kTinyEps>(a.x), log2_of<kTinyEps>(a.y));
                        const float2 lb = make_float2(log2_of<kTinyEps>(bb.x), log2_of<kTinyEps>(bb.y));
                        s2[(jj >> 1) & 1] = __ffma2_rn(e, __ffma2_rn(lb, minus2, la), s2[(jj >> 1) & 1]);
                    }
                const float a_self = e_self * inv_all;
                score = ((s2[0].x + s2[0].y) + (s2[1].x + s2[1].y)) * inv_all +
                        a_self * (log2_of<kTinyEps>(a_self + eps) - log2_of<kTinyEps>(eps));
                score *= 0.6931471805599453f;
            }
            // the score as an integer of the same order (NaN as -inf, -0 as 0): one comparison ranks two tokens
            const int bits = __float_as_int(isnan(score) ? -INFINITY : score + 0.f);
            const int key = bits ^ ((bits >> 31) & 0x7fffffff);
            keys[r] = t < N ? key : INT_MIN;   // (below the key of -inf)
            if (t < N && scores != nullptr) scores[(long long)bh * N + t] = score;
            asm volatile("bar.sync %0, 128;" ::"r"(group_bar) : "memory");
            if (lam > 0) {
                // top-k of each chunk of the tile: rank under (score descending, position ascending)
                const int cc = r / C, rr = r - cc * C;
                const int n_c = min(C, N - (R0 + cc * C));   // tokens of this row's chunk (<= 0: past the end)
                bool selected = false;
                // Tokens before this one outrank it with an equal key.  In the blocks of 32 tokens before the warp's own that is
                // a comparison with key - 1; in its own the equal keys of lower lanes are counted by one match.  A ragged
                // chunk's missing tokens rank below all.  (With a threshold chosen per token the ranking took 1750 of a tile's
                // 7500 cycles.)
                const uint32_t equal = __match_any_sync(0xffffffffu, keys[r]);
                if (rr < n_c) {
                    int rank = __popc(equal & ((1u << lane) - 1u));
#pragma unroll
                    for (int q = 0; q < C / 32; ++q) {
                        const int thr = q < (rr >> 5) ? key - 1 : key;
#pragma unroll
                        for (int j4 = 0; j4 < 8; ++j4) {
                            const int4 o = *reinterpret_cast<const int4 *>(keys + cc * C + q * 32 + j4 * 4);
                            rank += (o.x > thr ? 1 : 0) + (o.y > thr ? 1 : 0) + (o.z > thr ? 1 : 0) + (o.w > thr ? 1 : 0);
                        }
                    }
                    selected = rank < lam;
                }
                // place of a selected row in the ascending output = selected rows before it in its chunk
                const uint32_t votes = __ballot_sync(0xffffffffu, selected);
                if (lane == 0) ballots[wq] = votes;
                asm volatile("bar.sync %0, 128;" ::"r"(group_bar) : "memory");
                if (n_c > 0) {
                    int32_t *out = sel_idx + ((long long)bh * Tn + (R0 / C + cc)) * lam;
                    int before = __popc(votes & ((1u << lane) - 1u));
                    for (int w = cc * (C / 32); w < wq; ++w) before += __popc(ballots[w]);
                    if (selected) out[before] = R0 + cc * C + rr;
                    const int n_sel = n_c < lam ? n_c : lam;
                    if (rr >= n_sel && rr < lam) out[rr] = -1;
                }
            }
            // keys / ballots are written again in the group's next tile
            asm volatile("bar.sync %0, 128;" ::"r"(group_bar) : "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// K_sel / V_sel [B*H, sel_rows, d]: row j < n_valid is row sel_idx[j] of the head's K / V
// (a -1 entry, or a row of the padding, is zero).  One warp per row.
template <int D>
__global__ void __launch_bounds__(256)
compact_kernel(const __nv_bfloat16 *K, const __nv_bfloat16 *V,
               const int32_t *sel_idx, __nv_bfloat16 *Ksel,
               __nv_bfloat16 *Vsel, int H, int Hkv, long long N, long long n_idx, long long sel_rows) {
    grid_dep_wait();
    grid_dep_launch();
    const int bh = blockIdx.y, b = bh / H, h = bh % H, kvh = h / (H / Hkv);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long j = (long long)blockIdx.x * 8 + warp;
    if (j >= sel_rows) return;
    long long p = -1;
    if (j < n_idx) p = sel_idx[(long long)bh * n_idx + j];
    constexpr int kVec = D / 8;  // uint4 per row
    uint4 kk = make_uint4(0, 0, 0, 0), vv = kk;
    if (lane < kVec && p >= 0) {
        kk = reinterpret_cast<const uint4 *>(K + (((long long)b * Hkv + kvh) * N + p) * D)[lane];
        vv = reinterpret_cast<const uint4 *>(V + (((long long)b * Hkv + kvh) * N + p) * D)[lane];
    }
    if (lane < kVec) {
        reinterpret_cast<uint4 *>(Ksel + ((long long)bh * sel_rows + j) * D)[lane] = kk;
        reinterpret_cast<uint4 *>(Vsel + ((long long)bh * sel_rows + j) * D)[lane] = vv;
    }
}

// The bounded wait of the kernels above, alone: one warp, one mbarrier that expects an arrival which never
// comes.  No TMA, no tensor memory, no MMA: when the limit has passed the kernel records the timeout and ends.
__global__ void wait_timeout_selftest_kernel(int *status, long long limit_cycles) {
    __shared__ uint64_t bar;
    __shared__ int abort_word;
    volatile int *abort_flag = &abort_word;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) (void)mbar_wait_limit(&bar, 0, abort_flag, status, 99, limit_cycles);
    __syncthreads();
}

// ----------------------------------------------------------------- host side

// 2-D bf16 tensor [rows, d] tiled in boxes of [128 rows, 64 columns] with 128-byte swizzle.
bool make_map(CUtensorMap *m, const void *base, unsigned long long rows, int d) {
    return make_map_2d(m, base, rows, (unsigned long long)d, 128, false);
}

int set_of_heads(long long n_heads, int rep, long long bytes_per_head) {   // see row_block
    const long long fit = std::max<long long>(1, (64ll << 20) / (bytes_per_head * rep)) * rep;   // whole KV groups
    return (int)std::min(n_heads, fit);
}

template <int D>
int launch_tc(const still_params_t *p, long long N, const void *Q, const void *K, const void *V,
              const int32_t *sel_idx, const void *y_part, const float *d_part, int n_parts, void *Y, void *k_sel, void *v_sel,
              long long sel_rows, bool compact, int *status, cudaStream_t st, int *launches) {
    using bf = __nv_bfloat16;
    const long long T = (N + p->chunk - 1) / p->chunk, BH = (long long)p->B * p->H;
    const long long n_idx = T * p->topk;
    const bool identity = p->topk == p->chunk;  // the selection of every chunk is the chunk itself
    if (!identity && compact) {
        dim3 grid((unsigned)((sel_rows + 7) / 8), (unsigned)BH);
        if (launch_dependent(compact_kernel<D>, grid, dim3(256), 0, st, (const bf *)K, (const bf *)V, sel_idx, (bf *)k_sel, (bf *)v_sel,
                             p->H, p->Hkv, N, n_idx, sel_rows) != cudaSuccess)
            return STILL_ERR_CUDA;
        ++*launches;
    }
    const unsigned long long kv_rows = (unsigned long long)p->B * p->Hkv * N;
    const unsigned long long sel_total = identity ? kv_rows : (unsigned long long)BH * sel_rows;
    constexpr bool kPair = D == 128;   // head dim 128 runs on CTA pairs, each CTA holding 64 keys of a K tile
    CUtensorMap tq, tk, tv, tks, tvs;
    if (!make_map(&tq, Q, (unsigned long long)BH * N, D) ||
        !make_map_2d(&tk, K, kv_rows, D, kPair ? kBlockN / 2 : kBlockN, false) || !make_map(&tv, V, kv_rows, D) ||
        !make_map_2d(&tks, identity ? K : k_sel, sel_total, D, kPair ? kBlockN / 2 : kBlockN, false) ||
        !make_map(&tvs, identity ? V : v_sel, sel_total, D))
        return STILL_ERR_CUDA;
    const float scale_log2 = p->sm_scale * 1.4426950408889634f;
    const int rep = p->H / p->Hkv;
    const int set_heads = set_of_heads(BH, rep, ((identity ? 0 : sel_rows) + N / rep + 1) * D * 4);
    if constexpr (kPair) {
        const int n_pairs = (int)((N + 4 * kBlockM - 1) / (4 * kBlockM));
        if (ensure_dynamic_smem((const void *)sa_merge_pair_kernel<D>, (AttnPlan<D, true>::kAlloc)) != cudaSuccess) return STILL_ERR_CUDA;
        dim3 grid((unsigned)(2 * n_pairs * BH));   // clusters of two
        profile_mark_begin(st);
        const cudaError_t e = launch_dependent(sa_merge_pair_kernel<D>, grid, dim3(kThreads), (AttnPlan<D, true>::kAlloc), st,
            tq, tk, tv, tks, tvs, (const bf *)y_part, d_part, n_parts, (bf *)Y, status, p->H, p->Hkv, (int)N, p->chunk, p->topk, (int)p->max_salient, (int)sel_rows,
            identity ? 1 : 0, scale_log2, n_pairs, (int)BH, set_heads);
        profile_mark_end(st);
        if (e != cudaSuccess) return STILL_ERR_CUDA;
    } else {
        const int n_qblocks = (int)((N + 2 * kBlockM - 1) / (2 * kBlockM));
        if (ensure_dynamic_smem((const void *)sa_merge_tc_kernel<D>, (AttnPlan<D, false>::kAlloc)) != cudaSuccess) return STILL_ERR_CUDA;
        dim3 grid((unsigned)(n_qblocks * BH));
        profile_mark_begin(st);
        const cudaError_t e = launch_dependent(sa_merge_tc_kernel<D>, grid, dim3(kThreads), (AttnPlan<D, false>::kAlloc), st,
            tq, tk, tv, tks, tvs, (const bf *)y_part, d_part, n_parts, (bf *)Y, status, p->H, p->Hkv, (int)N, p->chunk, p->topk, (int)p->max_salient, (int)sel_rows,
            identity ? 1 : 0, scale_log2, n_qblocks, (int)BH, set_heads);
        profile_mark_end(st);
        if (e != cudaSuccess) return STILL_ERR_CUDA;
    }
    ++*launches;
    if (cudaGetLastError() != cudaSuccess) return STILL_ERR_CUDA;
    return STILL_OK;
}

template <int D, int C>
int launch_score_tc(const still_params_t *p, long long N, const void *Q, const void *K, float *scores,
                    int32_t *sel_idx, int *status, cudaStream_t st, int *launches) {
    CUtensorMap tq, tk;
    const long long BH = (long long)p->B * p->H;
    if (!make_map(&tq, Q, (unsigned long long)BH * N, D) ||
        !make_map(&tk, K, (unsigned long long)p->B * p->Hkv * N, D))
        return STILL_ERR_CUDA;
    constexpr int kSmem = ScoreSmem<D>::kAlloc;
    const auto kernel = p->eps < 1.17549435e-38f ? score_select_tc_kernel<D, C, true> : score_select_tc_kernel<D, C, false>;
    if (ensure_dynamic_smem((const void *)kernel, kSmem) != cudaSuccess) return STILL_ERR_CUDA;
    int dev = 0, n_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n_sm <= 0)
        return STILL_ERR_CUDA;
    const long long n_row_blocks = (N + kBlockM - 1) / kBlockM, n_tiles = n_row_blocks * BH;
    if (n_tiles >= (1ll << 31)) return STILL_ERR_UNSUPPORTED;
    const unsigned grid = (unsigned)std::min<long long>(n_tiles, n_sm);   // one persistent CTA per SM
    if (launch_dependent(kernel, dim3(grid), dim3(320), kSmem, st, tq, tk, scores, sel_idx, status, p->H, p->Hkv, (int)N, p->topk,
                         p->sm_scale * 1.4426950408889634f, p->eps, (int)n_row_blocks, (int)n_tiles) != cudaSuccess)
        return STILL_ERR_CUDA;
    ++*launches;
    return STILL_OK;
}

}  // namespace

int tc_score_select(const still_params_t *p, long long N, const void *Q, const void *K, float *scores,
                    int32_t *sel_idx, int *status_words, cudaStream_t st, int *launches) {
    if ((long long)p->B * p->H * N >= (1ll << 31)) return STILL_ERR_UNSUPPORTED;
    if (p->d == 64 && p->chunk == 64) return launch_score_tc<64, 64>(p, N, Q, K, scores, sel_idx, status_words, st, launches);
    if (p->d == 64 && p->chunk == 128) return launch_score_tc<64, 128>(p, N, Q, K, scores, sel_idx, status_words, st, launches);
    if (p->d == 128 && p->chunk == 64) return launch_score_tc<128, 64>(p, N, Q, K, scores, sel_idx, status_words, st, launches);
    return launch_score_tc<128, 128>(p, N, Q, K, scores, sel_idx, status_words, st, launches);
}

// N_LA / D_LA of the fp32-accumulating FMA kernels as one bf16 part: y = N_LA / D_LA, d = D_LA.
__global__ void la_to_part_kernel(const float *N_LA, const float *D_LA, __nv_bfloat16 *y,
                                  float *dp, long long rows, int d) {
    grid_dep_wait();
    grid_dep_launch();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * d) return;
    const long long r = i / d;
    const float dd = D_LA[r];
    y[i] = __float2bfloat16_rn(dd > 0.f ? N_LA[i] / dd : 0.f);
    if (i == r * d) dp[r] = dd;
}

int tc_la_to_part(const float *N_LA, const float *D_LA, void *y_part, float *d_part, long long rows, int d, cudaStream_t st,
                  int *launches) {
    const long long n = rows * d;
    ++*launches;
    return launch_dependent(la_to_part_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, N_LA, D_LA, (__nv_bfloat16 *)y_part,
                            d_part, rows, d) == cudaSuccess ? STILL_OK : STILL_ERR_CUDA;
}

int tc_selftest_wait_timeout(int *status_words, long long limit_cycles, cudaStream_t st) {
    wait_timeout_selftest_kernel<<<1, 32, 0, st>>>(status_words, limit_cycles);
    return cudaGetLastError() == cudaSuccess ? STILL_OK : STILL_ERR_CUDA;
}

bool tc_supported(const still_params_t *p) {
    return p->dtype == STILL_DTYPE_BF16 && (p->d == 64 || p->d == 128) && (p->chunk == 64 || p->chunk == 128);
}

long long tc_sel_rows(const still_params_t *p, long long N) {
    const long long T = (N + p->chunk - 1) / p->chunk;
    return (T * p->topk + kBlockN - 1) / kBlockN * kBlockN + kBlockN;
}

int tc_sa_merge(const still_params_t *p, long long N, const void *Q, const void *K, const void *V,
                const int32_t *sel_idx, const void *y_part, const float *d_part, int n_parts, void *Y, void *k_sel, void *v_sel,
                long long sel_rows, bool compact, int *status_words, cudaStream_t st, int *launches) {
    if ((long long)p->B * p->H * std::max(N, sel_rows) >= (1ll << 31)) return STILL_ERR_UNSUPPORTED;  // TMA row coordinate
    if (p->d == 64)
        return launch_tc<64>(p, N, Q, K, V, sel_idx, y_part, d_part, n_parts, Y, k_sel, v_sel, sel_rows, compact, status_words, st, launches);
    return launch_tc<128>(p, N, Q, K, V, sel_idx, y_part, d_part, n_parts, Y, k_sel, v_sel, sel_rows, compact, status_words, st, launches);
}

}  // namespace still
