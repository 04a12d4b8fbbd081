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
// An item is 256 consecutive query rows of one (batch, head), for a pair of CTAs 512: two query tiles A and B of 128
// (256) rows.  CTAs stay and take one item after the other (Work).  The keys of an item come as a stream of 128-key
// tiles: SEL tiles j (rows [128j, 128j+128) of K_sel / V_sel), and the LOC tiles around the rows (rows of K / V at
// positions [128m, 128m+128)).  First the SEL tiles that both query tiles see (before them what has already left the window of B), then what only one of them sees, by turns.  Which
// columns of a tile a query row sees is a per-row column interval, applied as a mask in the softmax.
//
// Warp roles (384 threads):
//   warps 0-7  softmax, four warps per query tile, one thread per query row (tcgen05.ld of the S row): online softmax in
//              the log2 domain with lazy rescaling of O, P to TMEM as bf16; then the epilogue: O / l merged with the
//              linear branch (N_LA, D_LA) under one denominator and left in shared memory as bf16
//   warp 8     TMA producer: Q tiles of an item, then K and V tiles and the linear branch's results through one ring
//   warp 9     MMA issuer (one elected thread): S = Q_X K^T (operands in shared memory, SWIZZLE_128B K-major),
//              O_X += P_X V (P_X read from TMEM, V in shared memory MN-major)
//   warps 10, 11  output: the rows of query tile A, of B, to memory by TMA
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
    static constexpr int kStage = kKTile + kVTile;
    // The output of a query tile leaves through stages of the ring (entries behind the item's keys), which the linear
    // branch's partial results come in by: at D = 128 a stage a part, at D = 64 both parts in one.
    static constexpr int kPartTile = kBlockM * D * 2, kPartsPerStage = kStage / kPartTile;
    static constexpr int kQ = 0;
    static constexpr int kK = kQ + 2 * kQTile;                 // stage s at kK + s kStage: its K tile, then its V tile
    static constexpr int kV = kK + kKTile;
    static constexpr int kBar = kK + kStages * kStage;         // mbarriers
    static constexpr int kNumBars = 2 + 2 * kStages + 2 + 2 + 2 + 2 + 6 + 4 + 3;
    static constexpr int kMisc = kBar + kNumBars * 8;          // tmem base, abort flag, "a CTA has failed before", -, item[2][2]
    static constexpr int kTotal = kMisc + 32;
    static constexpr int kAlloc = kTotal + 1024;               // slack to align the base to 1024
    // entries of the ring that the output of a query tile takes
    __host__ __device__ static constexpr int y_entries(int n_parts) { return n_parts > kPartsPerStage ? 2 : 1; }
    static_assert(kPartsPerStage == (D == 64 ? 2 : 1) && kKTile == kVTile, "attention kernel: a stage holds both parts at D = 64, one at D = 128");
    static_assert(kAlloc <= kMaxDynamicSmem, "attention kernel: the shared-memory plan exceeds what a CTA can have");
    static_assert(kMisc % 8 == 0 && kKTile % 1024 == 0 && kVTile % 1024 == 0, "attention kernel: operand tiles are swizzle-aligned");
};

struct AttnBars {
    uint64_t *q_full, *q_empty;     // ... and the item's last Q K^T has completed
    uint64_t *kv_full, *kv_empty;   // [kStages]
    uint64_t *s_full;    // [2] S of query tile x is in tensor memory
    uint64_t *s_free;    // [2] ... and has been read
    uint64_t *p_full;    // [2] P_x is in tensor memory
    uint64_t *pv_done;   // [2] O_x includes the tile's product (and P_x may be overwritten)
    uint64_t *y_full;    // [2] the linear branch's results for query tile x are in their stages
    uint64_t *y_ready;   // [2] ... and the output is where the first of them were
    uint64_t *y_taken;   // [2] ... and the output warp has passed y_ready, as the softmax warps have y_full: the next may be announced
    uint64_t *item_full, *item_empty;   // [2] an item to come is there; ... and has been read
    uint64_t *first_done;   // [2] (of a pair's second CTA) the first CTA's producer is done with an item
    uint64_t *drain;     // MMA warp: everything issued has completed (failure path)
    template <class P>
    __device__ __forceinline__ static AttnBars at(uint8_t *smem, P) {
        AttnBars b;
        b.q_full = reinterpret_cast<uint64_t *>(smem + P::kBar);
        b.q_empty = b.q_full + 1;
        b.kv_full = b.q_empty + 1;
        b.kv_empty = b.kv_full + P::kStages;
        b.s_full = b.kv_empty + P::kStages;
        b.s_free = b.s_full + 2;
        b.p_full = b.s_free + 2;
        b.pv_done = b.p_full + 2;
        b.y_full = b.pv_done + 2;
        b.y_ready = b.y_full + 2;
        b.y_taken = b.y_ready + 2;
        b.item_full = b.y_taken + 2;
        b.item_empty = b.item_full + 2;
        b.first_done = b.item_empty + 2;
        b.drain = b.first_done + 2;
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
    __device__ __forceinline__ void skip(int n, int n_stages) {
        for (int i = 0; i < n; ++i) next(n_stages);
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
    // k-th tile of query tile x: a SEL tile, or a LOC tile?  Returns its number.
    __device__ __forceinline__ int tile_of(int x, int k, bool &sel) const {
        const int n = x ? n_sel_b : n_sel_a;
        sel = k < n;
        return k + (sel ? (x ? sel_b : sel_a) : (x ? loc_b : loc_a) - n);
    }
    // ... as its softmax warps need it
    struct Mine {
        int n, n_sel, sel0, loc0;   // tiles, SEL tiles; the first SEL tile, the first LOC tile
    };
    __device__ __forceinline__ Mine mine(int x) const {
        return x ? Mine{entries_of(1), n_sel_b, sel_b, loc_b} : Mine{entries_of(0), n_sel_a, sel_a, loc_a};
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

__device__ __forceinline__ int sel_limit(int pos, int log2_c, int lam) {  // end of the visible range of K_sel
    const int c = pos >> log2_c;
    return c >= 2 ? (c - 1) * lam : 0;
}
// Start of the visible range: 0, or with a salient-cache budget of `budget` tokens per head (a multiple of lam;
// the oldest cached tokens have left for the linear state) the last `budget` entries before the end.
__device__ __forceinline__ int sel_start(int limit, int budget) { return budget > 0 ? max(limit - budget, 0) : 0; }

// The key stream of the query tiles that start at rows R0 and R0 + rows, of `rows` (a multiple of 128) rows each.
__device__ __forceinline__ Stream make_stream(int R0, int rows, int N, int log2_c, int lam, int budget) {
    Stream st;
    const int last_m = (N - 1) / kBlockN, m_a = R0 / kBlockN, m_b = m_a + rows / kBlockN;
    const int last_a = min(R0 + rows, N) - 1, last_b = min(R0 + 2 * rows, N) - 1;
    // SEL tiles [a0, a1) and [b0, b1): a tile's first row sees the oldest entries, its last row the newest
    const int a0 = sel_start(sel_limit(R0, log2_c, lam), budget) / kBlockN, a1 = (sel_limit(last_a, log2_c, lam) + kBlockN - 1) / kBlockN;
    st.sel_a = a0;
    st.n_sel_a = max(a1 - a0, 0);
    st.loc_a = max(m_a - 1, 0);
    st.n_lead = st.n_shared = st.sel_b = st.n_sel_b = st.loc_b = st.n_b = 0;
    if (R0 + rows < N) {
        const int b0 = sel_start(sel_limit(R0 + rows, log2_c, lam), budget) / kBlockN, b1 = (sel_limit(last_b, log2_c, lam) + kBlockN - 1) / kBlockN;
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

// What an attention kernel works on, and how its roles come to it.  A CTA (or pair) stays for the whole kernel and takes one
// item (the rows of two query tiles of a head) after the other: the first by its own number, the others from a counter (of the
// workspace's status block, which the call's first kernel clears), so that whoever is done first takes the next.  The producer
// of the first CTA asks for an item with the last keys of the one before, and hands it to the other roles (of both CTAs) in one of
// two places.  (Asked for with the first keys, items were dealt out in the order in which their predecessors began, not ended: us a
// call, like that and like this, with a CTA per item 92, 62, 155: 8 heads x 5700 tokens, d = 128, C = 128, 96 items for 74 pairs, 111 and
// 94; 16 x 3000, d = 128, 96 items, 77 and 60; 4 x 12000, d = 64, 188 items for 148 CTAs, 186 and 156; every token kept.)
struct Work {
    int n_blocks, n_heads, set_heads, rep, N, log2_c, lam, budget, sel_rows, sel_identity, n_parts;
    int rows;          // of a query tile: 128 a CTA
    int first, total;
    volatile int *item;   // [2][2]: head (-1: there are no more) and first row
    int bh, R0;           // the current item
    __device__ __forceinline__ void set(int i) {
        int rb;
        row_block(i, n_blocks, n_heads, set_heads, rb, bh);
        R0 = rb * 2 * rows;
    }
    __device__ __forceinline__ Stream stream() const { return make_stream(R0, rows, N, log2_c, lam, budget); }
    __device__ __forceinline__ int n_query_tiles() const { return R0 + rows < N ? 2 : 1; }
};
// One thread's wait for the n-th of the items that were handed out (n from 0).  Returns whether there is one; `taken` tells that
// the warp has read it.
template <bool kPair>
__device__ __forceinline__ bool next_item(Work &w, const AttnBars &bar, int n, volatile int *abort_flag, int *status, bool &ok) {
    ok = mbar_wait(bar.item_full + (n & 1), (uint32_t)(n >> 1) & 1u, abort_flag, status, 13);
    if constexpr (kPair) mbar_acquire_cluster(bar.item_full + (n & 1), (uint32_t)(n >> 1) & 1u);
    w.bh = w.item[2 * (n & 1)];
    w.R0 = w.item[2 * (n & 1) + 1];
    return ok && w.bh >= 0;
}
template <bool kPair>
__device__ __forceinline__ void item_taken(const AttnBars &bar, int n) {
    if constexpr (kPair) mbar_arrive_cluster(mapa(smem_u32(bar.item_empty + (n & 1)), 0));
    else mbar_arrive(bar.item_empty + (n & 1));
}
// ... by a whole warp
template <bool kPair>
__device__ __forceinline__ bool next_item_of_warp(Work &w, const AttnBars &bar, int n, volatile int *abort_flag, int *status, bool &ok) {
    (void)next_item<kPair>(w, bar, n, abort_flag, status, ok);
    ok = __all_sync(0xffffffffu, ok);
    w.bh = __shfl_sync(0xffffffffu, w.bh, 0);   // (known to be the same in all lanes, and so is what follows from it)
    w.R0 = __shfl_sync(0xffffffffu, w.R0, 0);
    if (ok && (threadIdx.x & 31) == 0) item_taken<kPair>(bar, n);
    return ok && w.bh >= 0;
}

// The tensor maps of an attention kernel (p0, p1: the linear branch's partial results).
struct AttnMaps {
    CUtensorMap q, k, v, ksel, vsel, p0, p1, y;
};

// Rows t0 .. t0 + rows - 1 of a head, whose rows start at head0, from their place in an output's stage, by a warp.
template <int D>
__device__ __forceinline__ void store_rows(const uint8_t *tile, __nv_bfloat16 *Y, long long head0, int t0, int rows) {
    constexpr int kPieces = D / 8;
#pragma unroll 4
    for (int id = threadIdx.x & 31; id < rows * kPieces; id += 32) {
        const int row = id / kPieces, c = id % kPieces;
        *reinterpret_cast<uint4 *>(Y + (head0 + t0 + row) * D + c * 8) =
            *reinterpret_cast<const uint4 *>(tile + (c >> 3) * (kBlockM * 128) + row * 128 + (((c & 7) ^ (row & 7)) << 4));
    }
}

// ---------------------------------------------------------------------------
// Softmax warps of the attention kernels (one warpgroup per query tile, a thread per query row) and the merge epilogue.
// x is the query tile (0: A, 1: B), tile_row0 the position of the tile's first row, ring the key ring in shared memory.  The
// barriers are this CTA's, except that in a CTA pair what the issuing warp waits for is announced on the first CTA's.  One item:
// my is query tile x's view of the stream, y_stage the ring stage of its output, flip the parity of the tiles that query tile x
// has had in the items before, y_flip that of these items; ahead(last)
// is called while the last product runs and says whether the item is the CTA's last.  Returns whether all
// waits ended.
// ---------------------------------------------------------------------------
template <int D, bool kPair, class Ahead>
__device__ __forceinline__ bool softmax_role(const Stream::Mine my, const AttnBars &bar, const int x, const int tile_row0,
                                             const uint32_t tmem_base, volatile int *abort_flag, int *status,
                                             uint8_t *ring, const int y_stage, const int flip, const int y_flip,
                                             const float *d_part, const int n_parts, const long long part_stride_d, __nv_bfloat16 *Y,
                                             const int bh, const int N, const int log2_c, const int lam, const int budget,
                                             const float scale_log2, Ahead ahead) {
    using P = AttnPlan<D, kPair>;
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
    const int n_mine = my.n;
    bool ok = true;
    const uint32_t lane_addr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t s_addr = lane_addr + TmemPlan<D>::s(x), p_addr = lane_addr + TmemPlan<D>::p(x), o_addr = lane_addr + TmemPlan<D>::o(x);
    const int tq = min(t, N - 1);              // rows past N mimic the last row (never stored)
    const int lim_sel = sel_limit(tq, log2_c, lam), lo_sel = sel_start(lim_sel, budget);
    const int loc_lo = max((tq >> log2_c) - 1, 0) << log2_c;
    float m_used = -INFINITY, l_sum = 0.f;     // log2 domain
    // A wait can end in one lane and run out in another, and the warp has to stay together for the instructions that take
    // it whole.  So no wait is left by a branch: the loop runs out with whatever has been read (a wait gives up at once
    // where a role has given up before), and the warp votes behind it.  (A vote behind every wait took 0.6 % longer at
    // 64 heads x 32768 tokens, d = 128, one a tile 0.5 % at 128 x 4096, d = 64; skipping the waits after a failure 2 %.)
    auto wait = [&](uint64_t *b, int parity, int where) {
        ok = mbar_wait(b, (uint32_t)(parity ^ flip), abort_flag, status, where) && ok;
    };
    int lo = lo_sel - my.sel0 * kBlockN, hi = lim_sel - 1 - my.sel0 * kBlockN;
    for (int k = 0; k < n_mine; ++k) {
        // visible column interval [lo, hi] of this row in the stream tile
        if (k == my.n_sel) {
            lo = loc_lo - my.loc0 * kBlockN;
            hi = tq - my.loc0 * kBlockN;
        }
        const bool need_mask = __any_sync(0xffffffffu, lo > 0 || hi < kBlockN - 1);
        const bool none = need_mask && !__any_sync(0xffffffffu, max(lo, 0) <= min(hi, kBlockN - 1));   // (a warp whose rows see none of it skips the arithmetic)
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
                tc_fence_after();
            }
            __syncwarp();
            tmem_st32(p_addr, masked);
            tmem_st32(p_addr + 32, masked);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_first(bar.p_full + x);
            lo -= kBlockN;
            hi -= kBlockN;
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
            __syncwarp();
        }
        tmem_st32(p_addr, pk[0]);
        tmem_st32(p_addr + 32, pk[1]);
        l_sum += acc.x + acc.y;
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_first(bar.p_full + x);
        lo -= kBlockN;
        hi -= kBlockN;
    }
    // ---- epilogue: y = (O e^{m-ms} + e^{-ms} N_LA) / (l e^{m-ms} + e^{-ms} D_LA), ms = max(m, 0)
    // The linear branch arrives as up to two partial results (one per feature half): y_p = N_p / D_p as bf16
    // and D_p, so N_LA = sum y_p D_p and D_LA = sum D_p.  A thread owns a row, but loads / stores in which
    // every lane touches a different row cost a memory instruction per 16 bytes and row; so the y_p come in by TMA, into
    // stages of the ring behind the item's keys (they are there by the time the last product is), and Y goes out the same
    // way (output_role), from where the first part lay.
    float da = 0.f, db = 0.f;
    if (n_parts > 0 && t < N) {
        da = d_part[(long long)bh * N + t];
        if (n_parts > 1) db = d_part[part_stride_d + (long long)bh * N + t];
    }
    bool last;
    const bool there = ahead(last);
    if (n_mine > 0) {                              // (in a pair also where none of this CTA's rows are below N)
        wait(bar.pv_done + x, (n_mine - 1) & 1, 9);   // (every query tile has a LOC tile)
        if (__all_sync(0xffffffffu, ok)) {
            tc_fence_after();
            wait(bar.y_full + x, y_flip ^ flip, 12);
            if (__all_sync(0xffffffffu, ok)) {
                // this warp's 32 rows of a part: 64 columns of 128 bytes a row, 16-byte pieces swizzled by the row
                uint8_t *part0 = ring + y_stage * P::kStage + (warp & 3) * 32 * 128;
                uint8_t *part1 = P::kPartsPerStage > 1 ? part0 + P::kPartTile : ring + (y_stage + 1) % P::kStages * P::kStage + (warp & 3) * 32 * 128;
                float fs = 1.f, fa = 0.f, fb = 0.f;
                const float dla = da + db;
                if (dla > 0.f) {
                    const float m_nat = m_used * 0.6931471805599453f;
                    const float ms = fmaxf(m_nat, 0.f);
                    fs = __expf(m_nat - ms);
                    const float fl = __expf(-ms);
                    fa = fl * da;
                    fb = fl * db;
                }
                const float inv = 1.f / (l_sum * fs + fa + fb);
                const bool with_la = (n_parts > 0) && __any_sync(0xffffffffu, dla > 0.f);
                const float2 fs2 = make_float2(fs, fs), fa2 = make_float2(fa, fa), fb2 = make_float2(fb, fb), inv2 = make_float2(inv, inv);
#pragma unroll 1
                for (int q = 0; q < D / 32; ++q) {
                    uint32_t orow[32];
                    tmem_ld32(o_addr + q * 32, orow);
                    auto offset = [&](int j8) { return (q >> 1) * (kBlockM * 128) + lane * 128 + ((((q & 1) * 4 + j8) ^ (lane & 7)) << 4); };
                    uint4 pa[4], pb[4];   // (read before the first is written over)
#pragma unroll
                    for (int j8 = 0; j8 < 4; ++j8) {
                        pa[j8] = pb[j8] = make_uint4(0, 0, 0, 0);
                        if (with_la) {
                            pa[j8] = *reinterpret_cast<const uint4 *>(part0 + offset(j8));
                            if (n_parts > 1) pb[j8] = *reinterpret_cast<const uint4 *>(part1 + offset(j8));
                        }
                    }
                    tmem_wait_ld();
#pragma unroll
                    for (int j8 = 0; j8 < 4; ++j8) {
                        const uint32_t wa[4] = {pa[j8].x, pa[j8].y, pa[j8].z, pa[j8].w}, wb[4] = {pb[j8].x, pb[j8].y, pb[j8].z, pb[j8].w};
                        uint32_t out[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {   // two columns per 32-bit word
                            const float2 a = make_float2(__uint_as_float(wa[e] << 16), __uint_as_float(wa[e] & 0xffff0000u));
                            const float2 b = make_float2(__uint_as_float(wb[e] << 16), __uint_as_float(wb[e] & 0xffff0000u));
                            const float2 la = __ffma2_rn(fa2, a, __fmul2_rn(fb2, b));
                            const float2 o2 = make_float2(__uint_as_float(orow[8 * j8 + 2 * e]), __uint_as_float(orow[8 * j8 + 2 * e + 1]));
                            const float2 y2 = __fmul2_rn(__ffma2_rn(o2, fs2, la), inv2);
                            out[e] = pack_bf16(y2.x, y2.y);
                        }
                        *reinterpret_cast<uint4 *>(part0 + offset(j8)) = make_uint4(out[0], out[1], out[2], out[3]);
                    }
                }
                tc_fence_before();
                if (last) {   // (nothing is left to hand the stores to an output warp for)
                    __syncwarp();
                    store_rows<D>(part0, Y, (long long)bh * N, tile_row0 + (warp & 3) * 32, min(N - tile_row0 - (warp & 3) * 32, 32));
                } else {
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar.y_ready + x);
                }
            }
        }
    }
    ok = ok && there;
    return __all_sync(0xffffffffu, ok);
}

// TMA producer (one thread): the Q tiles of an item, then the K and V tiles of its stream, as far ahead as the ring has free
// stages, then what the epilogue merges.  In a pair every CTA loads its halves; the byte counts of Q, K and V complete on the
// first CTA's barriers.
template <int D, bool kPair, class TellPeer>
__device__ __forceinline__ void producer_role(Work w, const AttnBars &bar, uint8_t *smem, const uint32_t rank,
                                              const CUtensorMap &tm_q, const CUtensorMap &tm_k, const CUtensorMap &tm_v,
                                              const CUtensorMap &tm_ksel, const CUtensorMap &tm_vsel, const CUtensorMap &tm_p0,
                                              const CUtensorMap &tm_p1, volatile int *abort_flag, int *status, TellPeer tell_peer) {
    using P = AttnPlan<D, kPair>;
    constexpr int kCtas = kPair ? 2 : 1, kStages = P::kStages;
    const uint32_t q_full0 = mapa(smem_u32(bar.q_full), 0), kv_full0 = mapa(smem_u32(bar.kv_full), 0);
    auto load = [&](uint8_t *dst, const CUtensorMap &map, uint64_t *b, uint32_t b0, int col, int row) {
        if constexpr (kPair) tma_load_2d_pair(dst, &map, b0, col, row);
        else tma_load_2d(dst, &map, b, col, row);
    };
    const int n_y = P::y_entries(w.n_parts);
    bool ok = true;
    int armed = 0, n = 0, q_armed = 0, a_armed = 0, b_armed = 0;
    RingPos pos{0, 0};
    prefetch_map(&tm_k);
    prefetch_map(&tm_v);
    if (w.n_parts > 0) prefetch_map(&tm_p0);
    if (w.n_parts > 1) prefetch_map(&tm_p1);
    for (bool more = true; more && ok; ++n) {
        const Stream st = w.stream();
        const int kv_row0 = w.bh / w.rep * w.N, q_row = w.bh * w.N + w.R0;
        // (with topk = chunk every token is selected and the compacted arrays would be copies of K / V: the salient prefix is
        // then read from K / V themselves, and tm_ksel / tm_vsel alias tm_k / tm_v)
        const int sel_row0 = w.sel_identity ? kv_row0 : w.bh * w.sel_rows;
        const int n_q = w.n_query_tiles(), entries = st.entries();   // (every query tile has a LOC tile)
        ok = mbar_wait(bar.q_empty, (n & 1) ^ 1, abort_flag, status, 2);
        if (!ok) break;
        if (rank == 0) mbar_expect_tx(bar.q_full, kCtas * n_q * P::kQTile);
        ++q_armed;
        for (int x = 0; x < n_q; ++x)
            for (int half = 0; half < D / 64; ++half)
                load(smem + P::kQ + x * P::kQTile + half * (kBlockM * 128), tm_q, bar.q_full, q_full0, half * 64,
                     q_row + ((int)rank + x * kCtas) * kBlockM);
        int next = 0, failed = 0;
        for (int e = 0; e < entries; ++e, ++armed) {
            if (rank == 0 && e == entries - 1) {
                // the item after this one, unless a CTA has failed: asked for ahead of the wait for the last stage, needed behind the loop
                next = atomicAdd(status + kNextItem, 1);
                failed = *reinterpret_cast<volatile int *>(status);
            }
            ok = mbar_wait(bar.kv_empty + pos.stage, pos.parity ^ 1, abort_flag, status, 1);
            if (!ok) break;
            bool sel;
            const int tile = st.tile(e, sel), row = (sel ? sel_row0 : kv_row0) + tile * kBlockN;
            if (rank == 0) mbar_expect_tx(bar.kv_full + pos.stage, kCtas * P::kStage);
            for (int half = 0; half < D / 64; ++half)   // (of a pair: this CTA's 64 keys)
                load(smem + P::kK + pos.stage * P::kStage + half * (P::kKRows * 128), sel ? tm_ksel : tm_k, bar.kv_full + pos.stage,
                     kv_full0 + pos.stage * 8, half * 64, row + (int)rank * P::kKRows);
            for (int q = 0; q < P::kVCols / 64; ++q)    // this CTA's value columns, 64 at a time
                load(smem + P::kV + pos.stage * P::kStage + q * (kBlockN * 128), sel ? tm_vsel : tm_v, bar.kv_full + pos.stage,
                     kv_full0 + pos.stage * 8, (int)rank * P::kVCols + q * 64, row);
            pos.next(kStages);
        }
        if (!ok) break;
        if (rank == 0) {   // (ahead of the outputs, which come only with the last products)
            ok = mbar_wait(bar.item_empty + (n & 1), (uint32_t)((n >> 1) & 1) ^ 1u, abort_flag, status, 14);
            if (!ok) break;
            next += (int)(gridDim.x / kCtas);
            more = failed == 0 && next < w.total;
            if (more) w.set(next);
            else w.bh = -1;
            volatile int *slot = w.item + 2 * (n & 1);
            slot[0] = w.bh;
            slot[1] = w.R0;
            mbar_arrive(bar.item_full + (n & 1));
            if constexpr (kPair) {
                const uint32_t peer_slot = mapa(smem_u32(const_cast<int *>(slot)), 1);
                st_cluster_u32(peer_slot, (uint32_t)w.bh);
                st_cluster_u32(peer_slot + 4, (uint32_t)w.R0);
                mbar_arrive_release_cluster(mapa(smem_u32(bar.item_full + (n & 1)), 1));
            }
        }
        // Entries of the outputs: the parts' rows of this CTA's query tiles (rows behind the last of a head are never used).
        // They pass the ring's full-barrier at once: nobody waits for it, but its phases count the rounds.
        // (An item of few tiles leaves the ring free for the outputs of the next one before the warps that wait for its own have
        // looked; they would look for a parity that has come round again.  So the next outputs wait for these to be taken up.  us a call,
        // without that and with it: 128 heads x 4096 tokens, d = 64, 478.4 and 481.0, a quarter kept 442.7 and 443.9; d = 128 the same.)
        for (int x = 0; x < n_q && ok; ++x) {
            ok = mbar_wait(bar.y_taken + x, (uint32_t)((x ? b_armed : a_armed) & 1) ^ 1u, abort_flag, status, 17);
            if (!ok) break;
            for (int y = 0; y < n_y; ++y, ++armed) {
                ok = mbar_wait(bar.kv_empty + pos.stage, pos.parity ^ 1, abort_flag, status, 10);
                if (!ok) {
                    if (y > 0) mbar_arrive(bar.y_full + x);   // (for the wait below)
                    break;
                }
                if (rank == 0) mbar_arrive(bar.kv_full + pos.stage);
                const int parts = min(w.n_parts - y * P::kPartsPerStage, P::kPartsPerStage);   // of this entry
                if (parts > 0) mbar_expect_tx(bar.y_full + x, parts * P::kPartTile);
                else mbar_arrive(bar.y_full + x);
                if (y == 0) ++(x ? b_armed : a_armed);
                for (int part = y * P::kPartsPerStage; part < y * P::kPartsPerStage + parts; ++part)
                    for (int half = 0; half < D / 64; ++half)
                        tma_load_2d(smem + P::kK + pos.stage * P::kStage + (part - y * P::kPartsPerStage) * P::kPartTile + half * (kBlockM * 128),
                                    part ? &tm_p1 : &tm_p0, bar.y_full + x, half * 64, q_row + ((int)rank + x * kCtas) * kBlockM);
                pos.next(kStages);
            }
        }
        if (!ok) break;
        if constexpr (kPair) {
            // The second CTA's loads count on the first's full-barriers, whose phases the first's own output entries move on as
            // well: it begins with an item when the first has passed those of the item before.  It gives the item's place back
            // behind that wait, and the first has waited for the place of the item before last, so that of the two
            // barriers, taken by turns, none is two phases ahead.
            if (rank == 0) {
                mbar_arrive_cluster(mapa(smem_u32(bar.first_done + (n & 1)), 1));
            } else {
                more = next_item<kPair>(w, bar, n, abort_flag, status, ok);
                ok = ok && mbar_wait(bar.first_done + (n & 1), (uint32_t)(n >> 1) & 1u, abort_flag, status, 16);
                if (ok) item_taken<kPair>(bar, n);
            }
        }
    }
    // leave no copy in flight behind.  In a pair the first CTA's barriers count both CTAs' bytes; the second, where it has
    // given up and the first may not know of its last copies, waits out a fixed stretch that is long against a tile load.
    const long long t0 = clock64();
    if constexpr (kPair) {
        if (!ok) tell_peer();
    }
    if (a_armed > 0) mbar_wait_drain(bar.y_full, (uint32_t)(a_armed - 1) & 1u, t0);
    if (b_armed > 0) mbar_wait_drain(bar.y_full + 1, (uint32_t)(b_armed - 1) & 1u, t0);
    if (rank == 0) {
        if (q_armed > 0) mbar_wait_drain(bar.q_full, (uint32_t)(q_armed - 1) & 1u, t0);
        mbar_drain_ring(bar.kv_full, kStages, armed, t0);
    } else if (!ok) {
        while (clock64() - t0 < 200000) {}
    }
}

// Stores of query tile x (a warp): the tile's rows as the softmax warps have left them in the output's first stage.  While an
// item runs, what its epilogue reads of D_p comes into L2.
template <int D, bool kPair>
__device__ __forceinline__ void output_role(Work w, const AttnBars &bar, const uint8_t *ring, const int x, const uint32_t rank,
                                            const CUtensorMap &tm_y, const float *d_part, __nv_bfloat16 *Y, volatile int *abort_flag,
                                            int *status) {
    using P = AttnPlan<D, kPair>;
    constexpr int kCtas = kPair ? 2 : 1, kStages = P::kStages;
    const int lane = threadIdx.x & 31, n_y = P::y_entries(w.n_parts);
    int ring0 = 0, y_odd = 0;
    bool ok = true;
    if (lane == 0) prefetch_map(&tm_y);
    bool more = true;
    for (int n = 0; more; ++n) {
        const Stream st = w.stream();
        const int y_entry = ring0 + st.entries() + x * n_y, t0 = w.R0 + (x * kCtas + (int)rank) * kBlockM, rows = min(w.N - t0, kBlockM);
        const int bh = w.bh;
        const bool live = x < w.n_query_tiles();   // (below, w is at the next item)
        ring0 = (ring0 + st.entries() + n_y * w.n_query_tiles()) % kStages;
        if (rows > 0 && lane < 8 && (lane >> 2) < w.n_parts)   // 128 bytes a lane
            prefetch_l2(d_part + ((long long)(lane >> 2) * w.n_heads + bh) * w.N + t0 + min((lane & 3) * 32, rows - 1));
        more = next_item_of_warp<kPair>(w, bar, n, abort_flag, status, ok);
        if (!ok || !more) break;   // (the last item's rows are stored by the softmax warps)
        if (!live) continue;
        ok = mbar_wait(bar.y_ready + x, y_odd, abort_flag, status, 15);
        if (!__all_sync(0xffffffffu, ok)) break;
        y_odd ^= 1;
        if (lane == 0) mbar_arrive(bar.y_taken + x);
        const uint8_t *tile = ring + y_entry % kStages * P::kStage;
        if (rows == kBlockM) {
            if (lane == 0) {
#pragma unroll
                for (int a = 0; a < D / 64; ++a) tma_store_2d(&tm_y, tile + a * (kBlockM * 128), a * 64, bh * w.N + t0);
                bulk_store_commit();
                bulk_store_wait_read();
            }
        } else {   // the last rows of a sequence (the map does not know where a head ends)
            store_rows<D>(tile, Y, (long long)bh * w.N, t0, rows);
            fence_proxy_async();   // (the stage is next written by TMA)
        }
        __syncwarp();
        if (lane == 0)
            for (int y = 0; y < n_y; ++y) mbar_arrive(bar.kv_empty + (y_entry + y) % kStages);
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
// arithmetic, two of them per scheduler (32768 tokens, d = 128: issue slots 52 %, special-function unit 52 %, tensor pipe 71 %;
// 4096 tokens, d = 64: 50, 47 and 32 %).  With P over S, S of a tile waited for the softmax warps of the tile before and these for
// it (us a call, then and with P in its own place, when a CTA ended with its item, in turn on one box: 64 heads x 32768
// tokens, d = 128, every token kept 15887 and 15154, a quarter 6665 and 6208; 32 x 131072, capped at 896, 8697 and 7809; 128 x
// 4096, d = 64, every token 551 and 502, a quarter 585 and 515; the scan and the score kernel have a part in the quarters and in
// the capped call).  Two threads per row instead of one (16 softmax warps) were slower by 10 %: the stream's bookkeeping doubles.
template <int D, bool kPair, class TellPeer>
__device__ __forceinline__ void mma_role(Work w, const AttnBars &bar, uint8_t *smem, const uint32_t tmem_base,
                                         volatile int *abort_flag, int *status, TellPeer tell_peer) {
    using P = AttnPlan<D, kPair>;
    using TM = TmemPlan<D>;
    constexpr int kM = kPair ? 2 * kBlockM : kBlockM, kStages = P::kStages, kAhead = 3;
    constexpr uint32_t idesc_qk = make_idesc(kM, kBlockN, false);
    constexpr uint32_t idesc_pv = make_idesc(kM, D, true);
    const bool leader = elect_one();
    bool ok = true;
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
    struct Item {
        int m, x, k;
        RingPos pos;
    };
    Item qk{0, 0, 0, {0, 0}}, pv{0, 0, 0, {0, 0}};
    const int n_y = P::y_entries(w.n_parts);
    uint32_t qk_odd = 0, pv_odd = 0;   // bit x: parity of the S (of the P V) of query tile x that there have been
    int x_prev = -1;                   // of the item whose S was formed last
    bool more = true;
    for (int n = 0; more; ++n) {
        const Stream st = w.stream();
        const int n_own0 = st.n_lead + 2 * st.n_shared, n_items = n_own0 + st.n_a + st.n_b;
        const int turns = min(st.n_a, st.n_b), x_last = st.n_a > st.n_b ? 0 : 1;
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
        auto issue_qk = [&]() {
            // K and V of the entry have arrived (B follows A on the entries that they share)
            if (qk.m >= n_own0 || qk.x == 0) wait(bar.kv_full + qk.pos.stage, qk.pos.parity, 7);
            // the place of S is free: its last tile has been read (before the first there is none)
            if constexpr (TM::kOneS) {
                if (x_prev >= 0) wait(bar.s_free + x_prev, ((qk_odd >> x_prev) & 1) ^ 1, 3);
            } else {
                wait(bar.s_free + qk.x, ((qk_odd >> qk.x) & 1) ^ 1, 3);
            }
            tc_fence_after();
            const uint32_t q_lo = q_lo0 + qk.x * (P::kQTile >> 4), k_lo = k_lo0 + qk.pos.stage * (P::kStage >> 4), d_s = tmem_base + TM::s(qk.x);
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
                if (qk.m + 1 == n_items) commit(bar.q_empty);
            }
            x_prev = qk.x;
            qk_odd ^= 1u << qk.x;
            advance(qk);
        };
        auto issue_pv = [&]() {
            const uint32_t v_lo = v_lo0 + pv.pos.stage * (P::kStage >> 4), d_o = tmem_base + TM::o(pv.x), a_p = tmem_base + TM::p(pv.x);
            const uint32_t acc0 = pv.k > 0 ? 1u : 0u;
            wait(bar.p_full + pv.x, (pv_odd >> pv.x) & 1, 5);
            tc_fence_after();
            if (leader && ok) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {   // 16 keys a step
                    if constexpr (kPair) mma_ts_lo_pair<idesc_pv>(d_o, a_p + j * 8, v_lo + j * (16 * 128 >> 4), j == 0 ? acc0 : 1u);
                    else mma_ts_lo<idesc_pv>(d_o, a_p + j * 8, v_lo + j * (16 * 128 >> 4), j == 0 ? acc0 : 1u);
                }
                commit(bar.pv_done + pv.x);
                // (an entry that both query tiles use is done with B's product)
                if (pv.x == 1 || pv.m < st.n_lead || pv.m >= n_own0) commit(bar.kv_empty + pv.pos.stage);
            }
            pv_odd ^= 1u << pv.x;
            advance(pv);
        };
        wait(bar.q_full, n & 1, 4);
        tc_fence_after();
        for (int m = 0; m < min(kAhead, n_items); ++m) issue_qk();
        while (pv.m < n_items) {
            issue_pv();
            if (qk.m < n_items) issue_qk();
        }
        // past the entries of the outputs
        qk.pos.skip(n_y * w.n_query_tiles(), kStages);
        pv = qk = Item{0, 0, 0, qk.pos};
        if (!__all_sync(0xffffffffu, ok)) break;
        more = next_item_of_warp<kPair>(w, bar, n, abort_flag, status, ok);
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

// Softmax-attention branch and merge: items of 256 (a pair: 512) rows of one (batch, head), see Work.  Between two items little
// comes: the next Q comes in while the last products run, its first S is formed while the softmax warps merge, and the linear
// branch's results and the output pass through the key ring, so that neither waits for memory.  (With a CTA per item an item
// had, beside 2900 to 3300 cycles for a tile of both query tiles, a start of some 3000 cycles and an end of 3000 to 5000 without
// a linear branch, 8000 with it, and 15000 to 38000 where its results had left L2; now 3000 to 6500 in all.  us of the
// kernel, then and now, in turn on one box: 128 heads x 4096 tokens, d = 64, a quarter kept 270 and 227; 64 x 32768, d = 128, a
// quarter kept 4229 and 3745; 32 x 131072, capped at 896, 3960 and 2865.)
template <int D, bool kPair>
__device__ __forceinline__ void attention_body(const AttnMaps &tm, const float *d_part, __nv_bfloat16 *Y, int *status, int H, int Hkv,
                                               int N, int C, int lam, int budget, int sel_rows, int sel_identity, int n_parts,
                                               float scale_log2, int n_blocks, int n_heads, int set_heads) {
    using P = AttnPlan<D, kPair>;
    constexpr int kCtas = kPair ? 2 : 1, kRows = kCtas * kBlockM, kStages = P::kStages;
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
    Work w{n_blocks, n_heads, set_heads, H / Hkv, N, C == 128 ? 7 : 6, lam, budget, sel_rows, sel_identity, n_parts, kRows,
           (int)(kPair ? blockIdx.x >> 1 : blockIdx.x), n_blocks * n_heads, reinterpret_cast<volatile int *>(smem + P::kMisc + 16), 0, 0};
    // Here, where all warps do it together, and the KV head by one division (rep): with the first in every role's own code and four
    // divisions an item took some 500 cycles more, the first S of a call came 600 later (us a call: 128 heads x 4096 tokens, d = 64, 477.3
    // and 474.1, a quarter kept 442.4 and 440.7, 128 x 1500 114.8 and 113.3, 64 x 214 18.55 and 18.09; d = 128, 16 x 1000 33.6 and 32.6).
    w.set(w.first);
    auto sync_all = [&]() {
        if constexpr (kPair) cluster_sync_all();
        else __syncthreads();
    };

    if (threadIdx.x == 0) {
        mbar_init(bar.q_full, 1);
        mbar_init(bar.q_empty, 1);
        for (int i = 0; i < kStages; ++i) {
            mbar_init(bar.kv_full + i, 1);
            mbar_init(bar.kv_empty + i, 1);   // the last product that reads the stage has, or the output has left it
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar.s_full + i, 1);
            mbar_init(bar.s_free + i, kCtas * 4);   // one arrival per softmax warp of the query tile
            mbar_init(bar.p_full + i, kCtas * 4);
            mbar_init(bar.pv_done + i, 1);
            mbar_init(bar.y_full + i, P::y_entries(n_parts));
            mbar_init(bar.item_full + i, 1);
            mbar_init(bar.y_ready + i, 4);
            mbar_init(bar.y_taken + i, 1);
            mbar_init(bar.first_done + i, 1);
            mbar_init(bar.item_empty + i, kCtas * 10 + 1 + (kCtas - 1));   // softmax and output warps, the issuing warp, the other producer
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

    // Registers move from the last four warps to the softmax warps, whose threads hold a row of S (per scheduler, of the 3 x 168
    // registers that the CTA was launched with).
    constexpr int kSoftmaxRegs = 224, kOtherRegs = 3 * 168 - 2 * kSoftmaxRegs;
    if (warp >= kProducerWarp) {
        reg_dec<kOtherRegs>();
        if (warp == kProducerWarp) {
            if (lane == 0)
                producer_role<D, kPair>(w, bar, smem, rank, tm.q, tm.k, tm.v, tm.ksel, tm.vsel, tm.p0, tm.p1, abort_flag, status, tell_peer);
        } else if (warp == kMmaWarp && rank == 0) {
            mma_role<D, kPair>(w, bar, smem, tmem_base, abort_flag, status, tell_peer);
        } else if (warp > kMmaWarp) {
            output_role<D, kPair>(w, bar, smem + P::kK, warp - kMmaWarp - 1, rank, tm.y, d_part, Y, abort_flag, status);
        }
    } else {
        reg_inc<kSoftmaxRegs>();
        const int x = warp >> 2;                       // 0: tile A, 1: tile B
        const int n_y = P::y_entries(n_parts);
        int ring0 = 0, flip = 0, y_flip = 0;           // ring stage of the item's first entry; see softmax_role
        bool ok = true, more = true;
        for (int n = 0; more && ok; ++n) {
            const Stream st = w.stream();
            const Stream::Mine my = st.mine(x);
            const int y_stage = (ring0 + st.entries() + x * n_y) % kStages;
            ring0 = (ring0 + st.entries() + n_y * w.n_query_tiles()) % kStages;
            const int row0 = w.R0 + (x * kCtas + (int)rank) * kBlockM, bh = w.bh;
            auto ahead = [&](bool &last) {   // (while the item's last product runs)
                bool waited;
                more = next_item_of_warp<kPair>(w, bar, n, abort_flag, status, waited);
                last = !more;
                return waited;
            };
            ok = softmax_role<D, kPair>(my, bar, x, row0, tmem_base, abort_flag, status, smem + P::kK, y_stage, flip, y_flip, d_part,
                                        n_parts, (long long)n_heads * N, Y, bh, N, w.log2_c, lam, budget, scale_log2, ahead);
            flip ^= my.n & 1;
            y_flip ^= my.n > 0 ? 1 : 0;
        }
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
sa_merge_tc_kernel(const __grid_constant__ AttnMaps tm, const float *d_part, __nv_bfloat16 *Y, int *status, int H, int Hkv, int N, int C,
                   int lam, int budget, int sel_rows, int sel_identity, int n_parts, float scale_log2, int n_blocks, int n_heads,
                   int set_heads) {
    grid_dep_wait();
    grid_dep_launch();
    attention_body<D, false>(tm, d_part, Y, status, H, Hkv, N, C, lam, budget, sel_rows, sel_identity, n_parts, scale_log2, n_blocks,
                             n_heads, set_heads);
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
// softmax warps of both CTAs arrive on rank 0's barriers.  Ring stages of keys are free in both CTAs with the commit of the last
// product that reads them, an output's stage when the CTA's own output warp is done with it.
template <int D>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
sa_merge_pair_kernel(const __grid_constant__ AttnMaps tm, const float *d_part, __nv_bfloat16 *Y, int *status, int H, int Hkv, int N, int C,
                     int lam, int budget, int sel_rows, int sel_identity, int n_parts, float scale_log2, int n_blocks, int n_heads,
                     int set_heads) {
    grid_dep_wait();
    grid_dep_launch();
    attention_body<D, true>(tm, d_part, Y, status, H, Hkv, N, C, lam, budget, sel_rows, sel_identity, n_parts, scale_log2, n_blocks,
                            n_heads, set_heads);
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
// six or seven others, by twelve warps an SM at C = 64, eight at C = 128, where a third group's rows spill (special-function unit
// 66 to 69 % busy and 61 %, issue slots 50 and 37 %).  us of the kernel: 32 heads x 32768 tokens, d = 128, 85.6, 128 x 4096, d = 64, 44.7;
// C = 128, 32 x 32768, 179.8.  us of a call for the scores alone with eight warps and with twelve, in turn on one box: 64 x 32768,
// d = 128, 201 to 219 and 175 to 180, 128 x 4096, d = 64, 60.5 and 56.
// Warps: 0 TMA producer, 1 MMA issuer, 2-5 score group 0, 6-9 score group 1, ...; TMEM lane quarter = warp % 4.
// ---------------------------------------------------------------------------
template <int D>
struct ScoreSmem {
    static constexpr int kQBytes = kBlockM * D * 2, kKBytes = 2 * kBlockN * D * 2;
    static constexpr int kStage = kQBytes + kKBytes;
    static constexpr int kBar = 2 * kStage;          // full[2], smem_free[2], tmem_free[2], mma_done[4]
    static constexpr int kMisc = kBar + 10 * 8;      // tmem base, abort flag
    static constexpr int kSc = kMisc + 16;           // [4][128] ranking keys of a group's tile (16-byte aligned)
    static constexpr int kBallot = kSc + 4 * kBlockM * 4;   // [4][4]
    static constexpr int kTotal = kBallot + 4 * 4 * 4;
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

// Score groups of four warps, which take a CTA's tiles in turn: three where a row's C values leave the registers for it (two at
// C = 128, where a third made the rows spill).
template <int C>
constexpr int kScoreGroups = C == 64 ? 3 : 2;
template <int C>
constexpr int kScoreThreads = 64 + 128 * kScoreGroups<C>;
template <int D, int C, bool kTinyEps>
__global__ void __launch_bounds__(kScoreThreads<C>, 1)
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
    // (mma_done: of a score group, which so sees every phase of the barrier that it waits on; smem_free, tmem_free: of a stage)
    uint64_t *smem_free = full + 2, *tmem_free = full + 4, *mma_done = full + 6;
    uint32_t *tmem_base_slot = reinterpret_cast<uint32_t *>(smem + P::kMisc);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + P::kMisc + 8);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int Tn = (N + C - 1) / C;

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(full + s, 1);
            mbar_init(smem_free + s, 1);
            mbar_init(tmem_free + s, 4);   // one arrival per warp of the score group
        }
        for (int g = 0; g < kScoreGroups<C>; ++g) mbar_init(mma_done + g, 1);
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
                tc_commit(mma_done + it % kScoreGroups<C>);
            }
            // no MMA may still be running when tensor memory is freed: after a failure wait (bounded) for the
            // last group issued (its commit covers everything before it)
            if (!ok && it > 0) mbar_wait_drain(mma_done + (it - 1) % kScoreGroups<C>, ((it - 1) / kScoreGroups<C>) & 1);
        }
    } else {
        constexpr int kGroups = kScoreGroups<C>;
        const int g = (warp - 2) >> 2;                 // score group: tiles g, g + kGroups, ... of the CTA
        const int wq = warp & 3;                       // TMEM lane quarter this warp may read
        const int r = wq * 32 + lane;                  // row of the tile owned by this thread
        int *keys = reinterpret_cast<int *>(smem + P::kSc) + g * kBlockM;
        uint32_t *ballots = reinterpret_cast<uint32_t *>(smem + P::kBallot) + g * 4;
        const uint32_t taddr0 = tmem_base + ((uint32_t)(wq * 32) << 16) + (uint32_t)(wq * 32 + kBlockN - C);
        const int group_bar = 1 + g;
        int it = g, j = 0;
        for (int n = blockIdx.x + g * gridDim.x; n < n_tiles; n += kGroups * gridDim.x, it += kGroups, ++j) {
            const int st = kGroups == 2 ? g : it & 1;      // stage and TMEM accumulator
            const uint32_t taddr = taddr0 + st * 256;
            const int bh = n / n_row_blocks, R0 = (n - bh * n_row_blocks) * kBlockM;
            const int t = R0 + r;
            bool ok = mbar_wait(mma_done + g, j & 1, abort_flag, status, 21);
            // the group leaves the loop together
            {
                uint32_t all_ok;
                asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 p, %1, 0;\nbarrier.cta.red.and.pred q, %2, 128, p;\nselp.b32 %0, 1, 0, q;\n}"
                             : "=r"(all_ok) : "r"((uint32_t)ok), "r"(group_bar) : "memory");
                ok = all_ok != 0;
            }
            if (!ok) break;
            tc_fence_after();
            if (r == 0) mbar_arrive(smem_free + st);   // the logits are complete: the stage's operands are free
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
                    if (lane == 0) mbar_arrive(tmem_free + st);
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
    const unsigned long long q_rows = (unsigned long long)BH * N;
    const bf *part = (const bf *)(n_parts > 0 ? y_part : Y);   // (the maps of absent parts are not used)
    AttnMaps tm;
    if (!make_map(&tm.q, Q, q_rows, D) || !make_map_2d(&tm.k, K, kv_rows, D, kPair ? kBlockN / 2 : kBlockN, false) ||
        !make_map(&tm.v, V, kv_rows, D) ||
        !make_map_2d(&tm.ksel, identity ? K : k_sel, sel_total, D, kPair ? kBlockN / 2 : kBlockN, false) ||
        !make_map(&tm.vsel, identity ? V : v_sel, sel_total, D) || !make_map(&tm.p0, part, q_rows, D) ||
        !make_map(&tm.p1, n_parts > 1 ? part + q_rows * D : part, q_rows, D) || !make_map(&tm.y, Y, q_rows, D))
        return STILL_ERR_CUDA;
    const float scale_log2 = p->sm_scale * 1.4426950408889634f;
    const int rep = p->H / p->Hkv;
    const int set_heads = set_of_heads(BH, rep, ((identity ? 0 : sel_rows) + N / rep + 1) * D * 4);
    int dev = 0, n_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n_sm <= 0)
        return STILL_ERR_CUDA;
    constexpr int kCtas = kPair ? 2 : 1, kSmem = AttnPlan<D, kPair>::kAlloc;
    const auto kernel = [] {
        if constexpr (kPair) return sa_merge_pair_kernel<D>;
        else return sa_merge_tc_kernel<D>;
    }();
    if (ensure_dynamic_smem((const void *)kernel, kSmem) != cudaSuccess) return STILL_ERR_CUDA;
    const long long n_blocks = (N + kCtas * 2 * kBlockM - 1) / (kCtas * 2 * kBlockM), items = n_blocks * BH;
    const dim3 grid((unsigned)(kCtas * std::min<long long>(items, std::max(1, n_sm / kCtas))));   // they stay (see Work)
    profile_mark_begin(st);
    const cudaError_t e = launch_dependent(kernel, grid, dim3(kThreads), kSmem, st, tm, d_part, (bf *)Y, status, p->H, p->Hkv, (int)N, p->chunk,
                                           p->topk, (int)p->max_salient, (int)sel_rows, identity ? 1 : 0, n_parts, scale_log2, (int)n_blocks,
                                           (int)BH, set_heads);
    profile_mark_end(st);
    if (e != cudaSuccess) return STILL_ERR_CUDA;
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
    if (launch_dependent(kernel, dim3(grid), dim3(kScoreThreads<C>), kSmem, st, tq, tk, scores, sel_idx, status, p->H, p->Hkv, (int)N, p->topk,
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
