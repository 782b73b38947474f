// Tensor-core sparse attention forward (tcgen05 MMA, TMEM accumulators, TMA-fed Q/K/V), one persistent
// kernel over a single queue of work items.
//
// Two kinds of items:
//   routed (key-chunk stationary): (head, chunk c, up to 256 entries of the list of (query, slot) pairs that
//     picked c).  The Q rows are gathered by TMA (four rows per copy), the keys are exactly the tokens of chunk
//     c, and each (query, slot) gets a partial result (normalised output + log-sum-exp) in the workspace;
//   anchor (query-tile stationary): (head, up to 256 consecutive rows of one chunk); keys are the chunk's
//     mandatory anchors (merged token ranges).  Its epilogue merges the row's <= k routed partials by
//     log-sum-exp and writes O and LSE.
// The queue holds, group of heads by group of heads, the group's routed items and then its anchor items.  One
// CTA per SM claims items in queue order (a global counter), so the two kinds need no separate launches and no
// CTA is set up or torn down per item: the tensor memory, the barriers and the K/V ring live for the whole
// kernel, and the next item's Q tiles and first K/V tiles are on their way while the current item finishes.
// What an anchor item needs from the routed items of its group (their partials) is awaited late, just before
// its merge, on a count of completed rows; by then every routed item of the group has long been claimed, by a
// CTA that is running, so the wait ends.  Partials of consecutive groups alternate between two buffers; a
// routed item waits, before it stores, for the anchor items that read its buffer two groups ago.
//
// 12 warps in three warpgroups (the third gives most of its registers to the other two); an item is two 128-row
// query tiles that share every K/V tile:
//   warps 0-3 / 4-7  softmax group of query tile 0 / 1, one row per thread (TMEM lane = row): read S from TMEM,
//              online softmax, write P back to TMEM as packed bf16 (aliasing S; the first 64 keys are released
//              to the issuer before the exponentials of the other 64), lazily rescale O, epilogue.  The
//              exponentials of the two tiles take turns;
//   warp 8     lane 0, TMA producer: the K and V tiles of 128 keys, two stages each, 128-byte swizzle; the ring
//              runs across items.  Lane 16, bookkeeping: waits for what an item depends on, and when the item's
//              rows are stored adds them to the queue's count of completed rows (the one thread that pays for
//              device-wide fences);
//   warps 9, 10  one MMA-issuing warp per query tile g:  S_g(0), then  O_g += P_g V(j),  S_g(j + 1)  per key
//              tile.  S = Q K^T takes both operands from shared memory, O += P V takes P from TMEM and V as an
//              MN-major shared-memory operand; all accumulators live in TMEM (S0, S1, O0, O1 = 512 columns);
//   warp 11    scheduler and Q loader: lane 0 claims the next item and hands its description to the others
//              through a ring of three slots; then the warp loads the item's Q tiles (plain tiles for anchor items,
//              row gathers, four rows per lane, for routed ones) into a ring of three tile buffers, so the next
//              item's first query tile is in place before the current item ends.  With short chunks four more warps,
//              12 to 15, load the tiles, 32 rows each.
// Every wait (mbarrier or global counter) is bounded; one that runs out flags the workspace status word and
// the CTA drains its copies and leaves.
#include <algorithm>

#include "moc_common.cuh"
#include "moc_tc.cuh"

namespace moc {

using namespace tc;

struct AttendParams {
    const __nv_bfloat16 *Q;
    __nv_bfloat16 *O;
    float *lse;
    __nv_bfloat16 *part_o;      // [2 or 1] buffers of the group in flight's partials (even / odd groups alternate), laid
                                // out query-innermost in blocks of 128 queries (part_line)
    float *part_lse;            // log-sum-exps of the partials, query-innermost (part_lse_at)
    size_t part_stride;         // elements between the two partial buffers (0 with a single group)
    const KeyRange *chunk_rng;  // [C] key range of a routed item (its chunk)
    const KeyRange *anc_rng;    // merged anchor ranges, indexed by the anchor items
    const WorkItem *ritems;     // routed items of every head, (head, chunk) order
    const WorkItem *aitems;     // anchor items of one head
    const int *tile_off;        // [H C + 1] running count of routed items over (head, chunk)
    const int32_t *qlist;       // [H][cap_total]
    int *queue;
    size_t cap_total;
    int *status;
    int H, L, C, k, hg, n_groups, n_aitems;
    SlotDiv kdiv;
    float scale_log2;           // softmax scale * log2(e)
    uint32_t cookie;
    WaitBound wait;
};

constexpr int kBN = 128;               // keys per tile
constexpr int kThreads = 384;          // three warpgroups: softmax 0, softmax 1, {producer, two MMA issuers, scheduler}
constexpr int kThreadsLoaders = 512;   // ... and a fourth one of Q loaders
constexpr int kTmemCols = 512;         // S0/P0 [0,128) S1/P1 [128,256) O0 [256,384) O1 [384,512)
constexpr int kItemSlots = 3;          // items handed over and not yet seen by every warp (no more than the ROWS_DONE allow)
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kRescaleThreshold = 8.0f;    // log2 units: O is rescaled only when the row max grows by more

enum WaitCode { W_QFULL = 1, W_KFULL, W_VFULL, W_SFULL, W_PFULL, W_OFULL, W_KEMPTY, W_VEMPTY, W_TURN, W_PHALF,
                W_QEMPTY, W_OFREE, W_ITEMFULL, W_ITEMEMPTY, W_ROWSDONE, W_DEPEND, W_MERGE };

// One claimed item, as the scheduler hands it over.
struct ItemSlot {
    int valid;          // 0: the queue is empty, everyone leaves
    int routed, h, first, rows, nrng, ntiles, phase;
    int qbuf;           // Q buffer of its first query tile
    const KeyRange *rng;
};

// Walks the ring of item slots: the slot of an item, and the phase of its barriers.
struct SlotIter {
    int at = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void next() {
        if (++at == kItemSlots) { at = 0; phase ^= 1; }
    }
};

// acc += w x (the bf16 pair u) where cond holds
__device__ __forceinline__ void add_weighted_if(bool cond, uint64_t &acc, uint32_t u, float w) {
    const uint64_t v = pack2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)), w2 = pack2(w, w);
    asm("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t@p fma.rn.f32x2 %0, %1, %2, %0;\n\t}" : "+l"(acc) : "l"(v), "l"(w2), "r"((int)cond));
}

// LOADERS: four more warps load the query tiles, for short routed items (see the rule where the kernel is launched)
template <int D, bool LOADERS>
__global__ void __launch_bounds__(LOADERS ? kThreadsLoaders : kThreads, 1) attend_tc_kernel(const __grid_constant__ CUtensorMap tmQ,
                                                                const __grid_constant__ CUtensorMap tmQrow,
                                                                const __grid_constant__ CUtensorMap tmK,
                                                                const __grid_constant__ CUtensorMap tmV,
                                                                const AttendParams p) {
    constexpr int TILE_BYTES = 128 * D * 2;
    constexpr int SUB = D / 64;            // 64-column (128-byte) sub-tiles per row
    constexpr int SUB_BYTES = 128 * 128;   // one sub-tile: 128 rows of 128 bytes
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[41 + 2 * kItemSlots + 8 * (D == 128 ? 2 : 3)];
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort, s_usable;      // s_usable: the workspace holds this plan's lists
    __shared__ ItemSlot s_item[kItemSlots];

    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    // shared tiles: Q ring of three | K stage 0,1 | V stage 0,1
    const uint32_t sQ = sbase, sK = sbase + 3 * TILE_BYTES, sV = sbase + 5 * TILE_BYTES;
    auto bar = [&](int i) { return smem_u32(&bars[i]); };
    // barrier indices (pairs: per query tile g, per K/V stage, or per item slot)
    constexpr int Q_FULL = 0, Q_EMPTY = 6, K_FULL = 9, K_EMPTY = 11, V_FULL = 13, V_EMPTY = 15, S_FULL = 17, P_HALF = 19, P_FULL = 21,
                  O_FULL = 23, O_FREE = 25, TURN = 27, ROWS_DONE = 29, DEPEND = 37, ITEM_FULL = 38, ITEM_EMPTY = ITEM_FULL + kItemSlots,
                  MERGED = ITEM_EMPTY + kItemSlots, MERGE = MERGED + 3;
    constexpr int kMergeStages = D == 128 ? 2 : 3;                     // blocks of partials under way per softmax warp
    // Registers of a thread after the split; warpgroup by warpgroup they add up to what the launch gave (3 x 168, 4 x 128).  (At
    // d = 64 the issuing warps need more than the loading ones: 210-token chunks, 25 picks 8.54 -> 8.35 ms, a 576-token clip 15.7 ->
    // 15.2 us; at d = 128 within half a per cent.)
    constexpr int kRegsSoftmax = 224, kRegsIssue = !LOADERS ? 56 : D == 64 ? 40 : 32, kRegsLoad = D == 64 ? 24 : 32;
    static_assert(!LOADERS || 2 * kRegsSoftmax + kRegsIssue + kRegsLoad == 512, "setmaxnreg would wait for registers that there are not");
    static_assert(LOADERS || 2 * kRegsSoftmax + kRegsIssue == 504, "setmaxnreg would wait for registers that there are not");
    // Who merges the routed partials how: see the epilogue of the anchor items.
    constexpr bool kMergeInRegs = D == 128 && LOADERS;
    constexpr int kItemReaders = 2 + 2 + 256 + (LOADERS ? 4 : 0);      // producer and bookkeeping lanes, two issuing warps, every softmax thread, loading warps

    if (threadIdx.x == 0) {
        s_abort = s_usable = 0;
        for (int t = 0; t < 3; ++t) {
            // A Q buffer has one full barrier per query tile g, so that each issuer waits for every phase of its own ones: on
            // a shared one, an issuer that leaves out the other's tiles could wait for a buffer whose previous load is still
            // on its way, and take that phase for the one it waits for.
            mbar_init(bar(Q_FULL + t), 1);             // [g][buffer]
            mbar_init(bar(Q_FULL + 3 + t), 1);
            mbar_init(bar(Q_EMPTY + t), 1);
        }
        mbar_init(bar(DEPEND), 1);
        for (int t = 0; t < 2; ++t) {
            mbar_init(bar(K_FULL + t), 1);
            mbar_init(bar(K_EMPTY + t), 2);            // one arrival per MMA issuer
            mbar_init(bar(V_FULL + t), 1);
            mbar_init(bar(V_EMPTY + t), 2);
            mbar_init(bar(S_FULL + t), 1);
            mbar_init(bar(P_HALF + t), 128);
            mbar_init(bar(P_FULL + t), 128);
            mbar_init(bar(O_FULL + t), 1);
            mbar_init(bar(O_FREE + t), 128);
            mbar_init(bar(TURN + t), 128);
        }
        for (int t = 0; t < kItemSlots; ++t) {
            mbar_init(bar(ITEM_FULL + t), 1);
            mbar_init(bar(ITEM_EMPTY + t), kItemReaders);
        }
        for (int t = 0; t < 3; ++t) mbar_init(bar(MERGED + t), 4);            // the softmax warps of the tile
        for (int t = 0; t < 8 * kMergeStages; ++t) mbar_init(bar(MERGE + t), 1);
        for (int t = 0; t < 8; ++t) mbar_init(bar(ROWS_DONE + t), 128);      // [item modulo 4][query tile]
        fence_barrier_init();
    }
    __syncthreads();
    if (warp == 8) {
        tmem_alloc(smem_u32(&tmem_slot), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // Launched early (see moc_common.cuh): barriers and tensor memory are set up while the routing's last launch runs; from
    // here on what it wrote is read.
    previous_done();
    const uint32_t tmem = tmem_slot;
    volatile int *abort_flag = &s_abort;
    int *phase_tab = p.queue + kQueueHeader;
    // Before a query tile is loaded into a buffer (whose last S, Q_EMPTY, is done): the wait for the merge that its previous
    // tile, if it was an anchor item's, did in it; `merges`: so will the tile to be loaded.
    auto merged = [&](int qb, bool merges, uint32_t &used, uint32_t &phase) -> bool {
        if (D != 128 || kMergeInRegs) return true;
        bool done = true;
        if ((used >> qb) & 1) {
            done = mbar_wait(bar(MERGED + qb), (phase >> qb) & 1, abort_flag, p.wait, W_MERGE);
            phase ^= 1u << qb;
        }
        used = (used & ~(1u << qb)) | ((uint32_t)(merges && p.k > 0) << qb);
        return done;
    };

    if (warp < 8) {
        // ------------------------------------------------------------ softmax / epilogue groups
        // the row-per-thread softmax holds a whole 128-key row of S in registers: take the
        // registers the third warpgroup gives up
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
        const int g = warp >> 2;                       // query tile of this group
        const int r = threadIdx.x & 127;               // row within the tile = TMEM lane
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + g * 128 + lane_off, tP = tS, tO = tmem + 256 + g * 128 + lane_off;
        const float c = p.scale_log2;
        // What gives every barrier's phase: of the running counts only the low bits, in one register.  (A row of S fills most of
        // the registers: each one that lives through the loop over the tiles is one the loop lacks.)
        enum : uint32_t { S_ODD = 1, TURN_ODD = 2, TURNED = 4, MINE_ODD = 8, DEP_ODD = 16, MERGE_AT = 5 };      // key tiles; key tiles in
                                                       // two-tile items, any at all; items with this tile; DEPENDs; MERGE phases; from bit 16 on, see `slots`
        uint32_t bits = 0;
        int n_item = 0, last_phase = -1;               // items seen, modulo 12 (three slots, four ROWS_DONE)
        bool ok = true;
        while (ok) {
            const int sl = n_item % kItemSlots;
            ok = mbar_wait(bar(ITEM_FULL + sl), (n_item / kItemSlots) & 1, abort_flag, p.wait, W_ITEMFULL);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const ItemSlot it_ = s_item[sl];
            mbar_arrive(bar(ITEM_EMPTY + sl));
            n_item = n_item == 11 ? 0 : n_item + 1;
            if (!it_.valid) break;
            const int h = it_.h, rows = it_.rows, first = it_.first, group = it_.phase >> 1;
            const bool routed = it_.routed != 0, two = rows > 128;
            // an item that depends on other items' rows (see the bookkeeping lane) is released through DEPEND; the first of a
            // phase speaks for the others
            const bool dep = (routed ? group >= 2 : p.k > 0) && it_.phase != last_phase;
            last_phase = it_.phase;
            const uint32_t dep_phase = (bits & DEP_ODD) ? 1 : 0;
            if (dep) bits ^= DEP_ODD;
            if (g == 1 && !two) {                       // this item has one query tile
                if (dep) {                              // ... and every thread sees every phase of DEPEND
                    ok = mbar_wait(bar(DEPEND), dep_phase, abort_flag, p.wait, W_DEPEND);
                    ok = __all_sync(0xffffffffu, ok);
                    const int b = ROWS_DONE + 2 * ((n_item - 1) & 3) + 1;
                    mbar_arrive(bar(b));
                }
                continue;
            }
            // Row of the tile and of the item.  With four loading warps the rows of an anchor item's tile are dealt to the four
            // softmax warps in equal parts, so that a tile of a few rows keeps all of them busy in the merge.
            const int tile_rows = min(128, rows - g * 128), warp_rows = LOADERS && !routed ? (tile_rows + 3) >> 2 : 32;
            const int row = (warp & 3) * warp_rows + lane, rt = g * 128 + row;
            // the list entry of a routed row is asked for here and looked at in the epilogue
            int qi = -1, entry = -1;
            if (lane < warp_rows && row < tile_rows) {
                if (!routed) qi = first + rt;
                else if (index_ok((size_t)first + rt < p.cap_total, p.status, IX_LIST_POSITION))
                    entry = p.qlist[(size_t)h * p.cap_total + first + rt];
            }
            // partials of the group in flight: even and odd groups alternate between two buffers
            const int h_loc = h - group * p.hg, LB = (p.L + 127) >> 7;
            char *part = reinterpret_cast<char *>(p.part_o + (size_t)(group & 1) * p.part_stride);
            if (!routed && qi >= 0 && p.k > 0) {
                // the epilogue will merge this row's routed partials: start them on their way into L2 now
                // (few picks only: what all CTAs ask for ahead has to stay in L2 until it is read)
                if ((qi & 31) == 0 || lane == 0)
                    for (int s = 0; s < p.k; ++s) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.part_lse + part_lse_at(h, LB, p.k, qi, s)));
                if (p.k <= 8)
                    for (int x = 0; x < p.k * (D / 64); ++x) asm volatile("prefetch.global.L2 [%0];" ::"l"(part + part_line(h_loc, LB, p.k, D / 64, qi, 0) + ((size_t)x << 14)));
            }

            float m_run = -INFINITY, l_run = 0.f;
            TileIter it(it_.rng, it_.nrng);
            int t0, valid, jt = 0;
            while (it.next(t0, valid)) {
                ok = mbar_wait(bar(S_FULL + g), bits & S_ODD, abort_flag, p.wait, W_SFULL);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                uint32_t v[4][32];
#pragma unroll
                for (int ch = 0; ch < 4; ++ch) tmem_ld32(tS + ch * 32, v[ch]);
                tmem_wait_ld();
                if (valid < kBN) {
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch)
#pragma unroll
                        for (int x = 0; x < 32; ++x)
                            if (ch * 32 + x >= valid) v[ch][x] = 0xff800000u;   // -inf
                }
                float m4[4];
#pragma unroll
                for (int ch = 0; ch < 4; ++ch) {
                    m4[ch] = -INFINITY;
#pragma unroll
                    for (int x = 0; x < 32; x += 2) m4[ch] = max3(m4[ch], __uint_as_float(v[ch][x]), __uint_as_float(v[ch][x + 1]));
                }
                // The turn is looked at here and awaited below, where a wait costs some hundred cycles even if it has come.  (At d = 64,
                // where it has rarely come by now, the look cost 2 %; at d = 128, 4 heads of 33k tokens 537 -> 526 us, 2 heads of 42k 411 -> 403,
                // 2 heads of 32k tokens, 512-token chunks, 1273 -> 1255, 24 heads of 33k at the power limit 3.33 -> 3.29 ms.)
                const bool my_turn = D == 128 && (!two || (g == 0 && !(bits & TURNED)) || mbar_test_wait(bar(TURN + (g ^ 1)), ((bits & TURN_ODD) ? 1 : 0) ^ (g == 1 ? 0 : 1)));
                const float m_new = fmaxf(m_run, fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * c);
                float alpha = 1.f;
                if (jt == 0) {
                    m_run = m_new;
                } else if (m_new - m_run > kRescaleThreshold) {
                    alpha = exp2f(m_run - m_new);
                    m_run = m_new;
                }
                // The exponentials of the two query tiles take turns (tile 0 of key tile j, tile 1
                // of j, tile 0 of j + 1, ...): each then has the arithmetic pipes to itself while
                // the other tile's MMAs run, instead of both drifting into lock step.
                // TURN + g is arrived on by group g when all but the last eight of its exponentials of a key tile are done: the
                // hand-over takes about as long as those.  (After the last one instead, with the epilogue as it is now, the same within
                // 0.3 %: 33k-token clip 3.407 and 3.404 ms, d = 64, 725-token frames 643.5 and 643.7 us; at half time it cost 5 %.)  (Tile 0 waits for
                // tile 1's previous turn even at the start of an item: the barrier must never get two phases ahead of
                // a group that has yet to wait on it.)
                if (D == 128 ? !__all_sync(0xffffffffu, my_turn) : two && (g == 1 || (bits & TURNED))) {
                    ok = mbar_wait(bar(TURN + (g ^ 1)), ((bits & TURN_ODD) ? 1 : 0) ^ (g == 1 ? 0 : 1), abort_flag, p.wait, W_TURN);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                }
                if (__any_sync(0xffffffffu, alpha != 1.f)) {
                    // this group's PV of the previous tile has completed (its commit precedes this tile's S)
#pragma unroll 1
                    for (int ch = 0; ch < D / 32; ++ch) {
                        uint32_t o[32];
                        tmem_ld32(tO + ch * 32, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int x = 0; x < 32; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * alpha);
                        tmem_st32(tO + ch * 32, o);
                    }
                }
                // P = exp2(s * c - m), packed bf16 into the P columns (aliasing S).  The first 64 keys
                // are handed to the MMA issuer as soon as they are stored: their P V product overlaps
                // the exponentials of the other 64.
                const uint64_t c2 = pack2(c, c), nm2 = pack2(-m_run, -m_run);
                uint64_t sum_a = 0ull, sum_b = 0ull;   // two packed partial row sums
#pragma unroll
                for (int ch = 0; ch < 4; ++ch) {
                    uint32_t u[16];
#pragma unroll
                    for (int x = 0; x < 16; ++x) {
                        float a0, a1;
                        unpack2(fma2(pack2(__uint_as_float(v[ch][2 * x]), __uint_as_float(v[ch][2 * x + 1])), c2, nm2), a0, a1);
                        a0 = ex2(a0);
                        a1 = ex2(a1);
                        if (x & 1) sum_b = add2(sum_b, pack2(a0, a1));
                        else sum_a = add2(sum_a, pack2(a0, a1));
                        u[x] = bf16x2(a0, a1);
                        if (ch == 3 && x == 11) {
                            // (the compiler must neither put off what comes before nor bring forward what comes after)
                            asm volatile("" ::"r"(u[x]), "r"(u[x - 1]), "r"(u[x - 2]) : "memory");
                            if (two) mbar_arrive(bar(TURN + g));
#pragma unroll
                            for (int y = x + 1; y < 16; ++y) asm volatile("" : "+r"(v[3][2 * y]), "+r"(v[3][2 * y + 1]));
                        }
                    }
                    tmem_st16(tP + ch * 16, u);
                    if (ch == 1) {
                        tmem_wait_st();
                        tc_fence_before();
                        mbar_arrive(bar(P_HALF + g));
                    }
                }
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(bar(P_FULL + g));
                float s0, s1;
                unpack2(add2(sum_a, sum_b), s0, s1);
                l_run = l_run * alpha + (s0 + s1);
                ++jt;
                bits ^= S_ODD;
                if (two) bits = (bits ^ TURN_ODD) | TURNED;
            }
            if (!ok) break;
            // ---- epilogue
            // what follows from the item's fields is worked out anew: kept from before the loop, it would take the loop's registers
            // (d = 64, frames of 725 and 923 tokens: 588 -> 572, 562 -> 552 us)
            int h_ = h, phase_ = it_.phase, first_ = first;
            asm volatile("" : "+r"(h_), "+r"(phase_), "+r"(first_));
            {
            const int h = h_, group = phase_ >> 1, first = first_, h_loc = h - group * p.hg, LB = (p.L + 127) >> 7;
            char *part = reinterpret_cast<char *>(p.part_o + (size_t)(group & 1) * p.part_stride);
            // Results move in the 16 x 256-bit load shape of the tensor memory: of a 16-row half of the warp's rows, lane
            // l holds rows l / 4 and l / 4 + 8, of every eight columns the two at 2 (l % 4).  Four lanes then write 128
            // contiguous bytes of a row.  (A row per lane, 32 bytes at a time, a warp's store touched 32 lines, and the 64 of
            // an item's partials kept the memory pipe busy for some 4000 cycles.)  A partial is stored with its columns in
            // the order of the lanes; only O, in the end, is put in the order of the columns.
            constexpr int CB = D / 64;                  // 64-column blocks
            const int l4 = lane >> 2, l2 = lane & 3;
            const float inv_l = 1.f / l_run;
            const float lse_own = (m_run + log2f(l_run)) * kLn2;
            // what this item depends on (an anchor item: the routed items of its group have stored all their partials;
            // a routed item: the anchor items two groups back have read the buffer it is about to store into) has been
            // awaited by the bookkeeping lane, which then arrives on DEPEND, once per phase of the queue
            if (dep) {
                ok = mbar_wait(bar(DEPEND), dep_phase, abort_flag, p.wait, W_DEPEND);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
            }
            if (routed) {
                size_t line = 0;                        // where this row's partial goes
                bool keep = false;
                if (g * 128 + r < rows) {
                    const int q = p.kdiv.query(entry), slot = entry - q * p.k;
                    (void)index_ok(entry >= 0 && q < p.L, p.status, IX_LIST_ENTRY);
                    if (entry >= 0 && q < p.L) {         // never follow an entry that is not a row of this head
                        line = part_line(h_loc, LB, p.k, CB, q, slot);
                        keep = true;
                        p.part_lse[part_lse_at(h, LB, p.k, q, slot)] = lse_own;
                    }
                }
                ok = mbar_wait(bar(O_FULL + g), (bits & MINE_ODD) ? 1 : 0, abort_flag, p.wait, W_OFULL);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                uint32_t o[2 * CB][32];
#pragma unroll
                for (int x = 0; x < 2 * CB; ++x) tmem_ld_16x256b(tO + ((x / CB) << 20) + (x % CB) * 64, o[x]);
                tmem_wait_ld();
                tc_fence_before();
                mbar_arrive(bar(O_FREE + g));            // the issuer may start the next item's P V (which overwrites O)
#pragma unroll
                for (int j = 0; j < 4; ++j) {            // rows 8 j + l4 of the warp's 32
                    const float w = __shfl_sync(0xffffffffu, inv_l, j * 8 + l4);
                    const size_t at = __shfl_sync(0xffffffffu, line, j * 8 + l4);
                    const bool some = __shfl_sync(0xffffffffu, keep, j * 8 + l4);
                    const int q7 = (int)(at >> 7) & 7;       // the query modulo 8
                    char *dst = part + at + ((kMergeInRegs ? l2 : l2 ^ (q7 >> 1)) << 5);
#pragma unroll
                    for (int cb = 0; cb < CB; ++cb) {
                        const uint32_t (&v)[32] = o[(j >> 1) * CB + cb];
                        uint32_t u[8];
#pragma unroll
                        for (int x = 0; x < 8; ++x)
                            u[x] = bf16x2(__uint_as_float(v[4 * x + 2 * (j & 1)]) * w, __uint_as_float(v[4 * x + 2 * (j & 1) + 1]) * w);
                        if (!kMergeInRegs && (q7 & 1)) {
#pragma unroll
                            for (int x = 0; x < 4; ++x) { const uint32_t t = u[x]; u[x] = u[4 + x]; u[4 + x] = t; }
                        }
                        if (some) st_256(dst + (cb << 14), u);
                    }
                }
            } else {
                // The weights of the merge depend only on log-sum-exps: have their sum ready before the last P V lands.  Slot s of
                // this lane's row counts exp(lse_s - big), its own part exp(lse_own - big) / l, and the sum is divided by wsum.
                float big = lse_own, wsum = 1.f;
                const bool merge = qi >= 0 && p.k > 0;
                const float *pl = p.part_lse + part_lse_at(h, LB, p.k, max(qi, 0), 0);        // slot s: pl[s * 128]
                // How the partials come.  With one loading warp, and at d = 64: by bulk copies, a 64-column block of one slot of the
                // warp's 32 rows at a time, into the query tile's buffer, whose last S is done (at d = 64, where there is room, into
                // space of the warp's own), two or three under way.  With short chunks at d = 128, where a row has many picks: by
                // loads into registers, 400 to 800 bytes a thread under way, in the shape in which the partials are stored.  (Cycles
                // for the epilogue of 256 rows, the loads of a row by its own thread before -> this: d = 128, 4 picks 15000 -> 13700 by
                // copies, 22900 by register loads; d = 64, 25 picks 38500 -> 33000, 56900; the whole launch on 256-token chunks, 30 picks,
                // 18.8 -> 13.8 ms by register loads, 15.2 by copies.)
                const int tile_rows = min(128, rows - g * 128), warp_rows = LOADERS ? (tile_rows + 3) >> 2 : 32;
                const int q0 = first + g * 128 + (warp & 3) * warp_rows, n_rows = min(warp_rows, first + g * 128 + tile_rows - q0);   // the warp's rows
                // Slots up to the last one that a row of the warp uses: early in a stream, and wherever rows may route to few chunks, most of
                // many are empty.  (All k slots -> these: 3 heads of 2.2k tokens, 512-token chunks, 30 picks 59.6 -> 43.4 us, d = 64 44.4 ->
                // 29.5; 12 heads of 66k tokens, 800-token chunks, 30 picks 11.41 -> 10.94 ms; with all in use within 2 %.)
                int n_slots = p.k, used = 0;
                const int qb = it_.qbuf + g < 3 ? it_.qbuf + g : it_.qbuf + g - 3;
                const uint32_t m_base = D == 128 ? sQ + qb * TILE_BYTES + (warp & 3) * (TILE_BYTES / 4) : sbase + 7 * TILE_BYTES + warp * (kMergeStages * 4096);
                int m_st = 0, m_next = 0, m_flight = 0;          // stage to read, block to ask for, blocks under way
                int c_st = 0, c_slot = 0, c_cb = 0;
                auto copy_next = [&]() {                         // the warp's next block
                    if (lane == 0) {
                        const uint32_t b = bar(MERGE + warp * kMergeStages + c_st), dst = m_base + c_st * 4096;
                        const int n1 = min(n_rows, 128 - (q0 & 127));        // rows in the first block of 128 queries
                        mbar_expect_tx(b, n_rows * 128);
                        bulk_load(dst, part + part_line(h_loc, LB, p.k, CB, q0, c_slot) + ((size_t)c_cb << 14), n1 * 128, b);
                        if (n1 < n_rows)
                            bulk_load(dst + n1 * 128, part + part_line(h_loc, LB, p.k, CB, q0 + n1, c_slot) + ((size_t)c_cb << 14), (n_rows - n1) * 128, b);
                    }
                    ++m_next;
                    ++m_flight;
                    if (++c_st == kMergeStages) c_st = 0;
                    if (++c_slot == n_slots) { c_slot = 0; ++c_cb; }
                };
                if (!kMergeInRegs && n_rows > 0 && p.k > 0) {
                    // other CTAs' stores, seen through DEPEND by the generic proxy, are read by the copy engine
                    if (lane == 0) asm volatile("fence.proxy.async;" ::: "memory");
                    for (int x = 0; x < kMergeStages && x < CB * p.k; ++x) copy_next();
                }
                if (merge) {
                    // eight slots requested together; running maximum and sum
#pragma unroll 1
                    for (int s0 = 0; s0 < p.k; s0 += 8) {
                        float plv[8], m = big;
#pragma unroll
                        for (int u = 0; u < 8; ++u) plv[u] = s0 + u < p.k ? __ldcg(pl + (s0 + u) * 128) : -INFINITY;
#pragma unroll
                        for (int u = 0; u < 8; ++u) m = fmaxf(m, plv[u]);
                        wsum *= __expf(big - m);
                        big = m;
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            wsum += __expf(plv[u] - big);
                            if (plv[u] != -INFINITY) used = s0 + u + 1;
                        }
                    }
                }
                if (kMergeInRegs) {
                    bits = (bits & 0xffff) | (uint32_t)__reduce_max_sync(0xffffffffu, used) << 16;
                } else {                                         // (the first few have been asked for already)
                    n_slots = max(__reduce_max_sync(0xffffffffu, used), min(kMergeStages, p.k));
                    if (c_slot >= n_slots) { c_slot = 0; ++c_cb; }
                    if (n_rows <= 0) n_slots = 0;
                }
                const float inv_w = 1.f / wsum, w_own = __expf(lse_own - big) * inv_l;
                if constexpr (kMergeInRegs) {
                    // Passes of eight of the warp's rows over the slots, a few at a time: the loads of the next few are on their way
                    // while these are added up.
                    constexpr int B = 3;
                    // The slots in use are kept beside the phases and taken out where they are wanted: in a register of their own, or as the
                    // bound of the loops (whose counters then are not the whole warp's), they made the loop over the tiles spill.
                    auto slots = [&]() __attribute__((always_inline)) {
                        int n;
                        asm volatile("shr.u32 %0, %1, 16;" : "=r"(n) : "r"(bits));
                        return n;
                    };
                    const int row0 = q0 + l4, row_end = q0 + n_rows, n_pass = max(1, (n_rows + 7) >> 3);
                    struct Batch { uint32_t v[B][CB][8]; float ls[B]; };
                    int ask_pass = 0, ask_s = 0;
                    auto ask = [&](Batch &b) __attribute__((always_inline)) {
                        const int q = row0 + ask_pass * 8;
                        const bool in = q < row_end;
                        const int n = slots();
                        const char *src = part + part_line(h_loc, LB, p.k, CB, q, ask_s) + l2 * 32;
                        const float *ls = p.part_lse + part_lse_at(h, LB, p.k, q, ask_s);
#pragma unroll
                        for (int u = 0; u < B; ++u) {
                            const bool some = in && ask_s + u < n;
                            const float x = __ldcg(some ? ls + u * 128 : pl);
                            b.ls[u] = some ? x : -INFINITY;
#pragma unroll
                            for (int cb = 0; cb < CB; ++cb) ld_cg_256_if(some, src + ((size_t)(u * CB + cb) << 14), b.v[u][cb]);
                        }
                        ask_s += B;
                        if (ask_s >= p.k) { ask_s = 0; ++ask_pass; }
                    };
                    uint64_t acc[CB][8];
                    int pass = 0, s0 = 0;
                    float row_big = 0.f;
                    auto add = [&](const Batch &b) __attribute__((always_inline)) {
                        const int src_lane = pass * 8 + l4;
                        if (s0 == 0) {
                            row_big = __shfl_sync(0xffffffffu, big, src_lane);
                            const float w = __shfl_sync(0xffffffffu, w_own, src_lane);
                            const uint64_t w2 = pack2(w, w);
#pragma unroll
                            for (int cb = 0; cb < CB; ++cb) {
                                uint32_t o[32];
                                tmem_ld_16x256b(tO + ((pass >> 1) << 20) + cb * 64, o);
                                tmem_wait_ld();
#pragma unroll
                                for (int x = 0; x < 8; ++x)
                                    acc[cb][x] = mul2(pack2(__uint_as_float((pass & 1) ? o[x * 4 + 2] : o[x * 4]), __uint_as_float((pass & 1) ? o[x * 4 + 3] : o[x * 4 + 1])), w2);
                            }
                            if (pass == n_pass - 1) {
                                // O has been read: the issuer may start the next item's P V (which overwrites it)
                                tc_fence_before();
                                mbar_arrive(bar(O_FREE + g));
                            }
                        }
                        if (s0 < slots()) {
#pragma unroll
                            for (int u = 0; u < B; ++u) {
                                // exp(-inf) = 0: an empty slot, and what its place holds is not a number to use.  (Formed as for wsum: with
                                // big * log2(e) rounded beforehand the weights of scores around 1e5 did not sum to one.)
                                const float w = __expf(b.ls[u] - row_big);
#pragma unroll
                                for (int cb = 0; cb < CB; ++cb)
#pragma unroll
                                    for (int x = 0; x < 8; ++x) add_weighted_if(w != 0.f, acc[cb][x], b.v[u][cb][x], w);
                            }
                        }
                        s0 += B;
                        if (s0 >= p.k) {
                            const float w = __shfl_sync(0xffffffffu, inv_w, src_lane);
                            const int q = row0 + pass * 8;
#pragma unroll
                            for (int cb = 0; cb < CB; ++cb) {
                                uint32_t u[8];
#pragma unroll
                                for (int x = 0; x < 8; ++x) {
                                    float lo, hi;
                                    unpack2(acc[cb][x], lo, hi);
                                    u[x] = bf16x2(lo * w, hi * w);
                                }
                                quad_transpose(u, l2);
                                if (q < row_end) store_quad(p.O + ((size_t)h * p.L + q) * D + cb * 64, l2, u);
                            }
                            s0 = 0;
                            ++pass;
                        }
                    };
                    Batch even = {}, odd = {};
                    ask(even);
                    ok = mbar_wait(bar(O_FULL + g), (bits & MINE_ODD) ? 1 : 0, abort_flag, p.wait, W_OFULL);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll 1
                    while (true) {                               // (past the last pass no row is asked for)
                        ask(odd);
                        add(even);
                        if (pass == n_pass) break;
                        ask(even);
                        add(odd);
                        if (pass == n_pass) break;
                    }
                } else {
                    ok = mbar_wait(bar(O_FULL + g), (bits & MINE_ODD) ? 1 : 0, abort_flag, p.wait, W_OFULL);
                    ok = __all_sync(0xffffffffu, ok);
                    tc_fence_after();
                    float ls1 = merge ? __ldcg(pl) : -INFINITY, ls2 = merge ? __ldcg(pl + min(1, p.k - 1) * 128) : -INFINITY;      // the next two slots'
                    const int row7 = (q0 + lane) & 7;
#pragma unroll 1
                    for (int cb = 0; ok && cb < CB; ++cb) {
                        uint64_t acc[32];                            // columns 2 x, 2 x + 1 of the block
                        const uint64_t w2 = pack2(w_own, w_own);
#pragma unroll
                        for (int x = 0; x < 2; ++x) {
                            uint32_t o[32];
                            __syncwarp();
                            tmem_ld32(tO + cb * 64 + x * 32, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int y = 0; y < 16; ++y) acc[x * 16 + y] = mul2(pack2(__uint_as_float(o[2 * y]), __uint_as_float(o[2 * y + 1])), w2);
                        }
                        if (cb == CB - 1) {
                            // O has been read: the issuer may start the next item's P V (which overwrites it)
                            tc_fence_before();
                            mbar_arrive(bar(O_FREE + g));
                        }
#pragma unroll 1
                        for (int s = 0; s < n_slots; ++s) {
                            const float w = __expf(ls1 - big);       // as for wsum; exp(-inf) = 0: an empty slot
                            ls1 = ls2;
                            const int s2 = s + 2 < n_slots ? s + 2 : s + 2 - n_slots;       // (the next block's first slots after the last)
                            ls2 = merge ? __ldcg(pl + min(s2, p.k - 1) * 128) : -INFINITY;
                            ok = mbar_wait(bar(MERGE + warp * kMergeStages + m_st), (bits >> (MERGE_AT + m_st)) & 1, abort_flag, p.wait, W_MERGE);
                            ok = __all_sync(0xffffffffu, ok);
                            if (!ok) break;
                            const uint32_t src = m_base + m_st * 4096 + lane * 128;
#pragma unroll
                            for (int c16 = 0; c16 < 8; ++c16) {
                                // what an empty slot's place holds is not a number to use
                                uint32_t v[4];
                                ld_shared_128(src + ((c16 ^ row7) << 4), v);
#pragma unroll
                                for (int y = 0; y < 4; ++y) add_weighted_if(w != 0.f, acc[((c16 & 1) * 4 + y) * 4 + (c16 >> 1)], v[y], w);
                            }
                            __syncwarp();
                            bits ^= 1u << (MERGE_AT + m_st);
                            --m_flight;
                            if (m_next < CB * n_slots) copy_next();
                            if (++m_st == kMergeStages) m_st = 0;
                        }
                        if (ok && qi >= 0) {
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                uint32_t u[8];
#pragma unroll
                                for (int y = 0; y < 8; ++y) {
                                    float lo, hi;
                                    unpack2(acc[x * 8 + y], lo, hi);
                                    u[y] = bf16x2(lo * inv_w, hi * inv_w);
                                }
                                uint4 *dst = reinterpret_cast<uint4 *>(p.O + ((size_t)h * p.L + qi) * D + cb * 64 + x * 16);
                                dst[0] = make_uint4(u[0], u[1], u[2], u[3]);     // (O is 16-byte aligned, not 32)
                                dst[1] = make_uint4(u[4], u[5], u[6], u[7]);
                            }
                        }
                    }
                    if (!ok) {       // copies under way must land before the shared memory is released
                        int dummy_flag = 0;
                        for (; m_flight > 0; --m_flight) {
                            mbar_wait(bar(MERGE + warp * kMergeStages + m_st), (bits >> (MERGE_AT + m_st)) & 1, &dummy_flag, p.wait, W_MERGE);
                            bits ^= 1u << (MERGE_AT + m_st);
                            if (++m_st == kMergeStages) m_st = 0;
                        }
                        break;
                    }
                    if (D == 128 && p.k > 0) {                   // the Q buffer is no longer in use
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar(MERGED + qb));
                    }
                }
                if (qi >= 0) p.lse[(size_t)h * p.L + qi] = merge ? big + __logf(wsum) : lse_own;
            }
            }
            // this tile's rows are stored; the bookkeeping lane counts them once all 128 threads are here
            mbar_arrive(bar(ROWS_DONE + 2 * ((n_item - 1) & 3) + g));
            bits ^= MINE_ODD;
        }
    } else if (warp == 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
        if (lane == 0) {
            // ------------------------------------------------------------ TMA producer of the K and V tiles
            prefetch_tensormap(&tmK);
            prefetch_tensormap(&tmV);
            int n_kv = 0;                                     // K/V tiles issued
            SlotIter slot_it;
            int k_last = -1, v_last = -1;                     // last tile whose K / V copy was issued
            bool ok = true;
            while (ok) {
                if (!mbar_wait(bar(ITEM_FULL + slot_it.at), slot_it.phase, abort_flag, p.wait, W_ITEMFULL)) break;
                const ItemSlot it_ = s_item[slot_it.at];
                mbar_arrive(bar(ITEM_EMPTY + slot_it.at));
                slot_it.next();
                if (!it_.valid) break;
                const int h = it_.h;
                // the ring of stages runs on from the previous item
                TileIter it(it_.rng, it_.nrng);
                int t0, valid;
                while (it.next(t0, valid)) {
                    const int st = n_kv & 1;
                    const uint32_t ph = (n_kv >> 1) & 1;
                    if (!mbar_wait(bar(K_EMPTY + st), ph ^ 1, abort_flag, p.wait, W_KEMPTY)) { ok = false; break; }
                    mbar_expect_tx(bar(K_FULL + st), TILE_BYTES);
#pragma unroll
                    for (int sub = 0; sub < SUB; ++sub)
                        tma_load_2d(sK + st * TILE_BYTES + sub * SUB_BYTES, &tmK, sub * 64, h * p.L + t0, bar(K_FULL + st));
                    k_last = n_kv;
                    if (!mbar_wait(bar(V_EMPTY + st), ph ^ 1, abort_flag, p.wait, W_VEMPTY)) { ok = false; break; }
                    mbar_expect_tx(bar(V_FULL + st), TILE_BYTES);
#pragma unroll
                    for (int sub = 0; sub < SUB; ++sub)
                        tma_load_2d(sV + st * TILE_BYTES + sub * SUB_BYTES, &tmV, sub * 64, h * p.L + t0, bar(V_FULL + st));
                    v_last = n_kv;
                    ++n_kv;
                }
            }
            if (*abort_flag) {
                // drain: copies already issued must land before the CTA's shared memory is released
                int dummy_flag = 0;
                for (int b = 0; b < 2; ++b) {
                    const int kj = k_last - b, vj = v_last - b;
                    if (kj >= 0) mbar_wait(bar(K_FULL + (kj & 1)), (kj >> 1) & 1, &dummy_flag, p.wait, W_KFULL);
                    if (vj >= 0) mbar_wait(bar(V_FULL + (vj & 1)), (vj >> 1) & 1, &dummy_flag, p.wait, W_VFULL);
                }
            }
        } else if (lane == 16) {
            // ------------------------------------------------------------ bookkeeping, item by item:
            // first what the item depends on - an anchor item: the routed items of its group have stored all their
            // partials; a routed item: the anchor items two groups back have read the buffer it will store into -
            // then, when the softmax groups have stored the item's rows, the rows join the phase's count.  The
            // groups' arrivals order their stores before this thread (CTA scope); its fence makes them visible
            // device-wide before the count moves.
            // An item that depends on nothing does not go through DEPEND at all, and of a phase's items only the first does: what
            // it waited for stays true.  DEPEND is arrived on when the previous item's rows have been seen to be stored, that is after
            // every softmax thread has passed its previous wait on it (a group without a tile in that item waits, and arrives
            // on ROWS_DONE, all the same).
            // The device-wide fence before the count waits for every store in flight, with short items longer than an item
            // takes.  So an item's slot is handed back before it, and the rows of a few items are counted together: at the end of a
            // phase, before a wait, and else every fourth item (with the ring of three slots, before the epilogue was cut: 256-token
            // chunks, 118 picks 23.1 -> 22.3 ms, 30 picks 18.4 -> 17.9).
            // A barrier must not complete two phases that nobody has waited for in between: the slot of item n + 1 is handed
            // back when item n has been seen to be stored, and item n + 4, the next to use the ROWS_DONE of item n, goes into that
            // slot.
            SlotIter slot_it;
            int n_item = 0, last_phase = -1;
            uint32_t rows_phase = 0;                            // bit 2 (item modulo 4) + tile: parity of the next phase of that ROWS_DONE
            int pend_tiles = 0, pend_item_rows = 0;             // the item before this one: barriers to wait for, rows
            int pend_phase = -1, pend_rows = 0, pend_n = 0;     // rows stored and not yet counted, of how many items
            auto count_rows = [&]() {
                if (pend_n == 0) return;
                __threadfence();
                atomicAdd(&phase_tab[3 * pend_phase + 2], pend_rows);
                pend_n = pend_rows = 0;
            };
            bool ok = true;
            while (ok) {
                const int sl = slot_it.at;
                if (!mbar_wait(bar(ITEM_FULL + sl), slot_it.phase, abort_flag, p.wait, W_ITEMFULL)) break;
                const ItemSlot it_ = s_item[sl];
                slot_it.next();
                ++n_item;
                for (int g = 0; ok && g < pend_tiles; ++g) {
                    const int b = 2 * ((n_item - 2) & 3) + g;          // the pending item is the one before this
                    ok = mbar_wait(bar(ROWS_DONE + b), (rows_phase >> b) & 1, abort_flag, p.wait, W_ROWSDONE);
                    rows_phase ^= 1u << b;
                }
                if (!ok) break;
                mbar_arrive(bar(ITEM_EMPTY + sl));
                if (pend_tiles) {
                    pend_rows += pend_item_rows;
                    ++pend_n;
                }
                const int group = it_.phase >> 1;
                const bool first = it_.valid && it_.phase != last_phase;
                const bool dep_anchor = first && !it_.routed && p.k > 0, dep_routed = first && it_.routed && group >= 2;
                if (!it_.valid || first || pend_n >= 4) count_rows();
                if (!it_.valid) break;
                if (dep_anchor)
                    ok = wait_count(&phase_tab[3 * (2 * group) + 2], phase_tab[3 * (2 * group) + 1], abort_flag, p.wait, W_DEPEND);
                if (dep_routed)
                    ok = wait_count(&phase_tab[3 * (2 * (group - 2) + 1) + 2], phase_tab[3 * (2 * (group - 2) + 1) + 1], abort_flag, p.wait, W_DEPEND);
                if (!ok) break;
                if (dep_anchor || dep_routed) {
                    __threadfence();
                    mbar_arrive(bar(DEPEND));
                }
                pend_phase = last_phase = it_.phase;
                pend_item_rows = it_.rows;
                pend_tiles = it_.rows > 128 || dep_anchor || dep_routed ? 2 : 1;
            }
        }
    } else if (warp < 11) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
        // ------------------------------------------------------------ MMA issuers (one warp per query tile; the warp stays
        // together, one lane of it issues)
        const int g = uniform(warp - 9);
        {
            constexpr uint32_t IDESC_PV = idesc_bf16_f32(128, D, 0, 1);
            // Descriptors are built once; inside the issue loops only the 14-bit start-address field
            // (low word, 16-byte units) moves, so one tcgen05.mma costs the issuing warp a few
            // integer instructions.
            const uint64_t q_desc0 = smem_desc_sw128(sQ, 16, 1024), k_desc0 = smem_desc_sw128(sK, 16, 1024);
            const uint64_t v_desc0 = smem_desc_sw128(sV, SUB_BYTES, 1024);
            constexpr uint64_t STAGE = TILE_BYTES >> 4;   // next tile / next stage, in address-field units
            int qb = 0;                                   // Q buffer of this tile in the current item
            auto issue_qk = [&](int st, int valid) {
                const int n_qk = max(16, (valid + 15) & ~15);
                const uint32_t idesc_qk = idesc_bf16_f32(128, n_qk, 0, 0);
                const uint64_t qd = q_desc0 + qb * STAGE, kd = k_desc0 + (st ? STAGE : 0);
                const uint32_t q_lo = (uint32_t)qd, q_hi = (uint32_t)(qd >> 32), k_lo = (uint32_t)kd, k_hi = (uint32_t)(kd >> 32);
                const uint32_t d_s = tmem + g * 128;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    const uint32_t o = ((ks >> 2) * SUB_BYTES + (ks & 3) * 32) >> 4;     // never carries out of the address field
                    mma_ss_elect(d_s, q_lo + o, q_hi, k_lo + o, k_hi, idesc_qk, ks > 0);
                }
            };
            // k-steps [ks0, ks1) of  O_g += P_g V(stage st)  (16 keys each)
            auto issue_pv = [&](int st, int ks0, int ks1, bool accumulate) {
                const uint64_t vd = v_desc0 + (st ? STAGE : 0);
                const uint32_t v_lo = (uint32_t)vd, v_hi = (uint32_t)(vd >> 32);
                const uint32_t d_o = tmem + 256 + g * 128, a_p = tmem + g * 128;
                if (ks1 - ks0 == 4) {
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        mma_ts_elect(d_o, a_p + (ks0 + ks) * 8, v_lo + (ks0 + ks) * (2048 >> 4), v_hi, IDESC_PV, accumulate || ks > 0);
                } else {
                    for (int ks = ks0; ks < ks1; ++ks) mma_ts_elect(d_o, a_p + ks * 8, v_lo + ks * (2048 >> 4), v_hi, IDESC_PV, accumulate || ks > ks0);
                }
            };
            // items with this tile, K/V tiles seen, P tiles consumed, query tiles loaded before this item
            int n_mine = 0, n_kv = 0, n_p = 0, n_qtile = 0;
            uint32_t q_phase = 0;                         // bit b: parity of the next load of this tile into buffer b
            bool ok = true;
            // the whole warp waits, and goes on or gives up together
            auto wait = [&](int b, uint32_t parity, int code) {
                // (with the loaders' traffic on every scheduler a parked issuer wakes later still: it polls)
                return __all_sync(0xffffffffu, LOADERS ? mbar_wait_spin(bar(b), parity, abort_flag, p.wait, code)
                                                       : mbar_wait(bar(b), parity, abort_flag, p.wait, code)) != 0;
            };
            SlotIter slot_it;
            while (ok) {
                const int sl = slot_it.at;
                if (!wait(ITEM_FULL + sl, slot_it.phase, W_ITEMFULL)) break;
                const ItemSlot it_ = s_item[sl];
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(ITEM_EMPTY + sl));
                slot_it.next();
                if (!uniform(it_.valid)) break;
                const int rows = uniform(it_.rows), n_tiles = uniform(it_.ntiles);
                const int q_seq = n_qtile + g;                      // this tile's place in the sequence of Q loads
                n_qtile += rows > 128 ? 2 : 1;
                if (g == 1 && rows <= 128) {
                    // no second query tile: this issuer only keeps the K/V ring's accounting (each stage is
                    // released by two arrivals)
                    for (int jt = 0; ok && jt < n_tiles; ++jt) {
                        const int st = n_kv & 1;
                        const uint32_t ph = (n_kv >> 1) & 1;
                        ok = wait(K_FULL + st, ph, W_KFULL) && wait(V_FULL + st, ph, W_VFULL);
                        if (!ok) break;
                        if (lane == 0) {
                            mbar_arrive(bar(K_EMPTY + st));
                            mbar_arrive(bar(V_EMPTY + st));
                        }
                        ++n_kv;
                    }
                    continue;
                }
                qb = q_seq % 3;
                // this issuer serves query tile g: S_g(0), then per key tile  O_g += P_g V(j),  S_g(j + 1)
                TileIter it(it_.rng, it_.nrng);
                int t0, valid, valid_next = 0;
                ok = it.next(t0, valid);
                valid = uniform(valid);
                ok = ok && wait(Q_FULL + 3 * g + qb, (q_phase >> qb) & 1, W_QFULL);
                q_phase ^= 1u << qb;
                ok = ok && wait(K_FULL + (n_kv & 1), (n_kv >> 1) & 1, W_KFULL);
                if (!ok) break;
                tc_fence_after();
                issue_qk(n_kv & 1, valid);
                tc_commit_elect(bar(S_FULL + g));
                tc_commit_elect(bar(K_EMPTY + (n_kv & 1)));
                if (n_tiles == 1) tc_commit_elect(bar(Q_EMPTY + qb));       // that was the item's only S: its Q buffer may be refilled
                for (int jt = 0; ok && jt < n_tiles; ++jt) {
                    const int st = n_kv & 1, sn = (n_kv + 1) & 1;
                    const uint32_t ph = (n_kv >> 1) & 1, phn = ((n_kv + 1) >> 1) & 1;
                    const bool more = jt + 1 < n_tiles;
                    if (more) { it.next(t0, valid_next); valid_next = uniform(valid_next); }
                    if (!wait(V_FULL + st, ph, W_VFULL)) { ok = false; break; }
                    if (more && !wait(K_FULL + sn, phn, W_KFULL)) { ok = false; break; }
                    const int steps = (valid + 15) >> 4, half = min(steps, 4);
                    if (!wait(P_HALF + g, n_p & 1, W_PHALF)) { ok = false; break; }
                    // the first P V of an item overwrites O: the previous item's epilogue must have read it
                    if (jt == 0 && n_mine > 0 && !wait(O_FREE + g, (n_mine - 1) & 1, W_OFREE)) { ok = false; break; }
                    tc_fence_after();
                    issue_pv(st, 0, half, jt > 0);
                    if (!wait(P_FULL + g, n_p & 1, W_PFULL)) { ok = false; break; }
                    tc_fence_after();
                    if (steps > half) issue_pv(st, half, steps, true);
                    // a commit between two groups of MMAs leaves the pipe idle: the next S goes out first, then all commits
                    if (more) {
                        issue_qk(sn, valid_next);
                        tc_commit_elect(bar(S_FULL + g));
                        tc_commit_elect(bar(V_EMPTY + st));
                        tc_commit_elect(bar(K_EMPTY + sn));
                        if (jt + 2 == n_tiles) tc_commit_elect(bar(Q_EMPTY + qb));      // the item's last S: its Q buffer may be refilled
                    } else {
                        tc_commit_elect(bar(V_EMPTY + st));
                        tc_commit_elect(bar(O_FULL + g));
                    }
                    valid = valid_next;
                    ++n_kv;
                    ++n_p;
                }
                ++n_mine;
            }
        }
    } else if (!LOADERS || warp == 11) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
        // ------------------------------------------------------------ scheduler (lane 0 claims items in queue order) and
        // Q loader (the whole warp): a claimed item is published at once, then its query tiles are loaded as their
        // buffers come free, which for the first tile is before the previous item has finished
        bool usable = false;
        int total = 0, n_phases = 0;
        if (lane == 0) {
            usable = *(volatile int *)p.status == 0 && (uint32_t)((volatile int *)p.status)[ST_COOKIE] == p.cookie;
            if (!usable) atomicCAS(p.status, 0, MOC_ERR_WORKSPACE);      // not this plan's lists: report, touch nothing else
            s_usable = usable;
            total = usable ? p.queue[1] : 0;
            n_phases = p.queue[2];
            prefetch_tensormap(&tmQ);
            prefetch_tensormap(&tmQrow);
        }
        int n_item = 0, n_qtile = 0, last_g = 0;       // last_g: query tile of the last one loaded or published
        uint32_t q_phase = 0;                          // bit 3 g + buffer: parity of the next phase of that Q_FULL
        uint32_t m_used = 0, m_phase = 0;              // bit b: buffer b's tile merges partials in it; parity of the next phase of its MERGED
        bool ok = true, late = false;
        SlotIter slot_it;
        while (ok) {
            const int sl = slot_it.at;
            ItemSlot s;
            s.valid = 0; s.routed = 0; s.h = 0; s.first = 0; s.rows = 0; s.nrng = 0; s.ntiles = 0; s.phase = 0; s.qbuf = n_qtile % 3; s.rng = nullptr;
            if (lane == 0) {
                if (n_item >= kItemSlots) ok = mbar_wait(bar(ITEM_EMPTY + sl), slot_it.phase ^ 1, abort_flag, p.wait, W_ITEMEMPTY);
                // Claimed early, an item's gathers are done before they are needed, but it is kept from a CTA that may be idle.
                // After an anchor item (whose successors have plain tiles to load, and which end the queue), and when there
                // are only a few items per CTA, the next one is claimed when the last S of this one has been issued.
                const bool wait_for_s = n_qtile > 0 && (late || total <= 2 * (int)gridDim.x);
                if (ok && wait_for_s && n_item >= 2) {       // every warp has seen the item before the last one
                    const bool wrap = sl + 1 == kItemSlots;
                    ok = mbar_wait(bar(ITEM_EMPTY + (wrap ? 0 : sl + 1)), slot_it.phase ^ (wrap ? 0 : 1), abort_flag, p.wait, W_ITEMEMPTY);
                }
                if (ok && wait_for_s) {
                    const int qb = (n_qtile - 1) % 3, qf = 3 * last_g + qb;
                    // Where others load the tiles, the buffer's release before this one may be yet to come, and its phase would be
                    // taken for this one's.  It has come when the item's last tile is there.  (That barrier's own phase
                    // before was of an item that the softmax warps have left, and the next is of one not yet published.)
                    if (LOADERS) ok = mbar_wait(bar(Q_FULL + qf), ((q_phase >> qf) & 1) ^ 1, abort_flag, p.wait, W_QFULL);
                    ok = ok && mbar_wait(bar(Q_EMPTY + qb), ((n_qtile - 1) / 3) & 1, abort_flag, p.wait, W_QEMPTY);
                }
                const int t = (ok && usable && !*abort_flag && *(volatile int *)p.status == 0) ? atomicAdd(&p.queue[0], 1) : total;
                if (t < total) {
                    int ph = 0;
                    while (ph + 1 < n_phases && phase_tab[3 * (ph + 1)] <= t) ++ph;
                    const int local = t - phase_tab[3 * ph], group = ph >> 1, h0 = group * p.hg;
                    WorkItem w;
                    s.routed = (ph & 1) == 0;
                    if (s.routed) {
                        w = p.ritems[p.tile_off[(size_t)h0 * p.C] + local];
                        s.h = w.h;
                        s.rng = p.chunk_rng + w.rng_off;
                    } else {
                        w = p.aitems[local % p.n_aitems];
                        s.h = h0 + local / p.n_aitems;
                        s.rng = p.anc_rng + w.rng_off;
                    }
                    s.first = w.first; s.rows = w.rows; s.nrng = w.nrng; s.ntiles = w.ntiles; s.phase = ph;
                    s.valid = 1;
                    if (s.routed && !index_ok((unsigned)w.h < (unsigned)p.H && w.rows > 0 && w.rows <= kQTileRows && w.first >= 0 &&
                                              (size_t)w.first + w.rows <= p.cap_total && w.nrng == 1, p.status, IX_ITEM_FIELDS))
                        s.valid = 0;
                }
                s_item[sl] = s;
                __threadfence_block();
                mbar_arrive(bar(ITEM_FULL + sl));
                late = !s.routed;
            }
            ++n_item;
            slot_it.next();
            // the rest of the warp learns the item from lane 0
            const int valid = __shfl_sync(0xffffffffu, s.valid, 0), routed = __shfl_sync(0xffffffffu, s.routed, 0);
            const int h = __shfl_sync(0xffffffffu, s.h, 0), first = __shfl_sync(0xffffffffu, s.first, 0), rows = __shfl_sync(0xffffffffu, s.rows, 0);
            ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
            if (!valid || !ok) break;
            const int n_qt = rows > 128 ? 2 : 1;
            last_g = n_qt - 1;
            if (LOADERS) {
                for (int g = 0; g < n_qt; ++g, ++n_qtile) q_phase ^= 1u << (3 * g + n_qtile % 3);
                continue;
            }
            for (int g = 0; ok && g < n_qt; ++g) {
                const int qb = n_qtile % 3, qf = 3 * g + qb;
                ok = mbar_wait(bar(Q_EMPTY + qb), ((n_qtile / 3) & 1) ^ 1, abort_flag, p.wait, W_QEMPTY) && merged(qb, !routed, m_used, m_phase);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (lane == 0) mbar_expect_tx(bar(Q_FULL + qf), TILE_BYTES);
                __syncwarp();
                if (!routed) {
                    if (lane == 0) {
#pragma unroll
                        for (int sub = 0; sub < SUB; ++sub)
                            tma_load_2d(sQ + qb * TILE_BYTES + sub * SUB_BYTES, &tmQ, sub * 64, h * p.L + first + g * 128, bar(Q_FULL + qf));
                    }
                } else {
                    // lane l gathers rows 4 l .. 4 l + 3 of the tile; a row past the item's end repeats the item's
                    // first query (its result is never stored)
                    int row[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int rt = g * 128 + lane * 4 + x;
                        const size_t at = (size_t)first + (rt < rows ? rt : 0);
                        const int e = at < p.cap_total ? p.qlist[(size_t)h * p.cap_total + at] : 0;
                        int qi = e / p.k;
                        if (e < 0 || qi >= p.L) qi = 0;
                        row[x] = h * p.L + qi;
                    }
#pragma unroll
                    for (int sub = 0; sub < SUB; ++sub)
                        tma_gather4(sQ + qb * TILE_BYTES + sub * SUB_BYTES + lane * 512, &tmQrow, sub * 64, row[0], row[1], row[2], row[3],
                                    bar(Q_FULL + qf));
                }
                q_phase ^= 1u << qf;
                ++n_qtile;
            }
        }
        if (!LOADERS && *abort_flag && lane == 0) {
            // drain: the Q copies already issued must land before the CTA's shared memory is released
            int dummy_flag = 0;
            // (a barrier that was never used is past the phase before its first)
            for (int b = 0; b < 6; ++b) mbar_wait(bar(Q_FULL + b), ((q_phase >> b) & 1) ^ 1, &dummy_flag, p.wait, W_QFULL);
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLoad));
        // ------------------------------------------------------------ Q loaders: rows 32 lw .. 32 lw + 31 of every query tile.
        // All four warps load a part of every tile, so a buffer cannot be filled and released without one of them: none
        // can miss a phase of Q_EMPTY.
        const int lw = warp - 12;
        int n_qtile = 0;
        SlotIter slot_it;
        uint32_t m_used = 0, m_phase = 0;              // as above
        uint32_t q_phase = 0;                          // bit 3 g + buffer: parity of the next phase of that Q_FULL
        bool ok = true;
        while (ok) {
            const int sl = slot_it.at;
            ok = mbar_wait(bar(ITEM_FULL + sl), slot_it.phase, abort_flag, p.wait, W_ITEMFULL);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const int valid = s_item[sl].valid, routed = s_item[sl].routed, h = s_item[sl].h, first = s_item[sl].first, rows = s_item[sl].rows;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(ITEM_EMPTY + sl));
            slot_it.next();
            if (!valid) break;
            const int n_qt = rows > 128 ? 2 : 1;
            // the queries of this lane's rows (a row past the item's end fetches row 0 of the head: its result is never stored)
            int qrow[2] = {0, 0};
            if (routed) {
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    const int rt = g * 128 + lw * 32 + lane;
                    const size_t at = (size_t)first + rt;
                    const int e = rt < rows && at < p.cap_total ? p.qlist[(size_t)h * p.cap_total + at] : -1;
                    qrow[g] = e < 0 ? 0 : e / p.k;
                    if (qrow[g] >= p.L) qrow[g] = 0;
                }
            }
            for (int g = 0; ok && g < n_qt; ++g) {
                const int qb = n_qtile % 3, qf = 3 * g + qb;
                int row[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) row[x] = h * p.L + __shfl_sync(0xffffffffu, qrow[g], (lane & 7) * 4 + x);
                ok = mbar_wait(bar(Q_EMPTY + qb), ((n_qtile / 3) & 1) ^ 1, abort_flag, p.wait, W_QEMPTY) && merged(qb, !routed, m_used, m_phase);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (lw == 0 && lane == 0) mbar_expect_tx(bar(Q_FULL + qf), TILE_BYTES);
                const uint32_t dst = sQ + qb * TILE_BYTES + lw * 32 * 128;
                if (!routed) {
                    if (lane == 0) {
#pragma unroll
                        for (int sub = 0; sub < SUB; ++sub)          // (32 rows, of which the tile's part for the warp comes first)
                            tma_load_2d(dst + sub * SUB_BYTES, &tmQ, sub * 64, h * p.L + first + g * 128 + lw * ((min(128, rows - g * 128) + 3) >> 2), bar(Q_FULL + qf));
                    }
                } else if (lane < 8) {                          // lane l gathers rows 4 l .. 4 l + 3 of the warp's 32
#pragma unroll
                    for (int sub = 0; sub < SUB; ++sub)
                        tma_gather4(dst + sub * SUB_BYTES + lane * 512, &tmQrow, sub * 64, row[0], row[1], row[2], row[3], bar(Q_FULL + qf));
                }
                __syncwarp();
                q_phase ^= 1u << qf;
                ++n_qtile;
            }
        }
        if (*abort_flag && lw == 0 && lane == 0) {
            // drain: the Q copies already issued must land before the CTA's shared memory is released
            int dummy_flag = 0;
            // (a barrier that was never used is past the phase before its first)
            for (int b = 0; b < 6; ++b) mbar_wait(bar(Q_FULL + b), ((q_phase >> b) & 1) ^ 1, &dummy_flag, p.wait, W_QFULL);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tmem, kTmemCols);
    if (threadIdx.x == 0) report_abort(p.status, s_abort);
    // the last CTA to leave rewinds the queue, so that the next call on this workspace needs no launch that prepares it
    if (threadIdx.x == 0 && s_usable) {
        __threadfence();
        if (atomicAdd(&p.queue[3], 1) == (int)gridDim.x - 1) {
            p.queue[0] = p.queue[3] = 0;
            for (int ph = 0; ph < 2 * p.n_groups; ++ph) phase_tab[3 * ph + 2] = 0;
        }
    }
}

// ---- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

int make_tmap_2d_bf16(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *sym = nullptr;
        cudaDriverEntryPointQueryResult q;
        MOC_CUDA_TRY(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q));
        if (!sym || q != cudaDriverEntryPointSuccess) { set_cuda_error(cudaErrorUnknown, "cuTensorMapEncodeTiled not found"); return MOC_ERR_CUDA; }
        fn = (EncodeTiledFn)sym;
    }
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * 2};
    cuuint32_t box[2] = {64, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { set_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled"); return MOC_ERR_CUDA; }
    return MOC_OK;
}

template <int D, bool LOADERS>
static int attend_tc_d(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *K, const __nv_bfloat16 *V,
                       __nv_bfloat16 *O, float *lse, void *ws, cudaStream_t s) {
    CUtensorMap tmQ, tmQrow, tmK, tmV;
    if (int r = make_tmap_2d_bf16(&tmQ, Q, (uint64_t)p->H * p->L, D, LOADERS ? 32 : 128)) return r;
    if (int r = make_tmap_2d_bf16(&tmQrow, Q, (uint64_t)p->H * p->L, D, 1)) return r;      // row gathers: a box one row high
    if (int r = make_tmap_2d_bf16(&tmK, K, (uint64_t)p->H * p->L, D, kBN)) return r;
    if (int r = make_tmap_2d_bf16(&tmV, V, (uint64_t)p->H * p->L, D, kBN)) return r;
    const int n_groups = (p->H + p->heads_per_group - 1) / p->heads_per_group;
    AttendParams a;
    a.Q = Q; a.O = O; a.lse = lse;
    a.part_o = ws_ptr<__nv_bfloat16>(ws, p->ws.part_o);
    a.part_lse = ws_ptr<float>(ws, p->ws.part_lse);
    a.part_stride = n_groups > 1 ? (size_t)p->heads_per_group * ((p->L + 127) / 128 * 128) * p->k * D : 0;
    a.chunk_rng = p->d_chunk_rng; a.anc_rng = p->d_anc_rng;
    a.ritems = ws_ptr<WorkItem>(ws, p->ws.rtiles);
    a.aitems = p->d_qitems;
    a.tile_off = ws_ptr<int>(ws, p->ws.tile_off);
    a.qlist = ws_ptr<int32_t>(ws, p->ws.qlist);
    a.queue = ws_ptr<int>(ws, p->ws.queue);
    a.cap_total = (size_t)p->cap_off[p->C];
    a.status = ws_ptr<int>(ws, p->ws.status);
    a.H = p->H; a.L = p->L; a.C = p->C; a.k = p->k; a.hg = p->heads_per_group; a.n_groups = n_groups;
    a.n_aitems = (int)p->qitems.size();
    a.kdiv = SlotDiv::of(p->k);
    a.scale_log2 = p->scale * 1.4426950408889634f;
    a.cookie = p->cookie;
    a.wait = WaitBound::of(p->wait_us);
    // always the d = 128 footprint: more than half an SM's shared memory, so CTAs (which each
    // take all 512 TMEM columns) never share an SM
    const size_t smem = 7 * (size_t)128 * 128 * 2 + 1024;      // Q ring of three, K and V two stages each
    MOC_CUDA_TRY(cudaFuncSetAttribute(attend_tc_kernel<D, LOADERS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // one CTA per SM, never more than there can be items
    const long long most = (long long)p->H * (a.n_aitems + ((long long)p->L * p->k + kQTileRows - 1) / kQTileRows + (p->k ? p->C : 0));
    const unsigned grid = (unsigned)std::max(1LL, std::min<long long>(p->n_sm, most));
    MOC_CUDA_TRY(launch_early(true, attend_tc_kernel<D, LOADERS>, grid, LOADERS ? kThreadsLoaders : kThreads, smem, s, tmQ, tmQrow, tmK, tmV, a));
    MOC_LAUNCH_CHECK();
    return MOC_OK;
}

int launch_attend_tc(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *K, const __nv_bfloat16 *V,
                     const int32_t *, __nv_bfloat16 *O, float *lse, void *ws, cudaStream_t s) {
    // Who loads the query tiles.  A row gather costs the warp that issues it some 65 cycles for four rows of 128 bytes: with
    // one warp a 256-row routed item cannot start more often than every 13000 cycles (half that at d = 64), with four every
    // 3000 to 4000 - but four loading warps, one on every scheduler, are in the way of the softmax.  Measured, one warp -> four
    // (which at d = 128 also takes the merge through registers; streams of 131k tokens, 3 to 32 picks):
    //   d = 64, 8 heads: chunks of 128 tokens 1.08 to 1.19 times faster, of 256 1.08 to 1.16 (24 picks 6.12 -> 5.28 ms), of 384 0.91 to
    //     0.95 (6.24 -> 6.54 ms), of 512 0.96, of 640 0.91 to 0.94;
    //   d = 128, 6 heads: 256 1.21 to 1.40 (32 picks 8.94 -> 6.59 ms), 384 1.02 to 1.19, 512 1.02 to 1.05 (9.57 -> 9.22 ms), 768 1.00 to 1.01,
    //     1024 0.99 to 1.00; a clip of 1560-token frames, 24 heads, 0.97.
    const int up_to = p->d == 64 ? 2 : 4;        // key tiles a chunk, on average
    const bool loaders = p->k > 0 && p->routed_key_tiles <= (int64_t)up_to * p->ncol;
    if (p->d == 64) return loaders ? attend_tc_d<64, true>(p, Q, K, V, O, lse, ws, s) : attend_tc_d<64, false>(p, Q, K, V, O, lse, ws, s);
    return loaders ? attend_tc_d<128, true>(p, Q, K, V, O, lse, ws, s) : attend_tc_d<128, false>(p, Q, K, V, O, lse, ws, s);
}

}  // namespace moc
