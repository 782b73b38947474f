// Tensor-core dQ of the sparse attention's backward (selection held constant): two persistent launches per group of heads.
//
// For a selected (query i, key t) pair:  P = exp(scale q.k - lse_i),  dP = dO_i . v_t,  dS = P (dP - delta_i),
// dQ_i += scale dS k_t.  A work item is 128 query rows against their key tiles, as in the forward: the ROUTED launch takes
// the rows of one chunk's query list against that chunk's keys and leaves one partial per (query, slot) in the workspace,
// the ANCHOR launch takes consecutive rows against their anchor ranges, adds the rows' partials and writes dQ.
//
//     T1 = Q K^T,  T2 = dO V^T          (both operands from shared memory, into TMEM)
//     threads (two per TMEM lane) turn T1 into P, then (P, T2) into dS, written back to TMEM as bf16 over the columns of T2
//     that the thread itself has read
//     ACC += dS K                        (A from TMEM, the K tile as an MN-major operand)
//
// One CTA per SM walks its items (an equal share of the launch's, which but for the empty ones are much alike): the tensor memory, the
// barriers and the K/V rings live for the whole launch, and the next item's rows are fetched while the last tile of the current
// one and its results are in work.  With a CTA per item, the launch of the CTA, its dependent look-ups and the gather of its
// rows took 8000 cycles before the first product, of 42000 for an item of 13 key tiles.
// 16 warps:
//   warps 0-7   lanes, two threads per TMEM lane: of the four 32-column chunks of a tile, thread `half` takes chunks half and
//               2 + half, and keeps its 64 P values between T1 and T2;
//   warp 8      lane 0, TMA producer of the K and V tiles (three and two stages, running across items);
//   warps 9-11  row loaders: the Q and dO rows of the next item by 16-byte asynchronous copies, its lse and delta, and its
//               description for the other warps;
//   warps 12,13 MMA issuers: warp 12 T1, warp 13 T2 and ACC.  T1(j + 1) is issued once the lanes have read T1(j); T2 has two
//               buffers, T2(j + 2) follows ACC(j), which reads the dS stored over T2(j);
//   warps 14,15 idle (they complete the fourth warpgroup).
// Every mbarrier wait is bounded; a wait that runs out flags the workspace status word and the CTA drains and leaves.
#include <algorithm>

#include "moc_common.cuh"
#include "moc_tc.cuh"

namespace moc {

using namespace tc;

enum DqWait { DW_XFULL = 96, DW_XEMPTY, DW_YFULL, DW_YEMPTY, DW_T1FULL, DW_T2FULL, DW_READ, DW_DSDONE, DW_ACCFULL, DW_ACCFREE, DW_SMEM };

struct DqParams {
    const __nv_bfloat16 *Q, *dO;
    const float *lse, *delta;
    __nv_bfloat16 *dQ;
    __nv_bfloat16 *part;          // routed dQ partials of the group of heads in flight (part_line)
    const float *part_lse;        // the forward's routed log-sum-exps (part_lse_at): -inf marks an empty slot
    const KeyRange *rng;          // key ranges the items index
    const WorkItem *items;        // up to 256 rows each: two of this kernel's items
    const int *item_lo, *item_hi; // routed: the group's item range on the device
    const int32_t *qlist;
    size_t cap_total;
    int *status;
    int H, L, k, h0, hg, n_items; // anchor: n_items items for each of the group's hg heads
    SlotDiv kdiv;
    float scale, scale_log2;
    uint32_t cookie;
    WaitBound wait;
};

constexpr int kDqThreads = 512, kKStages = 3, kVStages = 2, kLoaders = 3;

// acc += the bf16 pair u where cond holds
__device__ __forceinline__ void add_if(bool cond, uint64_t &acc, uint32_t u) {
    const uint64_t v = pack2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
    asm("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p add.rn.f32x2 %0, %0, %1;\n\t}" : "+l"(acc) : "l"(v), "r"((int)cond));
}

// description of an item, as the row loaders leave it for the other warps; rows = 0: no more items
struct DqItem { int h, first, rows, nrng, ntiles, rng_off, t0, t1; };

template <int D, bool ANCHOR>
__global__ void __launch_bounds__(kDqThreads, 1) attend_dq_tc_kernel(const __grid_constant__ CUtensorMap tmK,
                                                                     const __grid_constant__ CUtensorMap tmV, const DqParams p) {
    constexpr int TILE_BYTES = 128 * D * 2;
    constexpr int SUB = D / 64;
    constexpr int SUB_BYTES = 128 * 128;
    constexpr int CH = D / 8;               // 16-byte pieces per row
    constexpr int N_TILES_SMEM = 2 + kKStages + kVStages;
    enum { X_FULL = 0, X_EMPTY, K_FULL, K_EMPTY = K_FULL + kKStages, V_FULL = K_EMPTY + kKStages, V_EMPTY = V_FULL + kVStages,
           T1_FULL = V_EMPTY + kVStages, T1_READ, T2_FULL, DS_DONE = T2_FULL + 2, ACC_FULL = DS_DONE + 2, ACC_FREE, N_BARS };
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[N_BARS];
    __shared__ __align__(16) float s_ld[2][2][128];      // per item parity: -lse * log2(e) and -delta of the item's rows
    __shared__ DqItem s_item[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort, s_lo, s_total;

    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    // shared tiles: X1 (Q) X2 (dO) | K stages | V stages
    const uint32_t sX = sbase, sK = sbase + 2 * TILE_BYTES, sV = sbase + (2 + kKStages) * TILE_BYTES;
    auto bar = [&](int i) { return smem_u32(&bars[i]); };

    if (threadIdx.x == 0) {
        s_abort = 0;
        bool valid = *(volatile int *)p.status == 0;
        if (valid && (uint32_t)((volatile int *)p.status)[ST_COOKIE] != p.cookie) {
            atomicCAS(p.status, 0, MOC_ERR_WORKSPACE);      // not this plan's lists: report, touch nothing else
            valid = false;
        }
        uint32_t dyn_bytes;
        asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_bytes));
        if (valid && (sbase - smem_u32(smem_raw)) + (uint32_t)N_TILES_SMEM * TILE_BYTES > dyn_bytes) {
            // the launch gave less shared memory than the tiles need: report, touch nothing
            if (atomicCAS(p.status, 0, MOC_ERR_TIMEOUT) == 0) p.status[ST_DETAIL] = DW_SMEM;
            valid = false;
        }
        s_lo = (!ANCHOR && valid) ? *p.item_lo : 0;
        s_total = !valid ? 0 : 2 * (ANCHOR ? p.n_items * p.hg : *p.item_hi - s_lo);
        mbar_init(bar(X_FULL), kLoaders);
        mbar_init(bar(X_EMPTY), 2 + 8);                     // both issuers, and each lane warp when it has the item's data
        for (int t = 0; t < kKStages; ++t) { mbar_init(bar(K_FULL + t), 1); mbar_init(bar(K_EMPTY + t), 1); }
        for (int t = 0; t < kVStages; ++t) { mbar_init(bar(V_FULL + t), 1); mbar_init(bar(V_EMPTY + t), 1); }
        mbar_init(bar(T1_FULL), 1);
        mbar_init(bar(T1_READ), 256);
        for (int t = 0; t < 2; ++t) { mbar_init(bar(T2_FULL + t), 1); mbar_init(bar(DS_DONE + t), 256); }
        mbar_init(bar(ACC_FULL), 1);
        mbar_init(bar(ACC_FREE), 256);
        fence_barrier_init();
    }
    __syncthreads();
    next_may_start();
    if (s_total <= (int)blockIdx.x) {
        if (ANCHOR && blockIdx.x == 0) previous_done();
        return;
    }
    if (warp == 8) {
        tmem_alloc(smem_u32(&tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    // TMEM columns: T1 [0,128)  T2 of the even tiles [128,256)  ACC [256,384)  T2 of the odd tiles [384,512)
    const uint32_t tmem = tmem_slot;
    volatile int *abort_flag = &s_abort;
    // item x of the launch (x counts halves of 256-row work items); false: it has no rows
    auto fetch = [&](int x, DqItem &o) -> bool {
        int item = x >> 1, h = 0;
        if (ANCHOR) { h = p.h0 + item / p.n_items; item %= p.n_items; }
        else item += s_lo;
        const WorkItem w = p.items[item];
        const int skip = (x & 1) * 128;
        o.h = ANCHOR ? h : w.h;
        o.first = w.first + skip;
        o.rows = min(128, w.rows - skip);
        o.nrng = w.nrng; o.ntiles = w.ntiles; o.rng_off = w.rng_off; o.t0 = w.t0; o.t1 = w.t1;
        if (!ANCHOR && !index_ok((unsigned)w.h < (unsigned)p.H && w.rows > 0 && w.rows <= kQTileRows && w.first >= 0 &&
                                 (size_t)w.first + w.rows <= p.cap_total && w.nrng == 1, p.status, IX_BWD_ITEM_FIELDS))
            o.rows = 0;
        return o.rows > 0;
    };
    // The CTA's next item with rows, from `round` and `pos` on (which start at 0 and blockIdx.x).  Of an item of at most 128
    // rows the second half has none, and such items come in patterns: a CTA that kept its place in every round would, the
    // grid being even, take nothing but second halves, or, with chunks of 257 to 384 rows, only every other item.  So the
    // place moves by three, an odd number, from round to round.  (Training steps, the place kept -> moved: 64 frames of 128
    // tokens, 8 heads, no picks 484 -> 364 us; 256 of 64, 24 heads, 4 picks 3072 -> 2712 us.)
    auto next_item = [&](int &round, int &pos, DqItem &o) -> bool {
        while (round < s_total) {
            const int x = round + pos;
            round += gridDim.x;
            pos += 3;
            if (pos >= (int)gridDim.x) pos -= gridDim.x;
            if (x < s_total && fetch(x, o)) return true;
        }
        return false;
    };

    if (warp < 8) {
        // ------------------------------------------------------------ lane threads
        asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
        const int r = threadIdx.x & 127;              // row of the item = TMEM lane
        const int half = warp >> 2;
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
        const uint64_t c2 = pack2(p.scale_log2, p.scale_log2);
        const int LB = (p.L + 127) >> 7;
        char *part = reinterpret_cast<char *>(p.part);
        int g = 0;                                    // tiles processed
        bool ok = true;
        for (int n = 0; ok; ++n) {
            ok = mbar_wait(bar(X_FULL), n & 1, abort_flag, p.wait, DW_XFULL);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const int rows = s_item[n & 1].rows, h = s_item[n & 1].h, first = s_item[n & 1].first, n_tiles = s_item[n & 1].ntiles;
            if (rows == 0) break;
            TileIter it(p.rng + s_item[n & 1].rng_off, s_item[n & 1].nrng, s_item[n & 1].t0, s_item[n & 1].t1);
            const float nlse = s_ld[n & 1][0][r], ndlt = s_ld[n & 1][1][r];
            const uint64_t nlse2 = pack2(nlse, nlse), ndlt2 = pack2(ndlt, ndlt);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(X_EMPTY));
            // the list entry of this row, wanted at the end
            int e = -1;
            if (!ANCHOR && r < rows) e = p.qlist[(size_t)h * p.cap_total + first + r];
            float pv[64];
            // P = exp2(scale log2(e) S - lse log2(e))
            auto p_pair = [&](const uint32_t (&sv)[32], int x, float &p0, float &p1) {
                unpack2(fma2(pack2(__uint_as_float(sv[x]), __uint_as_float(sv[x + 1])), c2, nlse2), p0, p1);
                p0 = ex2(p0);
                p1 = ex2(p1);
            };
            // dS = P (dP - delta)
            auto ds_pair = [&](const uint32_t (&dp)[32], int rd, int x) {
                float a0, a1;
                unpack2(mul2(pack2(pv[rd * 32 + x], pv[rd * 32 + x + 1]), add2(pack2(__uint_as_float(dp[x]), __uint_as_float(dp[x + 1])), ndlt2)), a0, a1);
                return bf16x2(a0, a1);
            };
            auto mask = [&](int valid) {                     // keys past the end of the range
                if (valid < 128) {
#pragma unroll
                    for (int x = 0; x < 64; ++x)
                        if (((x >> 5) * 2 + half) * 32 + (x & 31) >= valid) pv[x] = 0.f;
                }
            };
            int valid, t0;
            bool t1_early = false, t2_early = false;         // looked at behind other work: see the dK/dV kernel
            // P of the tile
            auto form_p = [&]() __attribute__((always_inline)) -> bool {
                ok = t1_early || mbar_wait_spin(bar(T1_FULL), g & 1, abort_flag, p.wait, DW_T1FULL);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) return false;
                tc_fence_after();
                uint32_t sv[2][32];
                tmem_ld32(tmem + lane_off + half * 32, sv[0]);
                tmem_ld32(tmem + lane_off + (2 + half) * 32, sv[1]);
                tmem_wait_ld();
                tc_fence_before();
                mbar_arrive(bar(T1_READ));                   // T1 may be overwritten
                t2_early = mbar_test_wait(bar(T2_FULL + (g & 1)), (g >> 1) & 1);
#pragma unroll
                for (int rd = 0; rd < 2; ++rd) {
                    // a key tile's last 64 columns, where it has no keys: ACC takes no step over them.  (All 128 -> this, the whole backward: 4
                    // heads of 1560-token frames, 24 keys in the last tile, 1450 -> 1442 us, 24 heads at the power limit 9.93 -> 9.85 ms, 1 head of
                    // 1169-token frames 825 -> 811 us.  The same in dK/dV gained nothing, in the forward it cost 1 to 4 %.)
                    if (rd == 1 && valid <= 64) break;
#pragma unroll
                    for (int x = 0; x < 32; x += 2) p_pair(sv[rd], x, pv[rd * 32 + x], pv[rd * 32 + x + 1]);
                }
                mask(valid);
                return true;
            };
            // dS of the tile, and on to the next
            auto form_ds = [&]() __attribute__((always_inline)) -> bool {
                const int st = g & 1;
                const uint32_t t2 = tmem + lane_off + (st ? 384u : 128u);
                ok = t2_early || mbar_wait_spin(bar(T2_FULL + st), (g >> 1) & 1, abort_flag, p.wait, DW_T2FULL);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) return false;
                tc_fence_after();
                uint32_t dp[2][32];
                tmem_ld32(t2 + half * 32, dp[0]);
                tmem_ld32(t2 + (2 + half) * 32, dp[1]);
                t1_early = mbar_test_wait(bar(T1_FULL), (g + 1) & 1);
                tmem_wait_ld();
#pragma unroll
                for (int rd = 0; rd < 2; ++rd) {
                    if (rd == 1 && valid <= 64) break;
                    uint32_t uds[16];
#pragma unroll
                    for (int x = 0; x < 32; x += 2) uds[x >> 1] = ds_pair(dp[rd], rd, x);
                    // over the first half of the chunk's own columns, which this thread alone has read.  (With the chunks side by side
                    // the two threads of a lane waited for each other.  Without that, and with the partials as whole lines: 10.75 -> 10.21 ms
                    // for the whole backward of the 33k-token clip, 24 heads, by itself.)
                    tmem_st16(t2 + (rd * 2 + half) * 32, uds);
                }
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(bar(DS_DONE + st));
                ++g;
                return true;
            };
            it.next(t0, valid);
            if (!form_p()) break;
            for (int jt = 0; jt + 1 < n_tiles; ++jt) {
                if (!form_ds()) break;
                it.next(t0, valid);
                if (!form_p()) break;
            }
            if (!ok || !form_ds()) break;
            // ---- epilogue
            ok = mbar_wait(bar(ACC_FULL), n & 1, abort_flag, p.wait, DW_ACCFULL);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            // Results move in the 16 x 256-bit load shape of the tensor memory: of a 16-row half of the warp's rows, lane l holds
            // rows l / 4 and l / 4 + 8, of every eight columns the two at 2 (l % 4), so that four lanes write 128 contiguous bytes
            // of a row.  (With a row per lane a warp's 32-byte stores touched 32 lines each.)  Of the two warps that share the TMEM
            // lanes, each takes 64 columns of all rows (d = 128) or 16 rows (d = 64).  A partial keeps its columns in the order of the
            // lanes; dQ is put in the order of the columns.
            constexpr int NJ = D / 32;                       // groups of eight rows that this warp has
            const int l4 = lane >> 2, l2 = lane & 3, cb = D == 128 ? half : 0, j0 = D == 128 ? 0 : 2 * half;
            const uint32_t t_acc = tmem + lane_off + 256 + ((uint32_t)(j0 >> 1) << 20) + cb * 64;
            if (!ANCHOR) {
                uint32_t v[NJ / 2][32];
#pragma unroll
                for (int x = 0; x < NJ / 2; ++x) tmem_ld_16x256b(t_acc + ((uint32_t)x << 20), v[x]);
                tmem_wait_ld();
                tc_fence_before();
                mbar_arrive(bar(ACC_FREE));                  // the next item's dQ may be accumulated
                size_t line = 0;                             // where this row's partial goes
                bool keep = false;
                if (e >= 0) {
                    const int qi = p.kdiv.query(e), slot = e - qi * p.k;
                    if (index_ok((unsigned)qi < (unsigned)p.L, p.status, IX_BWD_LIST_ENTRY) && (unsigned)qi < (unsigned)p.L) {
                        line = part_line(h - p.h0, LB, p.k, D / 64, qi, slot);
                        keep = true;
                    }
                }
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const size_t at = __shfl_sync(0xffffffffu, line, (j0 + j) * 8 + l4);
                    const bool some = __shfl_sync(0xffffffffu, keep, (j0 + j) * 8 + l4);
                    uint32_t u[8];
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        u[x] = bf16x2(__uint_as_float(v[j >> 1][4 * x + 2 * (j & 1)]) * p.scale, __uint_as_float(v[j >> 1][4 * x + 2 * (j & 1) + 1]) * p.scale);
                    if (some) st_256(part + at + ((size_t)cb << 14) + l2 * 32, u);
                }
            } else {
                // the routed partials of a query, a few slots requested together, the next ones while these are added up; a slot is
                // in use if the forward left a finite log-sum-exp for it
                previous_done();                             // the routed launch's partials are complete
                constexpr int B = 4;
                struct Batch { uint32_t v[B][8]; float ls[B]; };
                const int row0 = first + j0 * 8 + (warp & 3) * 32 + l4, row_end = first + rows;
                int ask_j = 0, ask_s = 0;
                auto ask = [&](Batch &b) __attribute__((always_inline)) {
                    const int q = row0 + ask_j * 8;
                    const bool in = q < row_end;
                    const char *src = part + part_line(h - p.h0, LB, p.k, D / 64, q, ask_s) + ((size_t)cb << 14) + l2 * 32;
                    const float *ls = p.part_lse + part_lse_at(h, LB, p.k, q, ask_s);
#pragma unroll
                    for (int u = 0; u < B; ++u) {
                        const bool some = in && ask_s + u < p.k;
                        const float x = *(some ? ls + u * 128 : p.part_lse);
                        b.ls[u] = some ? x : -INFINITY;
                        ld_cg_256_if(some, src + ((size_t)(u * (D / 64)) << 14), b.v[u]);
                    }
                    ask_s += B;
                    if (ask_s >= p.k) { ask_s = 0; ++ask_j; }
                };
                uint64_t acc[8];
                uint32_t v[32];
                int j = 0, s0 = 0;
                auto add = [&](const Batch &b) __attribute__((always_inline)) {
                    if (s0 == 0) {
                        if (!(j & 1)) {                      // two groups of rows at a time
                            tmem_ld_16x256b(t_acc + ((uint32_t)(j >> 1) << 20), v);
                            tmem_wait_ld();
                            if (j == NJ - 2) {
                                tc_fence_before();
                                mbar_arrive(bar(ACC_FREE));  // the next item's dQ may be accumulated
                            }
                        }
                        const uint64_t sc2 = pack2(p.scale, p.scale);
#pragma unroll
                        for (int x = 0; x < 8; ++x)
                            acc[x] = mul2(pack2(__uint_as_float((j & 1) ? v[4 * x + 2] : v[4 * x]), __uint_as_float((j & 1) ? v[4 * x + 3] : v[4 * x + 1])), sc2);
                    }
#pragma unroll
                    for (int u = 0; u < B; ++u)
#pragma unroll
                        for (int x = 0; x < 8; ++x) add_if(b.ls[u] != -INFINITY, acc[x], b.v[u][x]);
                    s0 += B;
                    if (s0 >= p.k) {
                        uint32_t u[8];
#pragma unroll
                        for (int x = 0; x < 8; ++x) {
                            float lo, hi;
                            unpack2(acc[x], lo, hi);
                            u[x] = bf16x2(lo, hi);
                        }
                        quad_transpose(u, l2);
                        const int q = row0 + j * 8;
                        if (q < row_end) store_quad(p.dQ + ((size_t)h * p.L + q) * D + cb * 64, l2, u);
                        s0 = 0;
                        ++j;
                    }
                };
                Batch even = {}, odd = {};
                ask(even);
#pragma unroll 1
                while (j < NJ) {                             // an even number of row groups, so of batches
                    ask(odd);
                    add(even);
                    if (ask_j < NJ) ask(even);
                    add(odd);
                }
            }
        }
    } else if (warp == 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        // ------------------------------------------------------------ TMA producer of the K and V tiles
        if (lane == 0) {
            prefetch_tensormap(&tmK);
            prefetch_tensormap(&tmV);
            int n_k = 0, n_v = 0, s3 = 0, ph3 = 0;           // K and V tiles issued; K stage and its phase
            bool ok = true;
            DqItem w;
            for (int round = 0, pos = blockIdx.x; ok && next_item(round, pos, w);) {
                TileIter it(p.rng + w.rng_off, w.nrng, w.t0, w.t1);
                int t0, valid;
                while (it.next(t0, valid)) {
                    const int s2 = n_v & 1;
                    ok = mbar_wait(bar(K_EMPTY + s3), ph3 ^ 1, abort_flag, p.wait, DW_YEMPTY);
                    if (!ok) break;
                    mbar_expect_tx(bar(K_FULL + s3), TILE_BYTES);
#pragma unroll
                    for (int sub = 0; sub < SUB; ++sub)
                        tma_load_2d(sK + s3 * TILE_BYTES + sub * SUB_BYTES, &tmK, sub * 64, w.h * p.L + t0, bar(K_FULL + s3));
                    ++n_k;
                    ok = mbar_wait(bar(V_EMPTY + s2), ((n_v >> 1) & 1) ^ 1, abort_flag, p.wait, DW_YEMPTY);
                    if (!ok) break;
                    mbar_expect_tx(bar(V_FULL + s2), TILE_BYTES);
#pragma unroll
                    for (int sub = 0; sub < SUB; ++sub)
                        tma_load_2d(sV + s2 * TILE_BYTES + sub * SUB_BYTES, &tmV, sub * 64, w.h * p.L + t0, bar(V_FULL + s2));
                    ++n_v;
                    if (++s3 == kKStages) { s3 = 0; ph3 ^= 1; }
                }
            }
            if (*abort_flag) {      // copies already issued must land before the shared memory is released
                int dummy_flag = 0;
                for (int b = 1; b <= kKStages; ++b)
                    if (n_k - b >= 0) mbar_wait(bar(K_FULL + (n_k - b) % kKStages), ((n_k - b) / kKStages) & 1, &dummy_flag, p.wait, DW_YFULL);
                for (int b = 1; b <= kVStages; ++b)
                    if (n_v - b >= 0) mbar_wait(bar(V_FULL + ((n_v - b) & 1)), ((n_v - b) >> 1) & 1, &dummy_flag, p.wait, DW_YFULL);
            }
        }
    } else if (warp < 12) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        // ------------------------------------------------------------ row loaders.  The eight pieces of an item's rows - 32-row
        // block b & 3 of Q (b < 4) or dO - are dealt to the three warps; who brings a block of Q also brings its lse and
        // delta.  Everything an item needs is looked up before its buffers are free.
        const int lw = warp - 9;
        int n = 0;
        bool ok = true;
        int round = 0, pos = blockIdx.x;
        for (bool more = true; ok && more; ++n) {
            DqItem w = {};
            more = next_item(round, pos, w);
            if (!more) w.rows = 0;
            int q[3];
            float lse[3], del[3];
#pragma unroll
            for (int y = 0; y < 3; ++y) {
                const int b = lw + 3 * y, i = (b & 3) * 32 + lane;
                q[y] = -1; lse[y] = INFINITY; del[y] = 0.f;
                if (b < 8 && i < w.rows) {
                    q[y] = w.first + i;
                    if (!ANCHOR) {
                        q[y] = p.kdiv.query(p.qlist[(size_t)w.h * p.cap_total + w.first + i]);
                        if ((unsigned)q[y] >= (unsigned)p.L) q[y] = -1;      // never follow an entry that is not a row of this head
                    }
                    if (b < 4 && q[y] >= 0) {
                        lse[y] = p.lse[(size_t)w.h * p.L + q[y]];
                        del[y] = p.delta[(size_t)w.h * p.L + q[y]];
                    }
                }
            }
            if (n > 0) {
                ok = mbar_wait(bar(X_EMPTY), (n - 1) & 1, abort_flag, p.wait, DW_XEMPTY);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
            }
            if (more) {
#pragma unroll
                for (int y = 0; y < 3; ++y) {
                    const int b = lw + 3 * y;
                    if (b >= 8) break;
                    const __nv_bfloat16 *src = (b < 4 ? p.Q : p.dO) + (size_t)w.h * p.L * D;
                    const uint32_t dst = sX + (b >> 2) * TILE_BYTES;
                    constexpr int RP = 32 / CH;                // rows per instruction
                    const int c16 = lane % CH;
#pragma unroll 1
                    for (int r8 = 0; r8 < 32; r8 += 8)          // (eight rows at a time, in which the swizzle repeats)
#pragma unroll
                        for (int rb = 0; rb < 8; rb += RP) {
                            const int rl = rb + lane / CH, qq = __shfl_sync(0xffffffffu, q[y], r8 + rl);
                            cp_async16(dst + (c16 >> 3) * SUB_BYTES + ((b & 3) * 32 + r8) * 128 + sw128_offset(rl, c16 & 7),
                                       src + (size_t)max(qq, 0) * D + c16 * 8, qq >= 0 ? 16u : 0u);
                        }
                    if (b < 4) {                               // a row without a query gets lse = +inf: P and dS are zero
                        s_ld[n & 1][0][b * 32 + lane] = lse[y] * -1.4426950408889634f;
                        s_ld[n & 1][1][b * 32 + lane] = -del[y];
                    }
                }
            }
            if (lw == 0 && lane == 0) s_item[n & 1] = w;
            cp_async_wait_all();
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(X_FULL));
        }
        cp_async_wait_all();
    } else {
        // ------------------------------------------------------------ MMA issuers (a warp stays together, one lane of it issues)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        if (warp <= 13) {
            constexpr uint32_t IDESC_T = idesc_bf16_f32(128, 128, 0, 0);      // T = X Y^T, both K-major
            constexpr uint32_t IDESC_ACC = idesc_bf16_f32(128, D, 0, 1);      // ACC += dS K, K MN-major
            constexpr uint32_t STAGE = TILE_BYTES >> 4;
            auto lo = [](uint64_t d) { return (uint32_t)d; };
            auto hi = [](uint64_t d) { return (uint32_t)(d >> 32); };
            bool ok = true;
            auto wait = [&](int b, int parity, int code) { ok = ok && __all_sync(0xffffffffu, mbar_wait_spin(bar(b), parity, abort_flag, p.wait, code)); };
            int g = 0, s3 = 0, ph3 = 0;                        // tile, its K stage and phase
            if (uniform(warp) == 12) {
                const uint64_t x1 = smem_desc_sw128(sX, 16, 1024), kk = smem_desc_sw128(sK, 16, 1024);
                for (int n = 0; ok; ++n) {
                    wait(X_FULL, n & 1, DW_XFULL);
                    if (!ok) break;
                    const int n_tiles = uniform(s_item[n & 1].rows) ? uniform(s_item[n & 1].ntiles) : 0;
                    if (n_tiles == 0) break;
                    for (int j = 0; ok && j < n_tiles; ++j, ++g) {
                        wait(K_FULL + s3, ph3, DW_YFULL);
                        if (g > 0) wait(T1_READ, (g - 1) & 1, DW_READ);
                        if (!ok) break;
                        tc_fence_after();
#pragma unroll
                        for (int ks = 0; ks < D / 16; ++ks) {
                            const uint32_t o = ((ks >> 2) * SUB_BYTES + (ks & 3) * 32) >> 4;
                            mma_ss_elect(tmem, lo(x1) + o, hi(x1), lo(kk) + s3 * STAGE + o, hi(kk), IDESC_T, ks > 0);
                        }
                        tc_commit_elect(bar(T1_FULL));
                        if (j + 1 == n_tiles) tc_commit_elect(bar(X_EMPTY));
                        if (++s3 == kKStages) { s3 = 0; ph3 ^= 1; }
                    }
                }
            } else {
                const uint64_t x2 = smem_desc_sw128(sX + TILE_BYTES, 16, 1024), vv = smem_desc_sw128(sV, 16, 1024);
                const uint64_t km = smem_desc_sw128(sK, SUB_BYTES, 1024);
                // T2(t) = dO V(t)^T for tile t of the launch; `last`: it is the item's last
                auto t2 = [&](int t, bool last) {
                    const int s2 = t & 1;
                    wait(V_FULL + s2, (t >> 1) & 1, DW_YFULL);
                    if (!ok) return;
                    tc_fence_after();
                    const uint32_t d = tmem + (s2 ? 384u : 128u);
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        const uint32_t o = ((ks >> 2) * SUB_BYTES + (ks & 3) * 32) >> 4;
                        mma_ss_elect(d, lo(x2) + o, hi(x2), lo(vv) + s2 * STAGE + o, hi(vv), IDESC_T, ks > 0);
                    }
                    tc_commit_elect(bar(T2_FULL + s2));
                    tc_commit_elect(bar(V_EMPTY + s2));
                    if (last) tc_commit_elect(bar(X_EMPTY));
                };
                for (int n = 0; ok; ++n) {
                    wait(X_FULL, n & 1, DW_XFULL);
                    if (!ok) break;
                    const int n_tiles = uniform(s_item[n & 1].rows) ? uniform(s_item[n & 1].ntiles) : 0;
                    if (n_tiles == 0) break;
                    TileIter it(p.rng + uniform(s_item[n & 1].rng_off), uniform(s_item[n & 1].nrng), uniform(s_item[n & 1].t0), uniform(s_item[n & 1].t1));
                    int t0, valid;
                    t2(g, n_tiles == 1);
                    if (n_tiles > 1) t2(g + 1, n_tiles == 2);
                    for (int j = 0; ok && j < n_tiles; ++j, ++g) {
                        it.next(t0, valid);
                        const int steps = (uniform(valid) + 15) >> 4;
                        wait(DS_DONE + (g & 1), (g >> 1) & 1, DW_DSDONE);
                        if (j == 0 && n > 0) wait(ACC_FREE, (n - 1) & 1, DW_ACCFREE);      // the previous item's dQ has been read
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t ds = tmem + ((g & 1) ? 384u : 128u);
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            if (ks < steps)                  // dS of 32 keys lies over the first half of their T2 columns
                                mma_ts_elect(tmem + 256, ds + (ks >> 1) * 32 + (ks & 1) * 8, lo(km) + s3 * STAGE + ks * (2048 >> 4), hi(km), IDESC_ACC, j > 0 || ks > 0);
                        tc_commit_elect(bar(K_EMPTY + s3));
                        if (++s3 == kKStages) s3 = 0;
                        if (j + 2 < n_tiles) t2(g + 2, j + 3 == n_tiles);
                    }
                    if (ok) tc_commit_elect(bar(ACC_FULL));
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tmem, 512);
    if (threadIdx.x == 0) report_abort(p.status, s_abort);
    if (ANCHOR && blockIdx.x == 0) previous_done();      // an abandoned launch has not waited yet
}

template <int D>
static int dq_tc_d(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *K, const __nv_bfloat16 *V, const float *lse,
                   const float *delta, const __nv_bfloat16 *dO, __nv_bfloat16 *dQ, void *ws, cudaStream_t s) {
    CUtensorMap tmK, tmV;
    if (int r = make_tmap_2d_bf16(&tmK, K, (uint64_t)p->H * p->L, D, 128)) return r;
    if (int r = make_tmap_2d_bf16(&tmV, V, (uint64_t)p->H * p->L, D, 128)) return r;
    DqParams a;
    a.Q = Q; a.dO = dO; a.lse = lse; a.delta = delta; a.dQ = dQ;
    a.part = ws_ptr<__nv_bfloat16>(ws, p->ws.part_o);      // the forward's partial outputs are no longer needed
    a.part_lse = ws_ptr<float>(ws, p->ws.part_lse);
    a.qlist = ws_ptr<int32_t>(ws, p->ws.qlist);
    a.cap_total = (size_t)p->cap_off[p->C];
    a.status = ws_ptr<int>(ws, p->ws.status);
    a.H = p->H; a.L = p->L; a.k = p->k; a.kdiv = SlotDiv::of(p->k);
    a.n_items = (int)p->qitems.size();
    a.scale = p->scale; a.scale_log2 = p->scale * 1.4426950408889634f;
    a.cookie = p->cookie;
    a.wait = WaitBound::of(p->wait_us);
    // seven tiles (Q, dO, three K and two V stages; always the d = 128 footprint, so that CTAs, which each take all of the
    // tensor memory, never share an SM): all an SM has, so the request is what the static variables leave of the limit
    const size_t tiles = (size_t)(2 + kKStages + kVStages) * 128 * 128 * 2;
    size_t smem[2];
    int optin = 0;
    MOC_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, p->device));
    const void *fn[2] = {(const void *)attend_dq_tc_kernel<D, false>, (const void *)attend_dq_tc_kernel<D, true>};
    for (int m = 0; m < 2; ++m) {
        cudaFuncAttributes fa;
        MOC_CUDA_TRY(cudaFuncGetAttributes(&fa, fn[m]));
        smem[m] = std::min(tiles + 1024, (size_t)optin - fa.sharedSizeBytes);
        if (smem[m] < tiles) return MOC_ERR_SHAPE;
        MOC_CUDA_TRY(cudaFuncSetAttribute(fn[m], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem[m]));
    }
    const int *tile_off = ws_ptr<int>(ws, p->ws.tile_off);
    for (int h0 = 0; h0 < p->H; h0 += p->heads_per_group) {
        const int hg = std::min(p->heads_per_group, p->H - h0);
        a.h0 = h0; a.hg = hg;
        if (p->k > 0) {
            a.rng = p->d_chunk_rng;
            a.items = ws_ptr<WorkItem>(ws, p->ws.rtiles);
            a.item_lo = tile_off + (size_t)h0 * p->C;
            a.item_hi = tile_off + (size_t)(h0 + hg) * p->C;
            const long long most = 2LL * hg * (((long long)p->L * p->k + kQTileRows - 1) / kQTileRows + p->C);
            attend_dq_tc_kernel<D, false><<<(unsigned)std::min<long long>(p->n_sm, most), kDqThreads, smem[0], s>>>(tmK, tmV, a);
            MOC_LAUNCH_CHECK();
        }
        a.rng = p->d_anc_rng;
        a.items = p->d_qitems;
        a.item_lo = a.item_hi = nullptr;
        const long long n_anc = 2LL * a.n_items * hg;
        const unsigned anc_grid = (unsigned)std::min<long long>(p->n_sm, n_anc);
        MOC_CUDA_TRY(launch_early(p->k > 0 && backward_overlaps(p), attend_dq_tc_kernel<D, true>, anc_grid, kDqThreads, smem[1], s, tmK, tmV, a));
        MOC_LAUNCH_CHECK();
    }
    return MOC_OK;
}

int launch_dq_tc(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *K, const __nv_bfloat16 *V, const float *lse,
                 const float *delta, const __nv_bfloat16 *dO, __nv_bfloat16 *dQ, void *ws, cudaStream_t s) {
    return p->d == 128 ? dq_tc_d<128>(p, Q, K, V, lse, delta, dO, dQ, ws, s) : dq_tc_d<64>(p, Q, K, V, lse, delta, dO, dQ, ws, s);
}

}  // namespace moc
