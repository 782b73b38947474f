// Tensor-core backward of the sparse attention (selection held constant): dK and dV, and the launch of the whole backward
// (dQ: moc_attend_dq_tc.cu; delta_i = sum_x dO_ix O_ix: moc_attend_scalar.cu).
//
// For a selected (query i, key t) pair:  P = exp(scale q.k - lse_i),  dP = dO_i . v_t,
// dS = P (dP - delta_i);  dV_t += P dO_i,  dK_t += scale dS q_i.
//
// Key stationary: a CTA holds 128 keys of a chunk, X = (K, V), and streams Y = (Q, dO), 128 rows at a time, of every query
// that attends to the chunk - the query rows of the chunks that have it as an anchor, then the chunk's routed query list -
// through rings of three and two stages:
//     T1 = K Q^T,  T2 = V dO^T          (both operands from shared memory, into TMEM)
//     threads (two per TMEM lane) turn T1 into P, then (P, T2) into dS, written back to TMEM as bf16
//     ACC1 += dS Q,  ACC2 += P dO       (A from TMEM, the streamed tile as an MN-major operand)
// lse and delta belong to the column; ACC1 is dK, ACC2 is dV.  A key tile is owned by one CTA, except that in short streams
// several share the query tiles of one that most rows attend (derive_plan): each leaves its fp32 sums, and the last to leave, by an
// atomic counter, adds them in the order of the CTAs.
// Issue order: ACC2(j), T1(j+1), ACC1(j), T2(j+1), so that while the lanes form P(j+1) the pipe runs ACC1(j) and
// T2(j+1), and T1 / T2 are rewritten only after the contraction that reads the P / dS stored over them; ACC2(j) starts on the
// first half of P(j) while the lanes form the second.
// A tile takes 3300 cycles (33k-token clip) for 2048 cycles of MMAs at the pipe's best rate: P, dS and the wait for T1(j+1)
// between them are one chain per tile (at d = 128 two tiles in flight would need 768 columns of tensor memory, of 512; at d = 64,
// where the accumulators take 64 columns each, a second T1 would fit).
// 16 warps: 0-7 the lane threads (two per TMEM lane), 8-11 the producers, 12 and 13 the MMA issuers,
// 14-15 idle (they complete the fourth warpgroup; the lanes take the registers the others give up).  Every mbarrier wait is
// bounded; a wait that runs out flags the workspace status word and the CTA drains and leaves.
#include <algorithm>

#include "moc_common.cuh"
#include "moc_tc.cuh"

namespace moc {

using namespace tc;

enum BwdWait { BW_XFULL = 64, BW_YFULL, BW_YEMPTY, BW_T1FULL, BW_T2FULL, BW_PDONE, BW_DSDONE, BW_ACCFULL, BW_SMEM, BW_READ };

struct BwdParams {
    const __nv_bfloat16 *Q, *K, *V, *dO;
    const float *lse, *delta;
    __nv_bfloat16 *dK, *dV;
    uint32_t cookie;              // what the workspace's status area must hold
    const KTile *ktiles;
    int n_ktiles, n_long;         // tiles per head, and how many of them come first for every head
    int n_split;                  // blocks that are launched for each of those; the tile says how many of them share it
    float4 *split_sum;            // their sums, [tile][block][dK, dV], each as the lane threads hold it
    int *split_done;              // [tile] blocks that have left theirs
    const KeyRange *qry_rng;
    const int *cnt;
    const int32_t *qlist;
    size_t cap_total;
    int *status;
    int H, L, C, k;
    SlotDiv kdiv;
    float scale, scale_log2;
    WaitBound wait;
};

constexpr int kY1Stages = 3, kY2Stages = 2;   // stages of the streamed tiles Y1 (read twice per tile) and Y2
constexpr int kBwdThreads = 512;
constexpr float kLog2e = 1.4426950408889634f;

template <int D>
__global__ void __launch_bounds__(kBwdThreads, 1) attend_dkv_tc_kernel(const __grid_constant__ CUtensorMap tmK,
                                                                      const __grid_constant__ CUtensorMap tmV,
                                                                      const __grid_constant__ CUtensorMap tmQ,
                                                                      const __grid_constant__ CUtensorMap tmdO,
                                                                      const BwdParams p) {
    constexpr int TILE_BYTES = 128 * D * 2;
    constexpr int SUB = D / 64;
    constexpr int SUB_BYTES = 128 * 128;
    constexpr int CH = D / 8;               // 16-byte pieces per row
    constexpr int N_TILES_SMEM = 2 + kY1Stages + kY2Stages;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[24];
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort;
    __shared__ int w_valid, w_h, w_ntiles, w_list;       // w_list: entries of the chunk's query list
    __shared__ int w_skip, w_part, w_parts, w_split, s_last;      // query tiles of the blocks before this one, which is one of w_parts on tile w_split
    __shared__ KTile s_kt;
    // per streamed query, (-lse * log2(e), -delta), for tiles j and j + 1
    __shared__ __align__(16) float s_ld[2][2][128];

    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    // shared tiles: X1 X2 | Y1 stages | Y2 stages
    const uint32_t sX = sbase, sY1 = sbase + 2 * TILE_BYTES, sY2 = sbase + (2 + kY1Stages) * TILE_BYTES;
    auto bar = [&](int i) { return smem_u32(&bars[i]); };
    constexpr int X_FULL = 0, Y1_FULL = 1, Y1_EMPTY = 4, Y2_FULL = 7, Y2_EMPTY = 9, T1_FULL = 11, T2_FULL = 13,
                  P_HALF = 15, P_DONE = 16, DS_DONE = 17, ACC_FULL = 19, T1_ISSUED = 20, RD1 = 22, RD2 = 23, N_BARS = 24;

    // What a block needs before its first load, each in a warp of its own, and one lookup deep.  (By one thread, one after
    // another, with the chunk's anchors walked one by one: 3900 to 6000 cycles, of 45000 for a block of 13 query tiles.)
    if (warp == 0) {
        for (int b = lane; b < N_BARS; b += 32) {
            const int n = b >= Y1_FULL && b < Y1_EMPTY ? 2                       // the ring's two producer warps
                          : b >= Y2_FULL && b < T1_FULL ? 2                      // ... and T2 and ACC2, which both read the stage
                          : b == ACC_FULL ? 2                                    // both issuers
                          : b == P_HALF || b == P_DONE || (b >= DS_DONE && b < ACC_FULL) || b >= RD1 ? 256 : 1;
            mbar_init(bar(b), n);
        }
        fence_barrier_init();
    } else if (warp == 1) {
        if (lane == 0) {
            s_abort = 0;
            s_last = 0;                                    // (stays so if thread 0 gives up before it has counted the block)
            int valid = (*(volatile int *)p.status == 0);
            if (valid && (uint32_t)((volatile int *)p.status)[ST_COOKIE] != p.cookie) {
                atomicCAS(p.status, 0, MOC_ERR_WORKSPACE);      // not this plan's lists: report, touch nothing else
                valid = 0;
            }
            uint32_t dyn_bytes;
            asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_bytes));
            if (valid && (sbase - smem_u32(smem_raw)) + (uint32_t)N_TILES_SMEM * TILE_BYTES > dyn_bytes) {
                // the launch gave less shared memory than the tiles need: report, touch nothing
                if (atomicCAS(p.status, 0, MOC_ERR_TIMEOUT) == 0) p.status[1] = BW_SMEM;
                valid = 0;
            }
            w_valid = valid;
        }
    } else if (warp == 2) {
        if (lane == 0) {
            // block order: the long key tiles of every head, then the others head by head (tiles of one chunk next
            // to each other: they stream the same query rows)
            const int n_long_all = p.n_long * p.H * p.n_split;
            int b = blockIdx.x, hh, ti, part = 0;
            if (b < n_long_all) {
                part = b % p.n_split;
                b /= p.n_split;
                w_split = b;
                hh = b / p.n_long; ti = b - hh * p.n_long;
            } else { b -= n_long_all; const int n_rest = p.n_ktiles - p.n_long; hh = b / n_rest; ti = p.n_long + b - hh * n_rest; }
            const KTile kt = p.ktiles[ti];
            const int n_list = p.cnt[hh * p.C + kt.chunk];
            s_kt = kt;
            w_h = hh;
            w_list = n_list;
            const int nt = kt.n_anc + (n_list + 127) / 128;
            const int parts = min(kt.parts, p.n_split);
            w_part = part;
            w_parts = parts;
            w_skip = (int)((long long)nt * part / parts);
            w_ntiles = (int)((long long)nt * (part + 1) / parts) - w_skip;
        }
    } else if (warp == 8) {
        tmem_alloc(smem_u32(&tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (!w_valid || w_part >= w_parts) {                   // ... or a block that its tile has no use for
        if (warp == 8) tmem_dealloc(tmem_slot, 512);
        if (blockIdx.x == gridDim.x - 1) previous_done();
        return;
    }

    // TMEM columns: T1 [0,128)  T2 [128,256)  ACC1 [256,384)  ACC2 [384,512)
    const uint32_t tmem = tmem_slot;
    const int h = w_h, rows = s_kt.valid, n_tiles = w_ntiles, key0 = s_kt.t0;
    volatile int *abort_flag = &s_abort;

    if (warp < 8) {
        // ------------------------------------------------------------ lane threads: two per TMEM lane (warps w and
        // w + 4 reach the same lanes).  Of the four 32-column chunks of a tile, thread `half` takes chunks half and
        // 2 + half, so that the first two chunks - the first half of P for ACC2 - are finished first.  A thread
        // keeps its 64 P values between the two halves of a tile.
        asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
        const int half = warp >> 2;
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
        const uint64_t c2 = pack2(p.scale_log2, p.scale_log2);
        bool ok = true;
        int s3 = 0, ph3 = 0;                          // Y1 stage of tile jt and its phase
        // A barrier that has completed is looked at some hundred cycles before its wait, behind other work: a wait costs the lanes
        // that much even then, and their chain, P, ACC2, T1 of the next tile, P again, is what a tile takes.  P and dS lie over the first half
        // of the chunk's own columns, which the thread alone has read; side by side, the two threads of a lane waited for each other twice a
        // tile.  (Both, with the same looks ahead in the dQ kernel, the whole backward: 4 heads of 33k tokens 1450 -> 1425 us, 24 heads
        // at the power limit 9.77 -> 9.64 ms, 8 heads of 42k tokens 4.04 -> 3.97, 12 heads of 6.3k, d = 64, 240 -> 234 us, 3 heads of
        // 3.1k 70 -> 67.5.)  What is left of a tile's 2500 cycles (d = 128): 1024 of exponentials, the products after them, and 64 KB of
        // query rows out of L2, 25 bytes a cycle and SM.
        bool t1_early = false, y1_early = false;
        for (int jt = 0; jt < n_tiles; ++jt) {
            const int st = jt & 1;
            ok = t1_early || mbar_wait_spin(bar(T1_FULL + st), (jt >> 1) & 1, abort_flag, p.wait, BW_T1FULL);
            ok = ok && (y1_early || mbar_wait(bar(Y1_FULL + s3), ph3, abort_flag, p.wait, BW_YFULL));
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            // ---- P = exp2(scale log2(e) S - lse log2(e)) from T1
            constexpr uint32_t t2c = 128u;                // T2, then dS
            float pv[64];
            uint32_t sv[2][32];
            tmem_ld32(tmem + lane_off + half * 32, sv[0]);
            tmem_ld32(tmem + lane_off + (2 + half) * 32, sv[1]);
            tmem_wait_ld();
            bool t2_early = false;
#pragma unroll
            for (int rd = 0; rd < 2; ++rd) {
                const int ch = rd * 2 + half;
                const uint32_t (&s)[32] = sv[rd];
                if (rd == 1) t2_early = mbar_test_wait(bar(T2_FULL + st), (jt >> 1) & 1);
                // two columns per packed instruction; four columns' (negated) lse per shared-memory load
#pragma unroll
                for (int x = 0; x < 32; x += 4) {
                    const ulonglong2 l = *reinterpret_cast<const ulonglong2 *>(&s_ld[st][0][ch * 32 + x]);
                    const uint64_t nl[2] = {l.x, l.y};
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        float p0, p1;
                        unpack2(fma2(pack2(__uint_as_float(s[x + 2 * y]), __uint_as_float(s[x + 2 * y + 1])), c2, nl[y]), p0, p1);
                        pv[rd * 32 + x + 2 * y] = ex2(p0);
                        pv[rd * 32 + x + 2 * y + 1] = ex2(p1);
                    }
                }
                {
                    uint32_t ups[16];
#pragma unroll
                    for (int x = 0; x < 16; ++x) ups[x] = bf16x2(pv[rd * 32 + 2 * x], pv[rd * 32 + 2 * x + 1]);
                    tmem_st16(tmem + lane_off + ch * 32, ups);
                    tmem_wait_st();
                    tc_fence_before();
                    mbar_arrive(bar(rd == 0 ? P_HALF : P_DONE));      // the first, then the second 64 columns of P
                }
            }
            // ---- dS = P (dP - delta) from T2, written over T2 columns that have been read
            ok = t2_early || mbar_wait_spin(bar(T2_FULL + st), (jt >> 1) & 1, abort_flag, p.wait, BW_T2FULL);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            uint32_t dpv[2][32];
            tmem_ld32(tmem + lane_off + t2c + half * 32, dpv[0]);
            tmem_ld32(tmem + lane_off + t2c + (2 + half) * 32, dpv[1]);
            tmem_wait_ld();
#pragma unroll
            for (int rd = 0; rd < 2; ++rd) {
                const int ch = rd * 2 + half;
                const uint32_t (&dp)[32] = dpv[rd];
                uint32_t uds[16];
#pragma unroll
                for (int x = 0; x < 32; x += 4) {
                    const ulonglong2 d = *reinterpret_cast<const ulonglong2 *>(&s_ld[st][1][ch * 32 + x]);
                    const uint64_t nd[2] = {d.x, d.y};
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        float a0, a1;
                        unpack2(mul2(pack2(pv[rd * 32 + x + 2 * y], pv[rd * 32 + x + 2 * y + 1]),
                                     add2(pack2(__uint_as_float(dp[x + 2 * y]), __uint_as_float(dp[x + 2 * y + 1])), nd[y])), a0, a1);
                        uds[(x >> 1) + y] = bf16x2(a0, a1);
                    }
                }
                tmem_st16(tmem + lane_off + t2c + ch * 32, uds);
            }
            if (++s3 == kY1Stages) { s3 = 0; ph3 ^= 1; }
            t1_early = mbar_test_wait(bar(T1_FULL + (st ^ 1)), ((jt + 1) >> 1) & 1);
            y1_early = mbar_test_wait(bar(Y1_FULL + s3), ph3);
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(bar(DS_DONE + st));
        }
        // ---- epilogue
        if (ok) {
            ok = mbar_wait(bar(ACC_FULL), 0, abort_flag, p.wait, BW_ACCFULL);
            ok = __all_sync(0xffffffffu, ok);
        }
        if (ok) {
            tc_fence_after();
            // Four lanes write 128 contiguous bytes of a row (tmem_ld_16x256b).  Of the two warps that share the TMEM lanes, each
            // takes 64 columns of all rows (d = 128) or 16 rows (d = 64).
            constexpr int NJ = D / 32;                       // groups of eight rows that this warp has
            const int l4 = lane >> 2, l2 = lane & 3, cb = D == 128 ? half : 0, j0 = D == 128 ? 0 : 2 * half;
            const int slot = w_split, parts = w_parts, me = (half * 4 + (warp & 3)) * 32 + lane;
            constexpr int NV = NJ / 2 * 8;                   // float4s of a thread and side
            auto load = [&](int side, uint32_t (&v)[NJ / 2][32]) {
                __syncwarp();
#pragma unroll
                for (int x = 0; x < NJ / 2; ++x)
                    tmem_ld_16x256b(tmem + lane_off + 256 + side * 128 + ((uint32_t)(x + (j0 >> 1)) << 20) + cb * 64, v[x]);
                tmem_wait_ld();
            };
            auto store = [&](int side, const uint32_t (&v)[NJ / 2][32]) {       // dK = scale ACC1, dV = ACC2
                const float w = side ? 1.f : p.scale;
                __nv_bfloat16 *dst = (side ? p.dV : p.dK) + ((size_t)h * p.L + key0) * D + cb * 64;
#pragma unroll
                for (int y = 0; y < NJ; ++y) {
                    const int row = (warp & 3) * 32 + (j0 + y) * 8 + l4;
                    uint32_t u[8];
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        u[x] = bf16x2(__uint_as_float(v[y >> 1][4 * x + 2 * (y & 1)]) * w, __uint_as_float(v[y >> 1][4 * x + 2 * (y & 1) + 1]) * w);
                    quad_transpose(u, l2);
                    if (row < rows) store_quad(dst + (size_t)row * D, l2, u);
                }
            };
            uint32_t v[NJ / 2][32];
            if (parts == 1) {
#pragma unroll 1
                for (int side = 0; side < 2; ++side) {
                    load(side, v);
                    store(side, v);
                }
            } else {
                // Shared with other blocks: each leaves its sums, and the last one adds them up, in the order of the blocks whichever
                // is last.  They lie where dQ's routed partials were, which dQ's launches have done with.
                previous_done();
                auto sums = [&](int part, int side) { return p.split_sum + (((size_t)slot * p.n_split + part) * 2 + side) * (NV * 256) + me; };
#pragma unroll 1
                for (int side = 0; side < 2; ++side) {
                    load(side, v);
                    float4 *to = sums(w_part, side);
#pragma unroll
                    for (int x = 0; x < NV; ++x) {
                        const uint32_t *f = &v[x >> 3][4 * (x & 7)];
                        to[x * 256] = make_float4(__uint_as_float(f[0]), __uint_as_float(f[1]), __uint_as_float(f[2]), __uint_as_float(f[3]));
                    }
                }
                // (two barriers of the lane threads that serve here alone, once a block, and not a __syncthreads of theirs: every wait here is bounded)
                mbar_arrive(bar(RD1));
                ok = mbar_wait_spin(bar(RD1), 0, abort_flag, p.wait, BW_READ);
                if (threadIdx.x == 0 && ok) {
                    __threadfence();
                    s_last = atomicAdd(p.split_done + slot, 1) == parts - 1;
                    __threadfence();
                }
                mbar_arrive(bar(RD2));
                ok = ok && mbar_wait_spin(bar(RD2), 0, abort_flag, p.wait, BW_READ);
                ok = __all_sync(0xffffffffu, ok);
                if (ok && s_last) {
#pragma unroll 1
                    for (int side = 0; side < 2; ++side) {
                        __syncwarp();
#pragma unroll
                        for (int x = 0; x < NV; ++x)
#pragma unroll
                            for (int y = 0; y < 4; ++y) v[x >> 3][4 * (x & 7) + y] = 0u;
#pragma unroll 1
                        for (int part = 0; part < parts; ++part) {
                            const float4 *from = sums(part, side);
#pragma unroll
                            for (int x = 0; x < NV; ++x) {
                                const float4 f = __ldcg(from + x * 256);
                                uint32_t *a = &v[x >> 3][4 * (x & 7)];
                                a[0] = __float_as_uint(__uint_as_float(a[0]) + f.x);
                                a[1] = __float_as_uint(__uint_as_float(a[1]) + f.y);
                                a[2] = __float_as_uint(__uint_as_float(a[2]) + f.z);
                                a[3] = __float_as_uint(__uint_as_float(a[3]) + f.w);
                            }
                        }
                        store(side, v);
                    }
                }
            }
        }
    } else if (warp < 12) {
        // ------------------------------------------------------------ producers
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        // the key tile itself: K -> X1, V -> X2
        if (warp == 8 && lane == 0) {
            mbar_expect_tx(bar(X_FULL), 2 * TILE_BYTES);
#pragma unroll
            for (int sub = 0; sub < SUB; ++sub) {
                tma_load_2d(sX + sub * SUB_BYTES, &tmK, sub * 64, h * p.L + key0, bar(X_FULL));
                tma_load_2d(sX + TILE_BYTES + sub * SUB_BYTES, &tmV, sub * 64, h * p.L + key0, bar(X_FULL));
            }
        }
        // The queries that attend to this chunk, 128 at a time: Q rows -> Y1 by the first two producer warps, dO rows -> Y2
        // by the other two, each warp 64 rows of every tile.  The two rings run on their own: a tile's Q is fetched as
        // soon as a Y1 stage is free, whatever Y2 waits for (one loop for both left T1 of the next tile waiting for
        // 1400 of a tile's 3900 cycles).  Full tiles of consecutive queries come by TMA, the others by 16-byte
        // asynchronous copies (36 bytes a cycle and SM; TMA row gathers reach 24).
        const int pw = warp - 8, wsub = pw & 1;
        const bool y1 = pw < 2;
        const KeyRange *rng = p.qry_rng + s_kt.rng;
        int n_rng = s_kt.n_rng, r0 = 0, r1 = 0;          // ranges to come; current row range [r0, r1)
        const int n_list = w_list, list0 = s_kt.list;
        const int32_t *list = p.qlist + (size_t)h * p.cap_total + list0;
        int e0 = 0;                                        // next entry of the routed list
        bool ok = true;
        // This lane's two rows of a tile, in two steps so that no load is waited for: the list entries two tiles ahead,
        // then, one tile ahead, the queries with their lse and delta.
        int nx_whole = -1, nx_row = -1, nx_end = 0, nx_e[2] = {-1, -1};
        auto look_ahead = [&]() {
            if (r0 >= r1 && n_rng > 0) {                   // next range of anchor query rows
                r0 = rng->t0; r1 = rng->t1;
                ++rng;
                --n_rng;
            }
            const int i = wsub * 64 + lane;
            nx_whole = -1; nx_row = -1; nx_e[0] = nx_e[1] = -1;
            if (r0 < r1) {
                if (r0 + 128 <= r1) nx_whole = r0;         // a full tile of consecutive queries
                nx_row = r0 + i;
                nx_end = r1;
                r0 += 128;
            } else {
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const int e = e0 + i + 32 * x;
                    if (e < n_list && index_ok((size_t)list0 + e < p.cap_total, p.status, IX_BWD_LIST_POSITION)) nx_e[x] = list[e];
                }
                e0 += 128;
            }
        };
        int whole = -1, q[2] = {-1, -1};
        float q_lse[2] = {INFINITY, INFINITY}, q_del[2] = {0.f, 0.f};
        auto next_rows = [&]() {
            whole = nx_whole;
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                q[x] = -1;
                if (nx_row >= 0) {
                    if (nx_row + 32 * x < nx_end) q[x] = nx_row + 32 * x;
                } else if (nx_e[x] >= 0) {
                    q[x] = p.kdiv.query(nx_e[x]);
                    if (!index_ok((unsigned)q[x] < (unsigned)p.L, p.status, IX_BWD_LIST_ENTRY)) q[x] = -1;
                }
                // a column without a query gets lse = +inf: its P and dS come out as exact zeros
                // (used, that is waited for, when the tile's turn comes)
                q_lse[x] = INFINITY;
                q_del[x] = 0.f;
                if (y1 && q[x] >= 0) {
                    q_lse[x] = p.lse[(size_t)h * p.L + q[x]];
                    q_del[x] = p.delta[(size_t)h * p.L + q[x]];
                }
            }
            look_ahead();
        };
        for (int skip = w_skip; skip > 0; --skip) {        // the query tiles of the blocks before this one
            if (r0 >= r1 && n_rng > 0) {
                r0 = rng->t0; r1 = rng->t1;
                ++rng;
                --n_rng;
            }
            if (r0 < r1) r0 += 128;
            else e0 += 128;
        }
        if (n_tiles > 0) { look_ahead(); next_rows(); }
        int st = 0, ph = 0;                                // stage of tile jt in this warp's ring, and its phase
        int issued = 0;                                    // tiles whose copies this warp has issued
        const int n_st = y1 ? kY1Stages : kY2Stages, b_full = y1 ? Y1_FULL : Y2_FULL, b_empty = y1 ? Y1_EMPTY : Y2_EMPTY;
        const uint32_t ring = y1 ? sY1 : sY2;
        const CUtensorMap *tile_map = y1 ? &tmQ : &tmdO;
        const __nv_bfloat16 *rows_src = (y1 ? p.Q : p.dO) + (size_t)h * p.L * D;
        if (lane == 0) prefetch_tensormap(tile_map);
        for (int jt = 0; ok && jt < n_tiles; ++jt) {
            // the next tile's loads go out first: behind this tile's copies they would queue for a thousand cycles
            const bool by_tile = whole >= 0;
            const int t_whole = whole, t_q[2] = {q[0], q[1]};
            const float t_lse[2] = {q_lse[0], q_lse[1]}, t_del[2] = {q_del[0], q_del[1]};
            if (jt + 1 < n_tiles) next_rows();
            ok = mbar_wait(bar(b_empty + st), ph ^ 1, abort_flag, p.wait, BW_YEMPTY);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const uint32_t dst = ring + st * TILE_BYTES;
            if (by_tile) {
                if (lane == 0) {
#pragma unroll
                    for (int sub = 0; sub < SUB; ++sub)
                        tma_load_2d(dst + sub * SUB_BYTES + wsub * 64 * 128, tile_map, sub * 64, h * p.L + t_whole + wsub * 64, bar(b_full + st));
                }
            } else {
                constexpr int RP = 32 / CH;                // rows per instruction
                const int c16 = lane % CH;
                // (eight rows at a time, in which the swizzle repeats: all 64 of them unrolled were 10 KB of code)
#pragma unroll 1
                for (int r8 = 0; r8 < 64; r8 += 8) {
                    const int rows_q = r8 < 32 ? t_q[0] : t_q[1];
#pragma unroll
                    for (int rb = 0; rb < 8; rb += RP) {
                        const int rl = rb + lane / CH;
                        const int qq = __shfl_sync(0xffffffffu, rows_q, (r8 + rl) & 31);
                        cp_async16(dst + (c16 >> 3) * SUB_BYTES + (wsub * 64 + r8) * 128 + sw128_offset(rl, c16 & 7),
                                   rows_src + (size_t)max(qq, 0) * D + c16 * 8, qq >= 0 ? 16u : 0u);
                    }
                }
            }
            ++issued;
            if (y1) {
                // the lanes have finished with the lse / delta of tile jt - 2
                if (jt >= 2) ok = mbar_wait(bar(DS_DONE + (jt & 1)), ((jt - 2) >> 1) & 1, abort_flag, p.wait, BW_DSDONE);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    s_ld[jt & 1][0][wsub * 64 + x * 32 + lane] = t_lse[x] * -kLog2e;
                    s_ld[jt & 1][1][wsub * 64 + x * 32 + lane] = -t_del[x];
                }
            }
            if (!by_tile) {
                cp_async_wait_all();
                fence_proxy_async_smem();
            }
            __syncwarp();
            // one of the ring's two warps
            if (lane == 0) {
                if (by_tile) mbar_expect_tx(bar(b_full + st), TILE_BYTES / 2);
                else mbar_arrive(bar(b_full + st));
            }
            if (++st == n_st) { st = 0; ph ^= 1; }
        }
        if (*abort_flag) {      // copies already issued must land before the shared memory is released
            cp_async_wait_all();
            int dummy_flag = 0;
            for (int b = 1; b <= n_st; ++b)
                if (issued - b >= 0) mbar_wait(bar(b_full + (issued - b) % n_st), ((issued - b) / n_st) & 1, &dummy_flag, p.wait, BW_YFULL);
        }
    } else {
        // ------------------------------------------------------------ MMA issuers: warp 12 owns the T1 / P side
        // (T1, ACC2), warp 13 the T2 / dS side (T2, ACC1); each side's TMEM columns are touched by its issuer only, so the two
        // instruction streams need no ordering between them and one's waits and commits are covered by the other's MMAs.
        // The streamed tiles are read by both sides: each waits for every tile of either ring that it reads (Q: T1 and
        // ACC1, whose dS(j) follows T1(j); dO: T2 and ACC2, which nothing else orders).  Warps 14 and 15 idle.
        asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
        if (warp <= 13) {                       // the warp stays together, one lane of it issues
            const bool side1 = uniform(warp) == 12;
            const int n_tiles = uniform(w_ntiles);
            constexpr uint32_t IDESC_T = idesc_bf16_f32(128, 128, 0, 0);      // T = X Y^T, both K-major
            constexpr uint32_t IDESC_ACC = idesc_bf16_f32(128, D, 0, 1);      // ACC += (TMEM) Y, Y MN-major
            constexpr uint64_t STAGE = TILE_BYTES >> 4;
            const uint64_t x1 = smem_desc_sw128(sX, 16, 1024), x2 = smem_desc_sw128(sX + TILE_BYTES, 16, 1024);
            const uint64_t y1k = smem_desc_sw128(sY1, 16, 1024), y2k = smem_desc_sw128(sY2, 16, 1024);
            const uint64_t y1m = smem_desc_sw128(sY1, SUB_BYTES, 1024), y2m = smem_desc_sw128(sY2, SUB_BYTES, 1024);
            // only the start-address field (low word) of a descriptor moves: 32-bit arithmetic, never a carry out of it
            auto lo = [](uint64_t d) { return (uint32_t)d; };
            auto hi = [](uint64_t d) { return (uint32_t)(d >> 32); };
            bool ok = true;
            auto wait = [&](int b, int parity, int code) { ok = ok && __all_sync(0xffffffffu, mbar_wait_spin(bar(b), parity, abort_flag, p.wait, code)); };
            // the MMA groups, without their waits and commits
            // (s3 = j mod the Y1 stage count is carried along by the callers: no division on this warp)
            auto t1 = [&](int j, int s3) {  // T1(j) = X1 Y1(j)^T
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    const uint32_t o = ((ks >> 2) * SUB_BYTES + (ks & 3) * 32) >> 4;
                    mma_ss_elect(tmem, lo(x1) + o, hi(x1), lo(y1k) + s3 * (uint32_t)STAGE + o, hi(y1k), IDESC_T, ks > 0);
                }
            };
            auto t2 = [&](int j) {          // T2(j) = X2 Y2(j)^T
                const int s2 = j & 1;
                const uint32_t d = tmem + 128;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    const uint32_t o = ((ks >> 2) * SUB_BYTES + (ks & 3) * 32) >> 4;
                    mma_ss_elect(d, lo(x2) + o, hi(x2), lo(y2k) + s2 * (uint32_t)STAGE + o, hi(y2k), IDESC_T, ks > 0);
                }
            };
            auto acc1 = [&](int j, int s3) {   // ACC1 += dS(j) Y1(j)
                const uint32_t ds = tmem + 128;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)
                    mma_ts_elect(tmem + 256, ds + (ks >> 1) * 32 + (ks & 1) * 8, lo(y1m) + s3 * (uint32_t)STAGE + ks * (2048 >> 4), hi(y1m), IDESC_ACC, j > 0 || ks > 0);
            };
            auto acc2 = [&](int j, int half) {   // ACC2 += P(j) Y2(j), the K steps of one half of P
                const int s2 = j & 1;
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    mma_ts_elect(tmem + 384, tmem + (half * 2 + (ks >> 1)) * 32 + (ks & 1) * 8, lo(y2m) + s2 * (uint32_t)STAGE + (half * 4 + ks) * (2048 >> 4), hi(y2m),
                              IDESC_ACC, j > 0 || half > 0 || ks > 0);
            };
            // MMAs queue up behind one another, so a group goes out as soon as what it reads is there
            wait(X_FULL, 0, BW_XFULL);
            if (side1) {
                // ACC2(j) starts on the first half of P(j); T1(j+1) follows ACC2(j), which reads the P written over T1(j)
                if (n_tiles > 0) {
                    wait(Y1_FULL, 0, BW_YFULL);
                    if (ok) {
                        tc_fence_after();
                        t1(0, 0);
                        tc_commit_elect(bar(T1_FULL));
                    }
                }
                int s3n = 1 % kY1Stages, ph3n = 0;                       // stage and phase of tile j + 1
                for (int j = 0; ok && j < n_tiles; ++j) {
                    const bool more = j + 1 < n_tiles;
                    wait(Y2_FULL + (j & 1), (j >> 1) & 1, BW_YFULL);             // dO of the tile: P(j) comes of Q alone
                    wait(P_HALF, j & 1, BW_PDONE);
                    if (!ok) break;
                    tc_fence_after();
                    acc2(j, 0);
                    if (more) wait(Y1_FULL + s3n, ph3n, BW_YFULL);
                    wait(P_DONE, j & 1, BW_PDONE);
                    if (!ok) break;
                    tc_fence_after();
                    acc2(j, 1);
                    if (more) {
                        t1(j + 1, s3n);
                        tc_commit_elect(bar(T1_FULL + ((j + 1) & 1)));
                    }
                    if (++s3n == kY1Stages) { s3n = 0; ph3n ^= 1; }
                    tc_commit_elect(bar(Y2_EMPTY + (j & 1)));                    // the second of two arrivals
                    // the other side may use the pipe again.  Two barriers: nothing keeps this side from arriving for tile j + 1 before
                    // the other has looked at tile j's, and a wait by parity misses a phase that another one has followed.
                    if (more && lane == 0) mbar_arrive(bar(T1_ISSUED + (j & 1)));
                }
            } else {
                // The lanes wait for T1(j+1) as soon as dS(j) is done, so this side keeps out of the pipe while the
                // other issues it: ACC1(j) waits for that issue, and T2(j+1) follows ACC1(j), which reads the dS written over T2(j).
                if (n_tiles > 0) {
                    wait(Y2_FULL, 0, BW_YFULL);
                    if (ok) {
                        tc_fence_after();
                        t2(0);
                        tc_commit_elect(bar(T2_FULL));
                        tc_commit_elect(bar(Y2_EMPTY));
                    }
                }
                int s3 = 0;                                               // Y1 stage of tile j
                for (int j = 0; ok && j < n_tiles; ++j) {
                    const int jn = j + 1;
                    const bool more = jn < n_tiles;
                    if (more) wait(T1_ISSUED + (j & 1), (j >> 1) & 1, BW_T1FULL);
                    wait(DS_DONE + (j & 1), (j >> 1) & 1, BW_DSDONE);
                    if (!ok) break;
                    tc_fence_after();
                    acc1(j, s3);
                    tc_commit_elect(bar(Y1_EMPTY + s3));                  // at once: a later Q tile waits for this stage
                    if (++s3 == kY1Stages) s3 = 0;
                    if (more) {
                        wait(Y2_FULL + (jn & 1), (jn >> 1) & 1, BW_YFULL);
                        if (!ok) break;
                        t2(jn);
                        tc_commit_elect(bar(T2_FULL + (jn & 1)));
                        tc_commit_elect(bar(Y2_EMPTY + (jn & 1)));    // the first of two arrivals
                    }
                }
            }
            if (ok) tc_commit_elect(bar(ACC_FULL));
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tmem, 512);
    if (threadIdx.x == 0) report_abort(p.status, s_abort);
    if (blockIdx.x == gridDim.x - 1) previous_done();    // nothing here depends on dQ's launches, but what follows may
}

template <int D>
static int attend_bwd_tc_d(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *K, const __nv_bfloat16 *V,
                           const __nv_bfloat16 *O, const float *lse, const __nv_bfloat16 *dO, const int32_t *sel,
                           __nv_bfloat16 *dQ, __nv_bfloat16 *dK, __nv_bfloat16 *dV, void *ws, cudaStream_t s) {
    float *delta = ws_ptr<float>(ws, p->ws.delta);
    const int n_split = dkv_split(p);
    int *split_done = ws_ptr<int>(ws, p->ws.pool_done);
    if (int r = launch_delta(p, O, dO, delta, split_done, n_split > 1 ? p->n_long_ktiles * p->H : 0, s)) return r;
    CUtensorMap tmK, tmV, tmQ, tmdO;       // Q and dO: tiles of 64 rows
    if (int r = make_tmap_2d_bf16(&tmK, K, (uint64_t)p->H * p->L, D, 128)) return r;
    if (int r = make_tmap_2d_bf16(&tmV, V, (uint64_t)p->H * p->L, D, 128)) return r;
    if (int r = make_tmap_2d_bf16(&tmQ, Q, (uint64_t)p->H * p->L, D, 64)) return r;
    if (int r = make_tmap_2d_bf16(&tmdO, dO, (uint64_t)p->H * p->L, D, 64)) return r;
    BwdParams a;
    a.Q = Q; a.K = K; a.V = V; a.dO = dO; a.lse = lse; a.delta = delta;
    a.cookie = p->cookie;
    a.wait = WaitBound::of(p->wait_us);
    a.dK = dK; a.dV = dV;
    a.ktiles = p->d_ktiles; a.n_ktiles = (int)p->ktiles.size(); a.n_long = p->n_long_ktiles;
    a.n_split = n_split; a.split_sum = ws_ptr<float4>(ws, p->ws.part_o); a.split_done = split_done;
    a.qry_rng = p->d_qry_rng;
    a.cnt = ws_ptr<int>(ws, p->ws.cnt);
    a.qlist = ws_ptr<int32_t>(ws, p->ws.qlist);
    a.cap_total = (size_t)p->cap_off[p->C];
    a.status = ws_ptr<int>(ws, p->ws.status);
    a.H = p->H; a.L = p->L; a.C = p->C; a.k = p->k; a.kdiv = SlotDiv::of(p->k);
    a.scale = p->scale; a.scale_log2 = p->scale * kLog2e;
    // seven tiles (X1 X2, three Y1 stages, two Y2 stages) and the slack that aligns them to 1024 bytes; at
    // d = 128 that is all an SM has, so the request is what the kernel's static variables leave of the limit
    const size_t tiles = (size_t)(2 + kY1Stages + kY2Stages) * 128 * D * 2;
    int optin = 0;
    cudaFuncAttributes fa;
    MOC_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, p->device));
    MOC_CUDA_TRY(cudaFuncGetAttributes(&fa, attend_dkv_tc_kernel<D>));
    const size_t smem = std::min(tiles + 1024, (size_t)optin - fa.sharedSizeBytes);
    if (smem < tiles) return MOC_ERR_SHAPE;
    MOC_CUDA_TRY(cudaFuncSetAttribute(attend_dkv_tc_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (int r = launch_dq_tc(p, Q, K, V, lse, delta, dO, dQ, ws, s)) return r;
    MOC_CUDA_TRY(launch_early(backward_overlaps(p), attend_dkv_tc_kernel<D>, (unsigned)((p->ktiles.size() + (size_t)(n_split - 1) * p->n_long_ktiles) * p->H), kBwdThreads, smem, s, tmK, tmV, tmQ, tmdO, a));
    MOC_LAUNCH_CHECK();
    return MOC_OK;
}

int launch_attend_bwd_tc(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *K, const __nv_bfloat16 *V,
                         const __nv_bfloat16 *O, const float *lse, const __nv_bfloat16 *dO, const int32_t *sel,
                         __nv_bfloat16 *dQ, __nv_bfloat16 *dK, __nv_bfloat16 *dV, void *ws, cudaStream_t s) {
    return p->d == 128 ? attend_bwd_tc_d<128>(p, Q, K, V, O, lse, dO, sel, dQ, dK, dV, ws, s)
                       : attend_bwd_tc_d<64>(p, Q, K, V, O, lse, dO, sel, dQ, dK, dV, ws, s);
}

}  // namespace moc
