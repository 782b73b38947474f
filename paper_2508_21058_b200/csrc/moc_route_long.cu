// Routing where many chunks are picked per query: scores, causal mask, anchors removed, top-k and the query lists, as in
// moc_route.cu (same products, same order of the picks), with another selection.
//
// A thread per row that keeps its list sorted in registers pays five instructions per entry of the list for each candidate: from some
// twenty entries on that, and not the scores, is the time of routing (264k tokens, 1008 columns, 2 heads, 118 picks: 6.7 ms).  Here a
// row's threads only count: of the scores in tensor memory those that reach a threshold, until a few more than k do, two or three times; those
// alone are kept, and sorted by a whole warp.  (2 heads, a thread per row -> this, us: 264k tokens, 1008 columns: 20 picks 971 -> 755, 30 1122 ->
// 805, 60 3063 -> 1300, 118 6706 -> 1800; 504 columns: 20 680 -> 493, 32 802 -> 592, 64 2173 -> 998; 40k tokens, 200 columns, 20 picks 96 -> 82.)
// What bounds it now (118 picks, per tile of 122,000 cycles): the sorts 44,500, the list entries, four bytes here and there, 26,600, counting 17,900.
// Scores through a scratch in L2, so that a warp could hold a row, took 1.4 times as long: 64 KB a step each way.
//
// Persistent, one CTA per SM; the 128-query tiles ("units") are dealt round-robin, all heads' first tiles first (so that a query list is
// nearly in the order of the stream: head by head, with twice to six times as many tiles of a head under way, attention over the lists took 6 %
// longer).  18 warps:
//   warps 0-15  selection.  Four warps share the 32 rows of a quarter of the tensor memory, a thread per row, and each looks at a quarter of the
//               columns: sums for a first guess, counts, then the survivors into the row's list in shared memory.  At most 512 columns at a time
//               are in tensor memory; with more, the survivors so far are counted and thinned along with the next ones.  Then a row at a
//               time, a warp each: sort, sel_idx, pick counts; a range of each picked chunk's list is reserved by one global atomic per
//               (unit, chunk), and the list entries are written behind the next unit's scores;
//   warp 16     TMA producer: Q tiles, and the descriptors' three bf16 terms, 128 columns of one term at a time, through a ring;
//   warp 17     MMA issuer: 3 x d/16 MMAs per step of 128 columns, into one of four accumulators; the next unit's while this one's are sorted.
// Every mbarrier wait is bounded; one that runs out flags the workspace status word.
#include <float.h>
#include <limits.h>
#include <algorithm>

#include "moc_common.cuh"
#include "moc_route.cuh"
#include "moc_tc.cuh"

namespace moc {

using namespace tc;

constexpr int kLongSel = 16, kLongThreads = 32 * (kLongSel + 2), kLongRows = 128, kLongStep = 128, kLongAcc = 4, kLongSlots = 6;
// A row's survivors, 32 N of them: a score and a column each, with the padding that keeps a warp's accesses to 32 rows, and to one, apart in the
// banks.  Up to 128 they are in shared memory, beyond that in the workspace, where attention's partials will lie.
constexpr int kQueueShared = 4;
template <int N> constexpr int kQueueBytes = (32 * N + 1) * 4 + (32 * N + 2) * 2;

enum RouteLongWait { RL_QFULL = 48, RL_QEMPTY, RL_DFULL, RL_DEMPTY, RL_ACCFULL, RL_ACCEMPTY, RL_SYNC };

struct RouteLongParams {
    float *scratch;             // long rows' survivors, CTA by CTA
    int32_t *sel;
    float *part_lse;
    int *cnt;
    int32_t *qlist;
    const int32_t *tok_chunk;
    const uint32_t *cand_c;     // [C][cwords] candidate columns per query chunk
    const int32_t *lim;         // [C] prefix mode: the candidates of a query in chunk c are the columns [0, lim[c])
    const int32_t *reach;       // [C] columns any query up to chunk c can pick from
    const int32_t *col_chunk;   // [ncol] chunk of a score column
    const int32_t *cap_off;
    int *status;
    int H, L, C, c_pad, ncol, k, cwords, prefix;
    int n_units;
    int d_rows;                 // columns per step of the ring: 128, or all of them
    int q_stages, d_slots;
    int hists;                  // pick counters of two units (a unit's list entries are written behind the next one's scores), or of one
    int *tile_off;
    uint32_t cookie;
    size_t cap_total;
    WaitBound wait;
};

// Scores are counted, stored, thinned and sorted in one order: numbers, subnormal ones and -0 all taken as zero.  It is written out here, so
// that it does not hang on the compiler's flags: a store that told a subnormal threshold from zero, where the count did not, left
// fewer survivors than had been counted.
__device__ __forceinline__ int reaches(float f, float thr) {
    int r;
    asm("{\n\t.reg .pred p;\n\tsetp.ge.ftz.f32 p, %1, %2;\n\tselp.s32 %0, 1, 0, p;\n\t}" : "=r"(r) : "f"(f), "f"(thr));
    return r;
}
// (and, of equal ones, in the columns before `before`)
__device__ __forceinline__ int reaches(float f, int col, float thr, int before) {
    int r;
    asm("{\n\t.reg .pred p, q;\n\tsetp.lt.s32 p, %2, %4;\n\tsetp.eq.and.ftz.f32 p, %1, %3, p;\n\tsetp.gt.or.ftz.f32 q, %1, %3, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(r) : "f"(f), "r"(col), "f"(thr), "r"(before));
    return r;
}
// Scores as unsigned integers of the same order (of those that count as zero, subnormal ones keep theirs), and back.
__device__ __forceinline__ uint32_t ordered(float f) {
    const uint32_t b = __float_as_uint(f);
    return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
}
__device__ __forceinline__ float from_ordered(uint32_t u) { return __uint_as_float((u & 0x80000000u) ? u ^ 0x80000000u : ~u); }
// ... and with all that count as zero as +0.
__device__ __forceinline__ uint32_t sort_key(float f) {
    float z;
    asm("add.ftz.f32 %0, %1, 0f00000000;" : "=f"(z) : "f"(f));
    return ordered(z);
}

// The value that a standard normal variable exceeds with probability p (Abramowitz and Stegun 26.2.23, error below 5e-4).
__device__ __forceinline__ float normal_above(float p) {
    const float t = sqrtf(-2.f * __logf(fminf(p, 1.f - p)));
    const float z = t - (2.515517f + t * (0.802853f + t * 0.010328f)) / (1.f + t * (1.432788f + t * (0.189269f + t * 0.001308f)));
    return p <= 0.5f ? z : -z;
}

// R rows of keys of a warp, entry e = lane * N + i, sorted descending by a bitonic network, side by side (one row's shuffles wait for another's).
template <int R, int N>
__device__ __forceinline__ void warp_sort(uint64_t (&keys)[R][N], int lane) {
#pragma unroll
    for (int run = 2; run <= 32 * N; run <<= 1)
#pragma unroll
        for (int step = run >> 1; step > 0; step >>= 1)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                uint64_t(&key)[N] = keys[r];
                if (step >= N) {
                    // the other entry is another lane's: the lower entry keeps the larger key in a descending run
                    const bool down = run >= 32 * N || ((lane * N) & run) == 0, lower = (lane & (step / N)) == 0;
#pragma unroll
                    for (int i = 0; i < N; ++i) {
                        const uint64_t other = __shfl_xor_sync(0xffffffffu, key[i], step / N);
                        if ((key[i] < other) == (down == lower)) key[i] = other;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < N; ++i)
                        if (!(i & step)) {
                            const bool down = run >= 32 * N || ((lane * N + i) & run) == 0;
                            const uint64_t a = key[i], b = key[i | step];
                            const bool swap = (a < b) == down;
                            key[i] = swap ? b : a;
                            key[i | step] = swap ? a : b;
                        }
                }
            }
}

template <int D, int N>
__global__ void __launch_bounds__(kLongThreads, 1) route_long_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmD,
                                                                     const RouteLongParams p) {
    constexpr int SUB = D / 64, Q_SUB_BYTES = kLongRows * 128, Q_TILE_BYTES = SUB * Q_SUB_BYTES, CAP = 32 * N;
    constexpr uint32_t ALL = 0xffffffffu;
    extern __shared__ uint8_t smem_raw[];
    enum { Q_FULL = 0, Q_EMPTY = 2, D_FULL = 4, D_EMPTY = D_FULL + kLongSlots, ACC_FULL = D_EMPTY + kLongSlots, ACC_EMPTY = ACC_FULL + kLongAcc,
           SYNC = ACC_EMPTY + kLongAcc, ROWS, N_BARS = ROWS + 4 };
    __shared__ __align__(8) uint64_t bars[N_BARS];
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort;
    // of each row, by the four warps that look at it: sum of scores, of squares, candidates; and scores that reach a threshold
    __shared__ float s_stat[3][4][kLongRows];
    __shared__ int s_count[2][4][kLongRows];

    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *gbase = smem_raw + (sbase - smem_u32(smem_raw));
    // shared memory: descriptor ring (a slot: SUB sub-tiles of d_rows x 128 bytes) | Q stages | survivors, CAP per row | one or two histograms
    const uint32_t d_sub_bytes = p.d_rows * 128, d_slot_bytes = (SUB * d_sub_bytes + 1023) & ~1023u;
    const uint32_t sD = sbase, sQ = sD + p.d_slots * d_slot_bytes;
    float *queue_base = reinterpret_cast<float *>(gbase + (sQ - sbase) + p.q_stages * Q_TILE_BYTES);
    int *hist_base = reinterpret_cast<int *>(queue_base + (N <= kQueueShared ? kLongRows * kQueueBytes<N> / 4 : 0));
    auto bar = [&](int i) { return smem_u32(&bars[i]); };

    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int t = 0; t < 2; ++t) { mbar_init(bar(Q_FULL + t), 1); mbar_init(bar(Q_EMPTY + t), 1); }
        for (int t = 0; t < kLongSlots; ++t) { mbar_init(bar(D_FULL + t), 1); mbar_init(bar(D_EMPTY + t), 1); }
        for (int t = 0; t < kLongAcc; ++t) { mbar_init(bar(ACC_FULL + t), 1); mbar_init(bar(ACC_EMPTY + t), kLongSel); }
        mbar_init(bar(SYNC), kLongSel);
        for (int t = 0; t < 4; ++t) mbar_init(bar(ROWS + t), kLongSel / 4);
        fence_barrier_init();
    }
    for (int x = threadIdx.x; x < p.hists * p.C; x += kLongThreads) hist_base[x] = 0;
    if (warp == kLongSel) {
        tmem_alloc(smem_u32(&tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    volatile int *abort_flag = &s_abort;

    // columns that the rows of tile t can pick from, and the steps that hold them
    auto reach_of = [&](int t) { return p.reach[p.tok_chunk[min(p.L, (t + 1) * kLongRows) - 1]]; };
    auto steps_of = [&](int reach) { return max(1, (reach + kLongStep - 1) / kLongStep); };
    auto columns = [&](int sb, int reach) { return max(16, min(min(kLongStep, p.c_pad - sb * kLongStep), (reach - sb * kLongStep + 15) & ~15)); };

    if (warp == kLongSel) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            prefetch_tensormap(&tmQ);
            prefetch_tensormap(&tmD);
            int qn = 0, dn = 0, slot = 0;
            uint32_t dph = 0;
            bool ok = true;
            for (int u = blockIdx.x; ok && u < p.n_units; u += gridDim.x) {
                const int t = u / p.H, h = u - t * p.H, steps = steps_of(reach_of(t));
                const int st = p.q_stages == 2 ? qn & 1 : 0;
                const uint32_t ph = (p.q_stages == 2 ? qn >> 1 : qn) & 1;
                ok = mbar_wait(bar(Q_EMPTY + st), ph ^ 1, abort_flag, p.wait, RL_QEMPTY);
                if (!ok) break;
                mbar_expect_tx(bar(Q_FULL + st), Q_TILE_BYTES);
#pragma unroll
                for (int sub = 0; sub < SUB; ++sub)
                    tma_load_2d(sQ + st * Q_TILE_BYTES + sub * Q_SUB_BYTES, &tmQ, sub * 64, h * p.L + t * kLongRows, bar(Q_FULL + st));
                ++qn;
                for (int x = 0; x < 3 * steps; ++x) {
                    const int sb = x / 3, term = x - 3 * sb;
                    ok = mbar_wait(bar(D_EMPTY + slot), dph ^ 1, abort_flag, p.wait, RL_DEMPTY);
                    if (!ok) break;
                    mbar_expect_tx(bar(D_FULL + slot), SUB * d_sub_bytes);
#pragma unroll
                    for (int sub = 0; sub < SUB; ++sub)
                        tma_load_2d(sD + slot * d_slot_bytes + sub * d_sub_bytes, &tmD, sub * 64, (h * 3 + term) * p.c_pad + sb * kLongStep, bar(D_FULL + slot));
                    ++dn;
                    if (++slot == p.d_slots) { slot = 0; dph ^= 1; }
                }
            }
            if (*abort_flag) {
                // drain: copies already issued must land before the CTA's shared memory is released
                int dummy_flag = 0;
                for (int b = 1; b <= p.q_stages; ++b)
                    if (qn - b >= 0) mbar_wait(bar(Q_FULL + (qn - b) % p.q_stages), ((qn - b) / p.q_stages) & 1, &dummy_flag, p.wait, RL_QFULL);
                for (int b = 1; b <= p.d_slots; ++b)
                    if (dn - b >= 0) mbar_wait(bar(D_FULL + (dn - b) % p.d_slots), ((dn - b) / p.d_slots) & 1, &dummy_flag, p.wait, RL_DFULL);
            }
        }
    } else if (warp == kLongSel + 1) {
        // ------------------------------------------------------------ MMA issuer (the warp stays together, one lane of it issues)
        const uint64_t q_desc0 = smem_desc_sw128(sQ, 16, 1024), d_desc0 = smem_desc_sw128(sD, 16, 1024);
        int qn = 0, slot = 0;
        uint32_t dph = 0, acc_phase = 0;
        bool ok = true;
        auto wait = [&](int b, uint32_t parity, int code) { return __all_sync(ALL, mbar_wait(bar(b), parity, abort_flag, p.wait, code)) != 0; };
        for (int u = blockIdx.x; ok && u < p.n_units; u += gridDim.x) {
            const int reach = uniform(reach_of(u / p.H)), steps = steps_of(reach);
            const int st = p.q_stages == 2 ? qn & 1 : 0;
            ok = wait(Q_FULL + st, (p.q_stages == 2 ? qn >> 1 : qn) & 1, RL_QFULL);
            ++qn;
            const uint64_t qd = q_desc0 + (uint64_t)(st * (Q_TILE_BYTES >> 4));
            for (int sb = 0; ok && sb < steps; ++sb) {
                const int a = sb % kLongAcc;
                ok = wait(ACC_EMPTY + a, ((acc_phase >> a) & 1) ^ 1, RL_ACCEMPTY);
                acc_phase ^= 1u << a;
                const uint32_t idesc = idesc_bf16_f32(128, columns(sb, reach), 0, 0);
                for (int term = 0; ok && term < 3; ++term) {
                    ok = wait(D_FULL + slot, dph, RL_DFULL);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t dd = d_desc0 + (uint64_t)((slot * d_slot_bytes) >> 4);
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks)
                        mma_ss_elect(tmem + a * kLongStep, (uint32_t)qd + (((ks >> 2) * Q_SUB_BYTES + (ks & 3) * 32) >> 4), (uint32_t)(qd >> 32),
                                     (uint32_t)dd + (((ks >> 2) * d_sub_bytes + (ks & 3) * 32) >> 4), (uint32_t)(dd >> 32), idesc, (term | ks) != 0);
                    tc_commit_elect(bar(D_EMPTY + slot));
                    if (++slot == p.d_slots) { slot = 0; dph ^= 1; }
                }
                if (ok) tc_commit_elect(bar(ACC_FULL + a));
            }
            if (ok) tc_commit_elect(bar(Q_EMPTY + st));
        }
    } else {
        // ------------------------------------------------------------ selection
        const int quad = warp & 3, part = warp >> 2;          // 32 rows (TMEM lanes), of which this warp looks at every fourth block of 32 columns
        const int row = quad * 32 + lane;                     // this thread's row while the scores are looked at; then a warp has a row, quad * 32 + part + 4 y
        // a row's survivors: scores and columns
        float *const sc = N <= kQueueShared ? queue_base : p.scratch + (size_t)blockIdx.x * (kLongRows * kQueueBytes<N> / 4);
        uint16_t *const co = reinterpret_cast<uint16_t *>(sc + kLongRows * (CAP + 1));
        auto sc_at = [&](int r, int e) -> float & { return sc[r * (CAP + 1) + e]; };
        auto co_at = [&](int r, int e) -> uint16_t & { return co[r * (CAP + 2) + e]; };
        uint32_t acc_phase = 0, sync_phase = 0;               // bit s: parity of accumulator s's next phase; bit 0: of SYNC, bit 1: of ROWS
        int pass_no = 0;
        bool ok = true;
        auto meet = [&](int b, uint32_t bit) {                // warps that meet, bounded
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(b));
            const bool o = mbar_wait(bar(b), (sync_phase & bit) ? 1 : 0, abort_flag, p.wait, RL_SYNC);
            sync_phase ^= bit;
            return __all_sync(ALL, o) != 0;
        };
        auto all_warps = [&]() { return meet(SYNC, 1); };
        auto same_rows = [&]() { return meet(ROWS + quad, 2); };
        // the list entries of the eight rows that this warp has picked for, from the ranges that have been reserved
        auto write_entries = [&](int h, int t, int *hist) {
            int32_t *list = p.qlist + (size_t)h * p.cap_total;
            constexpr int B = N <= 4 ? 4 : 16 / N;            // rows at a time
#pragma unroll 1
            for (int y0 = 0; y0 < 8; y0 += B) {
                int j[B][N];
                const int i0 = t * kLongRows + quad * 32 + part + 4 * y0;
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    const int32_t *out = p.sel + ((size_t)h * p.L + i0 + 4 * b) * p.k + lane * N;
#pragma unroll
                    for (int e = 0; e < N; ++e) {
                        j[b][e] = -1;
                        if (i0 + 4 * b < p.L && lane * N + e < p.k) j[b][e] = out[e];
                    }
                }
#pragma unroll
                for (int b = 0; b < B; ++b)
#pragma unroll
                    for (int e = 0; e < N; ++e) {
                        if (j[b][e] < 0) continue;
                        const int at = atomicAdd(&hist[j[b][e]], 1);
                        if (index_ok((size_t)at < p.cap_total, p.status, IX_APPEND_POSITION)) list[at] = (i0 + 4 * b) * p.k + lane * N + e;
                    }
            }
        };
        int last_h = 0, last_t = -1, n = 0;
        for (int u = blockIdx.x; u < p.n_units; u += gridDim.x, ++n) {
            const int t = u / p.H, h = u - t * p.H;
            const int my_i = t * kLongRows + row, my_c = my_i < p.L ? p.tok_chunk[my_i] : 0, my_lim = p.prefix && my_i < p.L ? p.lim[my_c] : 0;
            const int reach = reach_of(t), steps = steps_of(reach);
            int *hist = hist_base + (p.hists == 2 ? (n & 1) * p.C : 0), *other = hist_base + (~n & 1) * p.C;
            // this row's candidates among the 32 columns from j0 on
            auto candidates = [&](int j0) -> uint32_t {
                if (p.prefix) {
                    const int m = my_lim - j0;
                    return m <= 0 ? 0u : (m >= 32 ? ALL : ((1u << m) - 1u));
                }
                return my_i < p.L ? p.cand_c[(size_t)my_c * p.cwords + (j0 >> 5)] : 0u;
            };
            float n_cand = 0.f, sum = 0.f, sq = 0.f;           // of the columns so far
            int len = 0;                                       // survivors
            for (int seg = 0; ok && seg < steps; seg += kLongAcc) {
                const int n_st = min(kLongAcc, steps - seg);
                // the warp's blocks of the segment: scores of 32 rows, and whether all are candidates; where not, the others are `none`
                auto each_block = [&](uint32_t none, auto &&f) __attribute__((always_inline)) {
#pragma unroll 1
                    for (int s = 0; s < n_st; ++s) {
                        const int j0 = (seg + s) * kLongStep + part * 32;
                        if (j0 >= reach) break;
                        uint32_t v[32];
                        tmem_ld32(tmem + s * kLongStep + part * 32 + ((uint32_t)(quad * 32) << 16), v);
                        const uint32_t cand = candidates(j0);
                        tmem_wait_ld();
                        if (!__all_sync(ALL, cand == ALL)) {
#pragma unroll
                            for (int c = 0; c < 32; ++c) v[c] = ((cand >> c) & 1u) ? v[c] : none;
                        }
                        f(v, j0, cand);
                    }
                };
                for (int s = 0; ok && s < n_st; ++s) ok = mbar_wait(bar(ACC_FULL + s), (acc_phase >> s) & 1, abort_flag, p.wait, RL_ACCFULL);
                ok = __all_sync(ALL, ok);
                if (!ok) break;
                acc_phase ^= (1u << n_st) - 1;
                tc_fence_after();
                {
                    uint64_t s2 = 0, q2 = 0;
                    int nc = 0;
                    each_block(0u, [&](const uint32_t (&v)[32], int, uint32_t cand) {
                        nc += __popc(cand);
#pragma unroll
                        for (int c = 0; c < 32; c += 2) {
                            const uint64_t x = pack2(__uint_as_float(v[c]), __uint_as_float(v[c + 1]));
                            s2 = add2(s2, x);
                            q2 = fma2(x, x, q2);
                        }
                    });
                    float a, b;
                    unpack2(s2, a, b);
                    s_stat[0][part][row] = a + b;
                    unpack2(q2, a, b);
                    s_stat[1][part][row] = a + b;
                    s_stat[2][part][row] = (float)nc;
                }
                ok = same_rows();
                if (!ok) break;
#pragma unroll
                for (int x = 0; x < 4; ++x) { sum += s_stat[0][x][row]; sq += s_stat[1][x][row]; n_cand += s_stat[2][x][row]; }
                // A threshold that at least k and at most CAP scores reach, of the survivors so far and of the segment.  First guess: as if the
                // scores were normally distributed, then between the nearest on either side on that assumption, every fourth time by halving the interval of
                // ordered integers; `low`: more than CAP reach it, `high`: fewer than k do.  Where the two meet, more than CAP scores are equal: of
                // those at the threshold the ones before column `before` are taken, which is found in the same way.
                const float inv = 1.f / n_cand, mean = sum * inv, sd = sqrtf(fmaxf(sq * inv - mean * mean, 0.f));
                const float z = normal_above(0.5f * (p.k + CAP) * inv);
                uint32_t low = ordered(-FLT_MAX), high = ordered(INFINITY) + 1;
                float z_low = NAN, z_high = NAN;               // where their counts lie on the normal distribution, once they have been seen
                int before = INT_MAX, b_low = 0, b_high = 0;
                bool found = n_cand <= (float)CAP;
                float thr = found ? -FLT_MAX : mean + z * sd;
                auto in_between = [&](bool guess) {            // keeps the threshold inside the interval
                    uint32_t key = ordered(thr);
                    if (!guess || !(key > low && key < high)) key = low + ((high - low) >> 1);
                    thr = from_ordered(key);
                };
                if (!found) in_between(true);
                const int max_len = __reduce_max_sync(ALL, len);
                int kept = 0, at = 0, total = 0;               // survivors so far that stay; where this thread's new ones go; all
                bool ties = false;                             // some row of the warp's has a column bound
                for (int it = 0;; ++it) {
                    int c_new = 0, c_old = 0;
                    if (!ties) {
                        each_block(0xff800000u, [&](const uint32_t (&v)[32], int, uint32_t) {
#pragma unroll
                            for (int c = 0; c < 32; ++c) c_new += reaches(__uint_as_float(v[c]), thr);
                        });
                    } else {
                        each_block(0xff800000u, [&](const uint32_t (&v)[32], int j0, uint32_t) {
#pragma unroll
                            for (int c = 0; c < 32; ++c) c_new += reaches(__uint_as_float(v[c]), j0 + c, thr, before);
                        });
                    }
#pragma unroll 4
                    for (int e = part; e < max_len; e += 4)
                        if (e < len) c_old += ties ? reaches(sc_at(row, e), co_at(row, e), thr, before) : reaches(sc_at(row, e), thr);
                    s_count[pass_no & 1][part][row] = c_new | c_old << 16;
                    ok = same_rows();
                    if (!ok) break;
                    kept = at = total = 0;
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int c = s_count[pass_no & 1][x][row];
                        kept += c >> 16;
                        total += c & 0xffff;
                        at += x < part ? c & 0xffff : 0;
                    }
                    ++pass_no;
                    total += kept;
                    at += kept;
                    found = found || (total >= p.k && total <= CAP);
                    if (__all_sync(ALL, found)) break;
                    if (!found) {
                        if (before == INT_MAX) {
                            const float z_thr = normal_above(fmaxf((float)total, 0.5f) * inv);
                            const float t = thr;
                            if (total > CAP) { low = ordered(t); z_low = z_thr; }
                            else { high = ordered(t); z_high = z_thr; }
                            if (high - low <= 1) {
                                thr = from_ordered(low);
                                b_high = 1 << 16;
                            } else {
                                const float t_low = from_ordered(low), t_high = from_ordered(high);
                                thr = t_low + (t_high - t_low) * ((z - z_low) / (z_high - z_low));      // between the two, or, with one, by the deviation
                                if (!(z_low < z_high)) thr = t + sd * (z - z_thr);
                                in_between((it & 3) != 3);
                            }
                        } else if (total > CAP) b_high = before;
                        else b_low = before;
                        if (b_high) before = b_low + ((b_high - b_low) >> 1);
                        if (b_high && b_high - b_low <= 1) { before = b_high; found = true; }      // (scores that are not numbers were counted on)
                    }
                    ties = __any_sync(ALL, before != INT_MAX);
                }
                if (!ok) break;
                // the survivors so far that stay, then the segment's
                if (seg > 0) {
                    if (part == 0) {
                        int to = 0;
#pragma unroll 1
                        for (int e0 = 0; e0 < max_len; e0 += 8) {      // (eight are read before any of them is overwritten)
                            float f[8];
                            int c[8];
#pragma unroll
                            for (int x = 0; x < 8; ++x) {
                                const int e = min(e0 + x, CAP - 1);
                                f[x] = sc_at(row, e);
                                c[x] = co_at(row, e);
                            }
#pragma unroll
                            for (int x = 0; x < 8; ++x)
                                if (e0 + x < len && reaches(f[x], c[x], thr, before)) { sc_at(row, to) = f[x]; co_at(row, to) = (uint16_t)c[x]; ++to; }
                        }
                    }
                    ok = same_rows();
                    if (!ok) break;
                }
                // (where this thread's entries have to end: survivors are stored by the rule that they were counted by)
                const int end = at + (s_count[(pass_no - 1) & 1][part][row] & 0xffff);
                // a survivor's score and column, and the places of the next one's
                auto store = [](auto &a_sc, auto &a_co, float f, int col, int take) __attribute__((always_inline)) {
                    if constexpr (N <= kQueueShared)
                        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %4, 0;\n\t@p st.shared.f32 [%0], %2;\n\t@p st.shared.u16 [%1], %3;\n\t"
                                     "@p add.u32 %0, %0, 4;\n\t@p add.u32 %1, %1, 2;\n\t}" : "+r"(a_sc), "+r"(a_co) : "f"(f), "h"((uint16_t)col), "r"(take) : "memory");
                    else
                        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %4, 0;\n\t@p st.global.f32 [%0], %2;\n\t@p st.global.u16 [%1], %3;\n\t"
                                     "@p add.u64 %0, %0, 4;\n\t@p add.u64 %1, %1, 2;\n\t}" : "+l"(a_sc), "+l"(a_co) : "f"(f), "h"((uint16_t)col), "r"(take) : "memory");
                };
                auto place = [](auto &x) { if constexpr (N <= kQueueShared) return smem_u32(&x); else return (uint64_t)__cvta_generic_to_global(&x); };
                auto a_sc = place(sc_at(row, at));
                auto a_co = place(co_at(row, at));
                if (!ties) {
                    each_block(0xff800000u, [&](const uint32_t (&v)[32], int j0, uint32_t) {
#pragma unroll
                        for (int c = 0; c < 32; ++c) store(a_sc, a_co, __uint_as_float(v[c]), j0 + c, reaches(__uint_as_float(v[c]), thr));
                    });
                } else {
                    each_block(0xff800000u, [&](const uint32_t (&v)[32], int j0, uint32_t) {
#pragma unroll
                        for (int c = 0; c < 32; ++c) store(a_sc, a_co, __uint_as_float(v[c]), j0 + c, reaches(__uint_as_float(v[c]), j0 + c, thr, before));
                    });
                }
                index_ok(a_sc == place(sc_at(row, end)), p.status, IX_ROUTE_SURVIVORS);
                len = total;
                tc_fence_before();
                __syncwarp();
                if (lane == 0)
                    for (int s = 0; s < n_st; ++s) mbar_arrive(bar(ACC_EMPTY + s));
                ok = same_rows();
            }
            if (!ok) break;
            // the ranges that the unit before reserved are all there
            ok = all_warps();
            if (!ok) break;
            if (last_t >= 0) write_entries(last_h, last_t, other);
            // a warp per row, two rows at a time: the survivors sorted, score descending, then column ascending
            constexpr int R = N <= 4 ? 2 : 1;
#pragma unroll 1
            for (int y = 0; y < 8; y += R) {
                const int r0 = quad * 32 + part + 4 * y, i0 = t * kLongRows + r0;
                if (i0 >= p.L) break;
                uint64_t key[R][N];
                int n_surv[R];
#pragma unroll
                for (int b = 0; b < R; ++b) {
                    n_surv[b] = __shfl_sync(ALL, len, part + 4 * (y + b));      // (0 past the end of the stream)
#pragma unroll
                    for (int e = 0; e < N; ++e) {
                        const int x = lane * N + e;
                        key[b][e] = 0;
                        if (x < n_surv[b]) key[b][e] = (uint64_t)sort_key(sc_at(r0 + 4 * b, x)) << 32 | (uint32_t)~(uint32_t)co_at(r0 + 4 * b, x);
                    }
                }
                warp_sort<R, N>(key, lane);
#pragma unroll
                for (int b = 0; b < R; ++b) {
                    const int i = i0 + 4 * b;
                    int32_t *out = p.sel + ((size_t)h * p.L + i) * p.k;
                    float *pl = p.part_lse + part_lse_at(h, (p.L + 127) >> 7, p.k, i, 0);     // slot x: pl[x * 128]
#pragma unroll
                    for (int e = 0; e < N; ++e) {
                        const int x = lane * N + e;
                        if (x >= p.k || i >= p.L) continue;
                        int j = -1;
                        const uint32_t col = ~(uint32_t)key[b][e];
                        if (x < n_surv[b] && index_ok(col < (uint32_t)p.ncol, p.status, IX_ROUTE_COLUMN) && col < (uint32_t)p.ncol) {
                            j = p.col_chunk[col];
                            atomicAdd(&hist[j], 1);
                        } else {
                            pl[x * 128] = -INFINITY;
                        }
                        out[x] = j;
                    }
                    if (i < p.L)
                        for (int x = CAP + lane; x < p.k; x += 32) {             // more picks asked for than there are columns
                            out[x] = -1;
                            pl[x * 128] = -INFINITY;
                        }
                }
            }
            // the unit's pick counts are complete: each thread reserves the ranges of its chunks, and clears the counters of the unit before
            ok = all_warps();
            if (!ok) break;
            for (int x0 = threadIdx.x; x0 < p.C; x0 += 4 * 32 * kLongSel) {
                int c[4];
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    const int x = x0 + y * 32 * kLongSel;
                    c[y] = x < p.C ? hist[x] : 0;
                    if (x < p.C && p.hists == 2) other[x] = 0;
                }
#pragma unroll
                for (int y = 0; y < 4; ++y)
                    if (c[y]) c[y] = p.cap_off[x0 + y * 32 * kLongSel] + atomicAdd(&p.cnt[h * p.C + x0 + y * 32 * kLongSel], c[y]);
#pragma unroll
                for (int y = 0; y < 4; ++y)
                    if (x0 + y * 32 * kLongSel < p.C) hist[x0 + y * 32 * kLongSel] = c[y];
            }
            if (p.hists == 2) {
                last_h = h;
                last_t = t;
                continue;
            }
            ok = all_warps();
            if (!ok) break;
            write_entries(h, t, hist);
            ok = all_warps();
            if (!ok) break;
            for (int x = threadIdx.x; x < p.C; x += 32 * kLongSel) hist[x] = 0;
        }
        if (ok && last_t >= 0 && all_warps()) write_entries(last_h, last_t, hist_base + ((n - 1) & 1) * p.C);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kLongSel) tmem_dealloc(tmem, 512);
    if (threadIdx.x == 0) report_abort(p.status, s_abort);
    finish_route(p.status, p.cnt, p.tile_off, p.H * p.C, p.cookie, kLongThreads);
}

// What an SM has, less the kernel's static variables.  The attribute is the same for every plan: another thread's call may come between it and the
// launch, and with the size of a plan of fewer chunks the launch would fail.
constexpr int kLongMost = 227 * 1024 - 11 * 1024;

template <int D, int N>
static int route_long_n(const RouteLongParams &a, const CUtensorMap &tmQ, const CUtensorMap &tmD, unsigned grid, size_t smem, cudaStream_t s) {
    MOC_CUDA_TRY(cudaFuncSetAttribute(route_long_kernel<D, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLongMost));
    route_long_kernel<D, N><<<grid, kLongThreads, smem, s>>>(tmQ, tmD, a);
    MOC_LAUNCH_CHECK();
    return MOC_OK;
}

template <int D>
static int route_long_d(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *desc3, int32_t *sel, void *ws, cudaStream_t s) {
    // The chunk counts that the header states: those whose tables, of three ints a chunk with more than 32 picks and four with fewer, fit
    // beside a block of descriptors and one or two Q tiles.
    {
        const int lists = p->k > 32 ? 1 : 2, ctas = std::max(1, std::min(p->n_sm / p->H, (p->L + kLongRows - 1) / kLongRows));
        const int rows = p->c_pad <= 192 ? p->c_pad : 128, tiles = p->c_pad <= 192 ? 1 : lists;
        const size_t tables = sizeof(int) * ((size_t)(lists + 1) * p->C + p->ncol + (p->L + kLongRows - 1) / kLongRows / ctas + 16);
        if ((((size_t)3 * rows * D * 2 + 1023) & ~(size_t)1023) + tiles * (size_t)kLongRows * D * 2 + tables > 227 * 1024 - 1024 - 512) return MOC_ERR_SHAPE;
    }
    RouteLongParams a;
    a.scratch = ws_ptr<float>(ws, p->ws.part_o);
    a.sel = sel; a.part_lse = ws_ptr<float>(ws, p->ws.part_lse); a.cnt = ws_ptr<int>(ws, p->ws.cnt);
    a.qlist = ws_ptr<int32_t>(ws, p->ws.qlist);
    a.tok_chunk = p->d_tok_chunk; a.cand_c = p->d_cand_c; a.lim = p->d_lim; a.reach = p->d_reach;
    a.col_chunk = p->d_col_chunk; a.cap_off = p->d_cap_off; a.status = ws_ptr<int>(ws, p->ws.status);
    a.H = p->H; a.L = p->L; a.C = p->C; a.c_pad = p->c_pad; a.ncol = p->ncol; a.k = p->k; a.cwords = p->cwords; a.prefix = p->prefix_mode;
    a.n_units = p->H * ((p->L + kLongRows - 1) / kLongRows);
    a.d_rows = std::min(p->c_pad, kLongStep);
    a.tile_off = ws_ptr<int>(ws, p->ws.tile_off);
    a.cookie = p->cookie;
    a.wait = WaitBound::of(p->wait_us);
    a.cap_total = (size_t)p->cap_off[p->C];
    // Survivors that are sorted: more than k, so that the first threshold is often good enough (30 of 504: any of 30 to 64), at most 512;
    // or all the columns there are.  With more columns than an accumulator holds each 512 of them have thresholds of their own, and a
    // wider choice gains more than it costs in the sort (1008 columns, 24 picks, 32 or 64 survivors: 900, 790 us).
    const bool one = p->c_pad <= kLongStep * kLongAcc;
    const int want = std::min(p->k <= (one ? 28 : 20) ? 32 : p->k <= (one ? 60 : 52) ? 64 : p->k <= 120 ? 128 : p->k <= 240 ? 256 : 512, p->c_pad);
    const int n = want <= 32 ? 1 : want <= 64 ? 2 : want <= 128 ? 4 : want <= 256 ? 8 : 16;
    const size_t budget = kLongMost - 1024;     // less the slack that aligns the tiles
    const size_t q_tile = (size_t)kLongRows * D * 2, slot = ((size_t)a.d_rows * D * 2 + 1023) & ~(size_t)1023;
    const size_t row_queue = (32 * n + 1) * 4 + (32 * n + 2) * 2, queue = n <= kQueueShared ? kLongRows * row_queue : 0, hist = sizeof(int) * (size_t)p->C;
    a.hists = q_tile + slot + queue + 2 * hist <= budget ? 2 : 1;
    const size_t other = queue + a.hists * hist;
    if (q_tile + slot + other > budget) return MOC_ERR_SHAPE;
    a.q_stages = 2 * q_tile + 3 * slot + other <= budget ? 2 : 1;
    a.d_slots = (int)std::min<size_t>(kLongSlots, (budget - other - a.q_stages * q_tile) / slot);
    const size_t smem = 1024 + a.d_slots * slot + a.q_stages * q_tile + other;
    // One CTA per SM, as far as there are units and room for their rows' survivors (1.5 KB to 3 KB a row with more than 120 picks, whose partials will
    // take 15 KB or more).
    unsigned grid = (unsigned)std::min(p->n_sm, a.n_units);
    if (n > kQueueShared) grid = (unsigned)std::min<size_t>(grid, (p->ws.part_lse - p->ws.part_o) / (kLongRows * row_queue));
    if (grid < 1) return MOC_ERR_SHAPE;
    CUtensorMap tmQ, tmD;
    if (int r = make_tmap_2d_bf16(&tmQ, Q, (uint64_t)p->H * p->L, D, kLongRows)) return r;
    if (int r = make_tmap_2d_bf16(&tmD, desc3, (uint64_t)p->H * 3 * p->c_pad, D, (uint32_t)a.d_rows)) return r;
    switch (n) {
        case 1: return route_long_n<D, 1>(a, tmQ, tmD, grid, smem, s);
        case 2: return route_long_n<D, 2>(a, tmQ, tmD, grid, smem, s);
        case 4: return route_long_n<D, 4>(a, tmQ, tmD, grid, smem, s);
        case 8: return route_long_n<D, 8>(a, tmQ, tmD, grid, smem, s);
        default: return route_long_n<D, 16>(a, tmQ, tmD, grid, smem, s);
    }
}

int launch_route_long(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *desc3, int32_t *sel, void *ws, cudaStream_t s) {
    return p->d == 128 ? route_long_d<128>(p, Q, desc3, sel, ws, s) : route_long_d<64>(p, Q, desc3, sel, ws, s);
}

}  // namespace moc
