// Shared declarations of the MoC library: plan object, workspace layout, launch helpers.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <atomic>
#include <vector>

#include "../../include/moc.h"
#include <nvtx3/nvToolsExt.h>

namespace moc {

constexpr int kQTileRows = 256;     // query rows per attention work item (two 128-row MMA tiles)
constexpr int kPoolSlice = 256;     // tokens per chunk-pool work unit
constexpr int kStatusWords = 16;    // status area at the head of the workspace (int32 each):
// [0] device status (a moc_status), [1] detail code, [2] cookie of the plan whose lists the workspace holds,
// [4] routing blocks that have finished
enum StatusWord { ST_STATUS = 0, ST_DETAIL = 1, ST_COOKIE = 2, ST_ARRIVE = 4 };
constexpr int kQueueHeader = 4;     // queue area: [0] next item to claim, [1] items, [2] phases, [3] CTAs that have left; then 3 ints per phase
constexpr unsigned kPrivFlagCudaCoreAttend = 0x80000000u;   // plan flag outside the public header: test hook

// How often a kernel's waits look before they give up: one to two seconds' worth, or one to two times `us` microseconds' (tests; never more than the
// default).  Measured with waits that nothing ends (moc_debug_wait_probe_form): a look takes 32.8 us where the thread parks, 86 ns
// where it polls (46 in a loop of nothing else), 257 to 512 ns where it looks at a counter in global memory; the default is 2.05, 1.4 and 1 to 2 s.
struct WaitBound {
    uint32_t parked, polled, looks;
    static WaitBound of(unsigned us) {
        if (us == 0 || us > 1000000u) us = 1000000u;
        return WaitBound{us / 16 + 1, us * 16u, us * 4u};
    }
};

// One contiguous range of key tokens [t0, t1).
struct KeyRange { int32_t t0, t1; };

// One attention work item: up to kQTileRows query rows of head h against the key ranges
// rng[rng_off .. rng_off + nrng) (ntiles key tiles of 128; [t0, t1) repeats the first range).  Anchor pass: `first` is the first of `rows`
// consecutive query rows of one chunk (h is implied by the item index).  Routed pass: `first` is the
// offset, inside the head's list area, of the `rows` entries of one chunk's query list.
struct WorkItem { int32_t h, first, rows, ntiles, rng_off, nrng, t0, t1; };

// One tile of up to 128 consecutive key tokens of a chunk (backward, key-stationary pass), with what its block looks up first:
// the rows that have the chunk as an anchor (n_rng ranges from rng on, n_anc tiles of 128 rows), where its query list starts, and
// how many blocks share its query tiles (no more than n_anc: each has one).
struct __align__(32) KTile { int32_t chunk, t0, valid, n_anc, rng, n_rng, list, parts; };

struct WsLayout {
    size_t status;      // int32[kStatusWords], see StatusWord
    size_t cnt;         // int32[H][C]     routed picks per (head, chunk); doubles as the list cursor while routing
    size_t tile_off;    // int32[H*C+1]    running count of routed attention tiles over (head, chunk) pairs
    size_t rtiles;      // WorkItem[H * (ceil(L k / 256) + C)]  routed work items, written after routing
    size_t qlist;       // int32[H][cap_total]  per (head, chunk) list at cap_off[c]: entries i*k+s of the picks of c
    size_t desc3;       // bf16 [H][3][Cpad][d]  descriptors split into three bf16 terms (hi + mid + lo)
    size_t pool_part;   // float[H][n_pool_units][d] partial key sums
    size_t pool_done;   // int32 arrival counters: of pooling, [H][C] (cleared at the start of every call), or in the backward, [H][n_long_ktiles], of
                        // the key tiles that several blocks share
    size_t queue;       // int32[kQueueHeader + 6 groups] work queue of the forward attention kernel
    size_t part_o;      // bf16 [1 or 2][Hg][L][k][d] routed partial outputs (normalised) of one group of Hg heads; with
                        // several groups, two buffers that consecutive groups alternate between
    size_t part_lse;    // float[H][ceil(L / 128)][k][128]  routed partial log-sum-exp (-inf = unused slot), see part_lse_at
    size_t fwd_end;
    size_t delta;       // float[H][L]       rowsum(dO * O)
    size_t bwd_end;
};

}  // namespace moc

struct moc_plan {
    int H, L, d, C, k, win_back, win_fwd;
    unsigned flags;
    float scale;
    int device;
    int n_sm;
    bool pool_direct = false;    // descriptors by one block per (head, chunk): every block resident at once, no long chunk
    std::vector<int32_t> off, shot;
    std::vector<uint8_t> mod;
    // host-side derived tables
    std::vector<int32_t> anc_off;            // [C+1] into anc_rng
    std::vector<moc::KeyRange> anc_rng;      // merged anchor token ranges per query chunk
    std::vector<int64_t> anc_tokens;         // [C] anchor key tokens per query chunk
    std::vector<int32_t> ranc_off, ranc;     // reverse anchors: key chunk -> query chunks
    std::vector<moc::WorkItem> qitems;       // anchor-pass work items of one head
    std::vector<moc::KeyRange> qry_rng;      // merged ranges of the query rows that have a chunk as an anchor, chunk by chunk
    std::vector<moc::KTile> ktiles;          // key tiles of one head: the long ones (see derive_plan) first, then chunk by chunk
    int n_long_ktiles = 0;
    int n_split = 1;                         // the largest number of blocks that share the query rows of a long key tile (see derive_plan)
    std::vector<int32_t> pool_unit_off;      // [C+1] prefix of pool units per chunk
    std::vector<moc::KeyRange> shot_chunks;  // [S] chunk range [t0, t1) of every shot (outer-loop routing)
    int words;                               // uint32 words per anchor bitmap row
    std::vector<int32_t> cap_off;            // [C+1] start of chunk c's query list inside a head's list area
    // Routing scores only the chunks that can ever be picked: text chunks are anchors of every query, so the score
    // matrix has one column per non-text chunk ("column" = index among those, in chunk order).
    int ncol;                                // number of columns
    int64_t routed_key_tiles;                // key tiles of all of them
    int cwords;                              // uint32 words per candidate bitmap row (over columns)
    int prefix_mode;                         // 1: every query chunk's candidates are exactly the columns [0, lim[c])
    int c_pad;                               // columns rounded up to a multiple of 16 (MMA N granularity)
    int n_pool_units;
    int heads_per_group;                     // Hg: heads whose routed partials are held at once (attention runs group by group)
    size_t partials_budget;                  // bytes the routed partials may take; sets Hg
    uint32_t cookie;                         // hash of the problem and the heads per group, written into a workspace this plan has routed on
    uint32_t wait_us;                        // limit of the kernels' bounded waits (0 = default); tests shorten it
    // device tables (one allocation)
    void *d_blob;
    int32_t *d_off, *d_shot, *d_tok_chunk, *d_anc_off, *d_ranc_off, *d_ranc, *d_pool_unit_off, *d_pool_unit_chunk, *d_cap_off;
    uint8_t *d_mod;
    uint32_t *d_anc_bits;
    uint32_t *d_cand_c;                      // [C][cwords] candidate columns of a query in chunk c (causality included)
    int32_t *d_lim, *d_reach, *d_col_chunk;  // [C] prefix length (-1: not a prefix); [C] columns any query up to chunk c can reach; [ncol] chunk of a column
    moc::KeyRange *d_anc_rng;
    moc::WorkItem *d_qitems;
    moc::KeyRange *d_chunk_rng;              // [C] token range of every chunk
    moc::KTile *d_ktiles;
    moc::KeyRange *d_qry_rng;
    moc::KeyRange *d_shot_chunks;            // [S]
    moc::WsLayout ws;
};

namespace moc {

extern std::atomic<long long> g_launches;
void set_cuda_error(cudaError_t e, const char *where);

#define MOC_CUDA_TRY(expr)                                         \
    do {                                                           \
        cudaError_t e_ = (expr);                                   \
        if (e_ != cudaSuccess) {                                   \
            moc::set_cuda_error(e_, #expr);                        \
            return MOC_ERR_CUDA;                                   \
        }                                                          \
    } while (0)

#define MOC_LAUNCH_CHECK()                                         \
    do {                                                           \
        moc::g_launches.fetch_add(1);                              \
        cudaError_t e_ = cudaGetLastError();                       \
        if (e_ != cudaSuccess) {                                   \
            moc::set_cuda_error(e_, "kernel launch");              \
            return MOC_ERR_CUDA;                                   \
        }                                                          \
    } while (0)

// A kernel that may start while the kernel before it in the stream still runs: once every block of that one has called
// next_may_start() or has left.  It calls previous_done() where it needs the other's results; and a kernel has to see to it
// that it does not finish before the previous one, for the sake of what follows in the stream.
__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void previous_done() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... P, typename... A>
static inline cudaError_t launch_early(bool early, void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A &&...args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = early;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid); c.blockDim = dim3(block); c.dynamicSmemBytes = smem; c.stream = s;
    c.attrs = &at; c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);
}

template <typename T>
static inline T *ws_ptr(void *ws, size_t off) { return reinterpret_cast<T *>(static_cast<char *>(ws) + off); }
template <typename T>
static inline const T *ws_ptr(const void *ws, size_t off) { return reinterpret_cast<const T *>(static_cast<const char *>(ws) + off); }

// Division of a list entry (query * k + slot) by k without the division sequence, whose reciprocal queues behind the
// exponentials of the same scheduler.  Exact for 0 <= e < 2^31: mul = ceil(2^(31 + s) / k) with 2^s >= k, so that
// 0 <= mul * k - 2^(31 + s) < k <= 2^s.
struct SlotDiv {
    uint32_t mul;
    int shift;
    static SlotDiv of(int k) {
        int s = 0;
        while ((1 << s) < k) ++s;
        const uint64_t two = 1ull << (31 + s), kk = k > 0 ? k : 1;
        return SlotDiv{(uint32_t)((two + kk - 1) / kk), 31 + s};
    }
#ifdef __CUDACC__
    __device__ __forceinline__ int query(int e) const { return e < 0 ? -1 : (int)(((uint64_t)(uint32_t)e * mul) >> shift); }
#endif
};

#ifdef __CUDACC__
// Debug build (-DMOC_DEBUG): every index a kernel takes from the workspace (list entries, list positions,
// work-item fields) is checked before it is used as an address; a bad one records MOC_ERR_INDEX with `code`
// in the status area and the access is skipped.  In the release build the checks cost nothing.
enum IndexCheck { IX_ITEM_FIELDS = 200, IX_LIST_POSITION, IX_LIST_ENTRY, IX_APPEND_POSITION, IX_BWD_ITEM_FIELDS,
                  IX_BWD_LIST_POSITION, IX_BWD_LIST_ENTRY, IX_ROUTE_SURVIVORS, IX_ROUTE_COLUMN };
#ifdef MOC_DEBUG
__device__ __forceinline__ bool index_ok(bool cond, int *status, int code) {
    if (!cond && atomicCAS(status, 0, MOC_ERR_INDEX) == 0) status[ST_DETAIL] = code;
    return cond;
}
#else
__device__ __forceinline__ bool index_ok(bool, int *, int) { return true; }
#endif

// Layout of the routed partials (the forward's outputs, and dQ in the backward): a row is d / 64 lines of 128 bytes, query-innermost
// within a block of 128 queries, so that a slot's lines of consecutive queries, which a warp of an anchor item fetches together,
// are contiguous.  Byte offset of the first line of (head-in-group hl, query qi, slot s); the next one is 16 KB (128 queries)
// further.  Within a line, the 16-byte piece 2 i + z (i = 0..3, z = 0, 1) holds the columns 32 z + 8 x + 2 i and the one after
// (x = 0..3), the order in which the tensor memory hands them out.  Where the forward's merge reads lines from shared memory, a row
// per lane, piece c sits at place c ^ (qi mod 8), so that lanes reading a piece of eight rows meet no bank twice; elsewhere at c.
__device__ __forceinline__ size_t part_line(int hl, int LB, int k, int lines, int qi, int s) {
    return ((((size_t)hl * LB + (qi >> 7)) * k + s) * lines << 14) + ((qi & 127) << 7);
}

// Index of the log-sum-exp of (head, query, slot): query-innermost like the partials, so that the lanes of an anchor
// item, which hold consecutive queries, read 128 contiguous bytes per slot.
__device__ __forceinline__ size_t part_lse_at(int h, int LB, int k, int qi, int s) {
    return (((size_t)h * LB + (qi >> 7)) * k + s) * 128 + (qi & 127);
}

// A named range around a call of the boundary, for timeline tools (NVTX; a no-op when no tool is attached).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// Walks the 128-key tiles of a list of key ranges (a tile never straddles two ranges).
struct TileIter {
    const KeyRange *rng;
    int n, ri, t, end;      // the current range's end is kept: one load per range, not per tile
    __device__ TileIter(const KeyRange *r, int n_) : rng(r), n(n_), ri(0), t(n_ > 0 ? r[0].t0 : 0), end(n_ > 0 ? r[0].t1 : 0) {}
    // the first range given by value
    __device__ TileIter(const KeyRange *r, int n_, int t0, int t1) : rng(r), n(n_), ri(0), t(t0), end(t1) {}
    __device__ bool next(int &t0, int &valid) {
        if (ri >= n) return false;
        t0 = t;
        valid = min(128, end - t);
        t += 128;
        if (t >= end) {
            ++ri;
            if (ri < n) { t = rng[ri].t0; end = rng[ri].t1; }
        }
        return true;
    }
};
#endif

void layout_workspace(moc_plan *p);

static inline bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// kernels' host launchers (each returns a moc_status)
int launch_chunk_pool(const moc_plan *p, const __nv_bfloat16 *K, float *desc, void *ws, cudaStream_t s);
int launch_route(const moc_plan *p, const __nv_bfloat16 *Q, const float *desc, int32_t *sel, void *ws, cudaStream_t s);
int launch_lists_from_sel(const moc_plan *p, int32_t *sel, void *ws, cudaStream_t s);
int launch_context_drop(const moc_plan *p, int32_t *sel, float p_max, float lambda, uint64_t seed, cudaStream_t s);
int pool_scratch_prepare(int device);     // looks up (once per device) the fixed scratch array of moc_chunk_pool_noalloc
int launch_attend_scalar(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *K, const __nv_bfloat16 *V,
                         const int32_t *sel, __nv_bfloat16 *O, float *lse, void *ws, cudaStream_t s);
int launch_attend_bwd_scalar(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *K, const __nv_bfloat16 *V,
                             const __nv_bfloat16 *O, const float *lse, const __nv_bfloat16 *dO, const int32_t *sel,
                             __nv_bfloat16 *dQ, __nv_bfloat16 *dK, __nv_bfloat16 *dV, void *ws, cudaStream_t s);
int launch_attend_bwd_tc(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *K, const __nv_bfloat16 *V,
                         const __nv_bfloat16 *O, const float *lse, const __nv_bfloat16 *dO, const int32_t *sel,
                         __nv_bfloat16 *dQ, __nv_bfloat16 *dK, __nv_bfloat16 *dV, void *ws, cudaStream_t s);
// Whether the launches of the backward start while the one before still runs: up to 16 dK/dV blocks per SM.  Training steps,
// in turn (one after another -> overlapping): 0.7 blocks per SM 158 -> 134 us, 4 447 -> 428 us; at 20, 45 and 111 the two are alike
// (6.64 / 6.64, 14.16 / 14.16 and 102.9 / 102.3 ms, where the runs of one side differ by 0.7 %).
inline bool backward_overlaps(const moc_plan *p) { return p->ktiles.size() * (size_t)p->H <= 16 * (size_t)p->n_sm; }
// Blocks per long key tile that dK/dV is launched with (a tile's own number may be smaller): the plan's, if the shared tiles' sums fit
// into the space of the routed partials, else one.
inline int dkv_split(const moc_plan *p) {
    const size_t sums = 2 * sizeof(float) * 128 * (size_t)p->d * p->n_long_ktiles * p->H;
    return p->n_split > 1 && sums * p->n_split <= p->ws.part_lse - p->ws.part_o ? p->n_split : 1;
}
int launch_dq_tc(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *K, const __nv_bfloat16 *V, const float *lse,
                 const float *delta, const __nv_bfloat16 *dO, __nv_bfloat16 *dQ, void *ws, cudaStream_t s);
// (also clears n_zero counters)
int launch_delta(const moc_plan *p, const __nv_bfloat16 *O, const __nv_bfloat16 *dO, float *delta, int *zero, int n_zero, cudaStream_t s);
int launch_attend_tc(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *K, const __nv_bfloat16 *V,
                     const int32_t *sel, __nv_bfloat16 *O, float *lse, void *ws, cudaStream_t s);

}  // namespace moc

// Test hooks: exported, but not part of the public header (tests declare them themselves).
extern "C" {
// attention and its backward on the plain fp32 CUDA-core kernels (an in-library cross-check that reads
// the selection straight from sel_idx)
int moc_debug_use_cuda_core_attention(moc_plan *plan, int on);
// limit of every bounded device-side wait, in microseconds, of the launches from now on (0 = default)
int moc_debug_set_wait_limit_us(moc_plan *plan, unsigned us);
// one block whose only wait is on a barrier that nothing ever arrives on: it must give up after the limit,
// record MOC_ERR_TIMEOUT with detail `code` in ws, and return.  `form`: 0 the wait parks, 1 it polls, 2 it looks at a counter in global memory
int moc_debug_wait_probe_form(const moc_plan *plan, void *ws, int form, int code, void *stream);
int moc_debug_wait_probe(const moc_plan *plan, void *ws, int code, void *stream);      // form 0
// host only: the long key tiles of dK/dV of a problem on a GPU with n_sm SMs (up to cap of them written): tiles of query rows that
// a tile has whatever is picked, and blocks that share them; and the bytes there are for the counters of all heads' tiles
int moc_debug_shared_key_tiles(const moc_problem *problem, int n_sm, int cap, int *n_tiles, int *query_tiles, int *blocks, size_t *counter_room);
}
