// Plan object (validated problem + derived chunk tables on the device), workspace layout,
// argument checking and the C entry points.
#include <cuda.h>
#include <math.h>
#include <algorithm>
#include <string.h>
#include <mutex>
#include <new>
#include <string>

#include "moc_common.cuh"

namespace moc {

std::atomic<long long> g_launches{0};
static std::mutex g_err_mu;
static std::string g_err = "";

void set_cuda_error(cudaError_t e, const char *where) {
    std::lock_guard<std::mutex> g(g_err_mu);
    g_err = std::string(cudaGetErrorName(e)) + ": " + cudaGetErrorString(e) + " (" + where + ")";
    (void)cudaGetLastError();
}

constexpr int kMaxSplit = 8;

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// FNV-1a over the problem and the heads per group: a workspace routed by one plan is not accepted by a plan of another problem,
// nor under another budget (routing lays the attention's work queue out by groups of heads)
static uint32_t plan_cookie(const moc_plan *p) {
    uint32_t hsh = 2166136261u;
    auto mix = [&](const void *data, size_t n) {
        const unsigned char *b = static_cast<const unsigned char *>(data);
        for (size_t i = 0; i < n; ++i) { hsh ^= b[i]; hsh *= 16777619u; }
    };
    const int32_t hdr[] = {p->H, p->L, p->d, p->C, p->k, p->win_back, p->win_fwd, (int32_t)(p->flags & MOC_FLAG_CAUSAL), p->heads_per_group};
    mix(hdr, sizeof hdr);
    mix(p->off.data(), p->off.size() * 4);
    mix(p->shot.data(), p->shot.size() * 4);
    mix(p->mod.data(), p->mod.size());
    return hsh ? hsh : 1u;
}

// tok_chunk[t] = the chunk of token t, a block per chunk.  (Made on the host and copied, with the caller's stream waited for, a plan
// of a 132k-token stream held the caller up for 214 us; now 140.)
__global__ void token_chunk_kernel(const int32_t *__restrict__ off, int32_t *__restrict__ tok_chunk) {
    for (int t = off[blockIdx.x] + threadIdx.x; t < off[blockIdx.x + 1]; t += blockDim.x) tok_chunk[t] = blockIdx.x;
}

// The stream on which plans get their tables, one per context for as long as the process lives (making one takes 100 us).  A stream
// belongs to the context it was made in, and a device can have several, or a new one after cudaDeviceReset.
static cudaError_t table_stream(cudaStream_t *out) {
    typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long *);
    struct Entry { unsigned long long ctx; cudaStream_t stream; };
    static std::mutex mu;
    static std::vector<Entry> streams;
    static CtxGetIdFn ctx_id = nullptr;
    std::lock_guard<std::mutex> hold(mu);
    if (!ctx_id) {
        void *sym = nullptr;
        cudaDriverEntryPointQueryResult q;
        const cudaError_t e = cudaGetDriverEntryPoint("cuCtxGetId", &sym, cudaEnableDefault, &q);
        if (e != cudaSuccess) return e;
        if (!sym || q != cudaDriverEntryPointSuccess) return cudaErrorSymbolNotFound;
        ctx_id = (CtxGetIdFn)sym;
    }
    unsigned long long id = 0;                                   // of the current context; never used twice
    if (ctx_id(nullptr, &id) != CUDA_SUCCESS) return cudaErrorInvalidResourceHandle;
    for (const Entry &x : streams)
        if (x.ctx == id) { *out = x.stream; return cudaSuccess; }
    const cudaError_t e = cudaStreamCreateWithFlags(out, cudaStreamNonBlocking);
    if (e == cudaSuccess) streams.push_back(Entry{id, *out});
    return e;
}

// Workspace layout.  The routed partial outputs ([heads][L][k][d] bf16, k times the size of O) are held for
// one group of Hg heads at a time; attention and its backward run group by group.  If all heads fit the plan's
// budget there is one group and one buffer; otherwise two buffers of Hg heads each (consecutive groups
// alternate, so that one group's routed items can run while the previous group's anchor items still merge),
// Hg the largest even split of the heads for which both stay within the budget (at least one head).
void layout_workspace(moc_plan *p) {
    WsLayout &w = p->ws;
    const size_t H = p->H, L = p->L, d = p->d, C = p->C, k = p->k;
    const size_t per_head = sizeof(__nv_bfloat16) * ((L + 127) / 128 * 128) * k * d;      // whole blocks of 128 queries
    size_t groups = 1, buffers = 1;
    p->heads_per_group = (int)H;
    if (per_head * H > p->partials_budget) {
        const size_t hg = std::max<size_t>(1, p->partials_budget / (2 * per_head));
        groups = (H + hg - 1) / hg;
        p->heads_per_group = (int)((H + groups - 1) / groups);
        groups = (H + p->heads_per_group - 1) / p->heads_per_group;
        buffers = groups > 1 ? 2 : 1;
    }
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, 256); return at; };
    w.status = take(sizeof(int32_t) * kStatusWords);
    w.cnt = take(sizeof(int32_t) * H * C);
    w.tile_off = take(sizeof(int32_t) * (H * C + 1));
    w.rtiles = take(sizeof(WorkItem) * H * ((L * (k ? k : 1) + kQTileRows - 1) / kQTileRows + C));
    w.qlist = take(sizeof(int32_t) * H * (size_t)std::max(p->cap_off[C], 1));
    w.desc3 = take(sizeof(__nv_bfloat16) * H * 3 * (size_t)p->c_pad * d);
    w.pool_part = take(sizeof(float) * H * (size_t)p->n_pool_units * d);
    w.pool_done = take(sizeof(int32_t) * H * std::max<size_t>(C, p->n_split > 1 ? p->n_long_ktiles : 0));
    w.queue = take(sizeof(int32_t) * (kQueueHeader + 6 * groups));
    w.part_o = take(per_head * (size_t)p->heads_per_group * buffers);
    w.part_lse = take(sizeof(float) * H * ((L + 127) / 128 * 128) * (k ? k : 1));
    w.fwd_end = o;
    w.delta = take(sizeof(float) * H * L);
    w.bwd_end = o;
    p->cookie = plan_cookie(p);
}

// What the derivation leaves for the device alone.
struct DeviceTables {
    std::vector<uint32_t> bits, cand_c;
    std::vector<int32_t> unit_chunk, lim, reach, col_chunk;
    std::vector<KeyRange> chunk_rng;
};

static int check_problem(const moc_problem *pr) {
    if (!pr->chunk_off || !pr->chunk_shot || !pr->chunk_mod) return MOC_ERR_NULL;
    if (pr->n_heads < 1 || pr->n_tokens < 1 || pr->n_chunks < 1 || pr->n_chunks > pr->n_tokens) return MOC_ERR_SHAPE;
    // heads index grid.y; head * L + token is a 32-bit row coordinate of the tensor maps
    if (pr->n_heads > 65535 || (double)pr->n_heads * pr->n_tokens >= 2147483647.0) return MOC_ERR_SHAPE;
    if (pr->head_dim != 64 && pr->head_dim != 128) return MOC_ERR_SHAPE;
    if (pr->top_k < 0 || pr->top_k > 512) return MOC_ERR_SHAPE;
    if (pr->win_back < MOC_WHOLE_SHOT || pr->win_fwd < MOC_WHOLE_SHOT) return MOC_ERR_SHAPE;
    if ((double)pr->n_tokens * (pr->top_k ? pr->top_k : 1) >= 2147483647.0) return MOC_ERR_SHAPE;
    if ((double)pr->n_heads * pr->n_chunks >= 1e8) return MOC_ERR_SHAPE;
    if (pr->flags & ~MOC_FLAG_CAUSAL) return MOC_ERR_SHAPE;
    if (!(pr->softmax_scale >= 0.f) || isinf(pr->softmax_scale)) return MOC_ERR_SHAPE;
    const int C = pr->n_chunks, L = pr->n_tokens;
    if (pr->chunk_off[0] != 0 || pr->chunk_off[C] != L) return MOC_ERR_CHUNK_TABLE;
    for (int c = 0; c < C; ++c) {
        if (pr->chunk_off[c + 1] <= pr->chunk_off[c]) return MOC_ERR_CHUNK_TABLE;
        if (pr->chunk_mod[c] > 1) return MOC_ERR_CHUNK_TABLE;
        if (c > 0 && pr->chunk_shot[c] < pr->chunk_shot[c - 1]) return MOC_ERR_CHUNK_TABLE;
    }
    return MOC_OK;
}

// Everything of a plan that a checked problem and the number of SMs determine; no device work.
static int derive_plan(moc_plan *p, const moc_problem *pr, int n_sm, DeviceTables &tab) {
    const int C = pr->n_chunks, L = pr->n_tokens;
    p->H = pr->n_heads; p->L = L; p->d = pr->head_dim; p->C = C; p->k = pr->top_k;
    p->win_back = pr->win_back; p->win_fwd = pr->win_fwd; p->flags = pr->flags;
    p->scale = pr->softmax_scale > 0.f ? pr->softmax_scale : 1.0f / sqrtf((float)pr->head_dim);
    p->n_sm = n_sm;
    p->off.assign(pr->chunk_off, pr->chunk_off + C + 1);
    p->shot.assign(pr->chunk_shot, pr->chunk_shot + C);
    p->mod.assign(pr->chunk_mod, pr->chunk_mod + C);

    // Sec. 3.2: text chunks are anchors of every query; so are the chunks of the query's shot
    // inside the window around its own chunk.  (Asked C * C times, twice: on values that no store can change.)
    const auto is_anchor = [mod = p->mod.data(), shot = p->shot.data(), back = p->win_back, fwd = p->win_fwd](int c, int j) {
        if (mod[j] == 1) return true;
        if (shot[j] != shot[c]) return false;
        if (j < c && back != MOC_WHOLE_SHOT && c - j > back) return false;
        if (j > c && fwd != MOC_WHOLE_SHOT && j - c > fwd) return false;
        return true;
    };
    // anchor bitmaps, merged anchor key ranges, reverse anchors
    p->words = (C + 31) / 32;
    tab.bits.assign((size_t)C * p->words, 0u);
    uint32_t *bits = tab.bits.data();
    std::vector<std::vector<int32_t>> rev(C);
    p->anc_off.assign(C + 1, 0);
    p->anc_tokens.assign(C, 0);
    for (int c = 0; c < C; ++c) {
        uint32_t *row = bits + (size_t)c * p->words;
        for (int j = 0; j < C; ++j) {
            if (!is_anchor(c, j)) continue;
            row[j / 32] |= 1u << (j % 32);
            rev[j].push_back(c);
            p->anc_tokens[c] += p->off[j + 1] - p->off[j];
            if ((int)p->anc_rng.size() > p->anc_off[c] && p->anc_rng.back().t1 == p->off[j])
                p->anc_rng.back().t1 = p->off[j + 1];
            else
                p->anc_rng.push_back(KeyRange{p->off[j], p->off[j + 1]});
        }
        p->anc_off[c + 1] = (int32_t)p->anc_rng.size();
    }
    p->ranc_off.assign(C + 1, 0);
    for (int j = 0; j < C; ++j) {
        p->ranc.insert(p->ranc.end(), rev[j].begin(), rev[j].end());
        p->ranc_off[j + 1] = (int32_t)p->ranc.size();
    }
    // query tiles (never straddle a chunk) and pool work units
    std::vector<int32_t> &unit_chunk = tab.unit_chunk;
    for (int c = 0; c < C; ++c) tab.chunk_rng.push_back(KeyRange{p->off[c], p->off[c + 1]});
    p->pool_unit_off.assign(C + 1, 0);
    for (int c = 0; c < C; ++c) {
        int anc_tiles = 0;
        for (int a = p->anc_off[c]; a < p->anc_off[c + 1]; ++a) anc_tiles += (p->anc_rng[a].t1 - p->anc_rng[a].t0 + 127) / 128;
        for (int r = p->off[c]; r < p->off[c + 1]; r += kQTileRows)
            p->qitems.push_back(WorkItem{0, r, std::min(kQTileRows, p->off[c + 1] - r), anc_tiles, p->anc_off[c],
                                         p->anc_off[c + 1] - p->anc_off[c], p->anc_rng[p->anc_off[c]].t0,
                                         p->anc_rng[p->anc_off[c]].t1});
        int units = (p->off[c + 1] - p->off[c] + kPoolSlice - 1) / kPoolSlice;
        p->pool_unit_off[c + 1] = p->pool_unit_off[c] + units;
        for (int u = 0; u < units; ++u) unit_chunk.push_back(c);
    }
    p->n_pool_units = p->pool_unit_off[C];
    {
        int longest = 0;
        for (int c = 0; c < C; ++c) longest = std::max(longest, p->off[c + 1] - p->off[c]);
        p->pool_direct = (int64_t)p->H * C <= 8LL * p->n_sm && C <= 65535 && longest <= 4096;
    }
    // Key tiles of the backward's key-stationary pass.  A tile's block streams every query that attends its chunk:
    // the rows of the chunks that have it as an anchor (known here) and the routed list.  Tiles of chunks whose
    // anchor rows are far above the average (a caption, which every query attends) go first, for all heads, so
    // that the longest blocks start at once instead of forming the tail of the launch.
    {
        std::vector<int64_t> anc_rows(C, 0);
        int64_t total = 0, tiles = 0;
        for (int c = 0; c < C; ++c) {
            for (int a = p->ranc_off[c]; a < p->ranc_off[c + 1]; ++a) anc_rows[c] += p->off[p->ranc[a] + 1] - p->off[p->ranc[a]];
            const int nt = (p->off[c + 1] - p->off[c] + 127) / 128;
            total += anc_rows[c] * nt;
            tiles += nt;
        }
        const int64_t mean_rows = total / std::max<int64_t>(tiles, 1);
        // the rows, as ranges: consecutive chunks are one
        std::vector<int32_t> rng_off(C + 1, 0), rng_tiles(C, 0);
        for (int c = 0; c < C; ++c) {
            for (int a = p->ranc_off[c]; a < p->ranc_off[c + 1];) {
                int qc = p->ranc[a];
                KeyRange r{p->off[qc], p->off[qc + 1]};
                for (++a; a < p->ranc_off[c + 1] && p->ranc[a] == qc + 1; ++a) r.t1 = p->off[++qc + 1];
                p->qry_rng.push_back(r);
                rng_tiles[c] += (r.t1 - r.t0 + 127) / 128;
            }
            rng_off[c + 1] = (int32_t)p->qry_rng.size();
        }
        for (int pass = 0; pass < 2; ++pass) {
            for (int c = 0; c < C; ++c) {
                const bool is_long = anc_rows[c] > 4 * mean_rows;
                if (is_long != (pass == 0)) continue;
                for (int t = p->off[c]; t < p->off[c + 1]; t += 128)
                    p->ktiles.push_back(KTile{c, t, std::min(128, p->off[c + 1] - t), rng_tiles[c], rng_off[c], rng_off[c + 1] - rng_off[c], 0, 1});
            }
            if (pass == 0) p->n_long_ktiles = (int)p->ktiles.size();
        }
        // A long tile is one block's serial work.  Where that is more than an SM's share of the whole launch (short streams: a
        // caption's block alone then takes as long as all else), its query rows are dealt to several blocks, each with about
        // that share, or what the other blocks have if that is more.  From twice the share on.  Tile by tile: next to a caption that
        // every row attends, a chunk that is much longer than its neighbours may have fewer query tiles than the caption has blocks,
        // and a block must have one.  (Whole backward passes, one block -> several: 2 heads of 4.6k tokens 108 -> 91 us, 3 heads of 3.3k
        // tokens at d = 64 79 -> 68, three small scenes 73.5 -> 71.3; below the line 1 % slower, 6 heads of 3.7k tokens 128.8 -> 130.3.)
        if (p->n_long_ktiles > 0) {
            const int64_t routed = (int64_t)L * p->k / 128, n_kt = (int64_t)p->ktiles.size();        // (tiles of picks, all chunks)
            int64_t all = 0;
            for (const KTile &kt : p->ktiles) all += kt.n_anc;
            all += routed * n_kt / std::max(C, 1);
            const int64_t share = std::max<int64_t>(4, std::max(all * p->H / p->n_sm, all / n_kt));
            for (int x = 0; x < p->n_long_ktiles; ++x) {
                KTile &kt = p->ktiles[x];
                if (kt.n_anc >= 2 * share) kt.parts = (int32_t)std::min<int64_t>(kMaxSplit, (kt.n_anc + share - 1) / share);
                p->n_split = std::max(p->n_split, kt.parts);
            }
        }
    }
    // Query-list capacities: chunk c can be picked by at most the rows after it (causal) or by
    // every row (non-causal); the lists sit back to back at these fixed offsets, so routing can
    // append to them without a counting pass.
    p->cap_off.assign(C + 1, 0);
    for (int c = 0; c < C; ++c) {
        const int64_t cap = p->k == 0 ? 0 : ((p->flags & MOC_FLAG_CAUSAL) ? L - p->off[c + 1] : L);
        const int64_t next = (int64_t)p->cap_off[c] + cap;
        if (next >= 2147483647LL) return MOC_ERR_SHAPE;
        p->cap_off[c + 1] = (int32_t)next;
    }
    for (KTile &kt : p->ktiles) kt.list = p->cap_off[kt.chunk];
    // score columns: the chunks that are not text; per query chunk its candidate columns (not an anchor, strictly
    // earlier if causal), whether they form a prefix of the columns (they do under the causal rule: everything
    // before the own shot's window), and how far any query up to that chunk can reach
    std::vector<int32_t> &col_chunk = tab.col_chunk, col_of(C, -1);
    for (int j = 0; j < C; ++j)
        if (p->mod[j] != 1) { col_of[j] = (int32_t)col_chunk.size(); col_chunk.push_back(j); }
    p->ncol = (int)col_chunk.size();
    p->routed_key_tiles = 0;
    for (int j : col_chunk) p->routed_key_tiles += (p->off[j + 1] - p->off[j] + 127) / 128;
    p->cwords = std::max(1, (p->ncol + 31) / 32);
    p->c_pad = std::max(16, (p->ncol + 15) / 16 * 16);
    tab.cand_c.assign((size_t)C * p->cwords, 0u);
    tab.lim.assign(C, 0);
    tab.reach.assign(C, 0);
    uint32_t *cand_c = tab.cand_c.data();
    int32_t *lim = tab.lim.data(), *reach = tab.reach.data();
    const bool causal = p->flags & MOC_FLAG_CAUSAL;
    p->prefix_mode = 1;
    for (int c = 0; c < C; ++c) {
        int n_cand = 0, top = 0;
        uint32_t *row = cand_c + (size_t)c * p->cwords;
        for (int j = 0; j < (causal ? c : C); ++j) {
            if (is_anchor(c, j)) continue;
            const int col = col_of[j];          // a non-anchor is never text
            row[col / 32] |= 1u << (col % 32);
            ++n_cand;
            top = col + 1;
        }
        lim[c] = top == n_cand ? n_cand : -1;
        if (lim[c] < 0) p->prefix_mode = 0;
        reach[c] = std::max(top, c ? reach[c - 1] : 0);
    }
    for (int c = 0; c < C; ++c) {
        if (c == 0 || p->shot[c] != p->shot[c - 1]) p->shot_chunks.push_back(KeyRange{c, c});
        p->shot_chunks.back().t1 = c + 1;
    }
    p->partials_budget = (size_t)6 << 30;
    p->wait_us = 0;
    layout_workspace(p);
    return MOC_OK;
}

}  // namespace moc

using namespace moc;

extern "C" int moc_plan_create(const moc_problem *pr, moc_plan **out) {
    if (!pr || !out) return MOC_ERR_NULL;
    *out = nullptr;
    if (int r = check_problem(pr)) return r;
    const int C = pr->n_chunks, L = pr->n_tokens;
    int dev = 0;
    MOC_CUDA_TRY(cudaGetDevice(&dev));
    // two attributes, not the whole property structure, which takes the driver a millisecond or two to fill in
    int cc_major = 0, n_sm = 0;
    MOC_CUDA_TRY(cudaDeviceGetAttribute(&cc_major, cudaDevAttrComputeCapabilityMajor, dev));
    MOC_CUDA_TRY(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
    if (cc_major != 10) return MOC_ERR_ARCH;

    moc_plan *p = new (std::nothrow) moc_plan();
    if (!p) return MOC_ERR_CUDA;
    p->device = dev;
    DeviceTables tab;
    if (int r = derive_plan(p, pr, n_sm, tab)) { delete p; return r; }
    const std::vector<uint32_t> &bits = tab.bits, &cand_c = tab.cand_c;
    const std::vector<int32_t> &unit_chunk = tab.unit_chunk, &lim = tab.lim, &reach = tab.reach, &col_chunk = tab.col_chunk;
    // the fixed scratch of moc_chunk_pool_noalloc: its address is looked up here, where allocating is allowed
    if (int r = pool_scratch_prepare(dev)) { delete p; return r; }

    // one device blob
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, 256); return at; };
    size_t o_off = take(4 * (C + 1)), o_shot = take(4 * C), o_mod = take(C);
    size_t o_bits = take(4 * bits.size()), o_aoff = take(4 * (C + 1)), o_arng = take(sizeof(KeyRange) * p->anc_rng.size());
    size_t o_roff = take(4 * (C + 1)), o_ranc = take(4 * p->ranc.size()), o_qt = take(sizeof(WorkItem) * p->qitems.size());
    size_t o_puo = take(4 * (C + 1)), o_puc = take(4 * unit_chunk.size()), o_cap = take(4 * (C + 1)), o_crng = take(sizeof(KeyRange) * C), o_kt = take(sizeof(KTile) * p->ktiles.size()), o_qrng = take(sizeof(KeyRange) * p->qry_rng.size());
    size_t o_shots = take(sizeof(KeyRange) * p->shot_chunks.size());
    size_t o_candc = take(4 * cand_c.size()), o_lim = take(4 * C), o_reach = take(4 * C), o_colc = take(4 * std::max<size_t>(col_chunk.size(), 1));
    const size_t from_host = o, o_tok = take(4 * (size_t)L);             // the token table is made on the device
    cudaError_t e = cudaMalloc(&p->d_blob, o);
    if (e != cudaSuccess) { set_cuda_error(e, "cudaMalloc(plan tables)"); delete p; return MOC_ERR_CUDA; }
    char *b = static_cast<char *>(p->d_blob);
    // the tables are put together on the host and go over in one copy (twenty small ones took longer than everything else here)
    std::vector<char> host(from_host);
    auto up = [&](size_t at, const void *src, size_t bytes) { if (bytes) memcpy(host.data() + at, src, bytes); };
    up(o_off, p->off.data(), 4 * (C + 1));
    up(o_shot, p->shot.data(), 4 * C);
    up(o_mod, p->mod.data(), C);
    up(o_bits, bits.data(), 4 * bits.size());
    up(o_aoff, p->anc_off.data(), 4 * (C + 1));
    up(o_arng, p->anc_rng.data(), sizeof(KeyRange) * p->anc_rng.size());
    up(o_roff, p->ranc_off.data(), 4 * (C + 1));
    up(o_ranc, p->ranc.data(), 4 * p->ranc.size());
    up(o_qt, p->qitems.data(), sizeof(WorkItem) * p->qitems.size());
    up(o_puo, p->pool_unit_off.data(), 4 * (C + 1));
    up(o_puc, unit_chunk.data(), 4 * unit_chunk.size());
    up(o_cap, p->cap_off.data(), 4 * (C + 1));
    up(o_crng, tab.chunk_rng.data(), sizeof(KeyRange) * C);
    up(o_kt, p->ktiles.data(), sizeof(KTile) * p->ktiles.size());
    up(o_qrng, p->qry_rng.data(), sizeof(KeyRange) * p->qry_rng.size());
    up(o_candc, cand_c.data(), 4 * cand_c.size());
    up(o_lim, lim.data(), 4 * C);
    up(o_reach, reach.data(), 4 * C);
    up(o_colc, col_chunk.data(), 4 * col_chunk.size());
    up(o_shots, p->shot_chunks.data(), sizeof(KeyRange) * p->shot_chunks.size());
    // On a stream of its own: on the legacy stream the copy would wait for what the caller has under way there.  The plan is
    // handed out when the tables are there, for a stream of any kind.
    cudaStream_t st = nullptr;
    e = table_stream(&st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b, host.data(), from_host, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        token_chunk_kernel<<<(unsigned)C, 256, 0, st>>>((const int32_t *)(b + o_off), (int32_t *)(b + o_tok));
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { set_cuda_error(e, "plan tables"); cudaFree(p->d_blob); delete p; return MOC_ERR_CUDA; }
    p->d_off = (int32_t *)(b + o_off); p->d_shot = (int32_t *)(b + o_shot); p->d_mod = (uint8_t *)(b + o_mod);
    p->d_tok_chunk = (int32_t *)(b + o_tok); p->d_anc_bits = (uint32_t *)(b + o_bits);
    p->d_anc_off = (int32_t *)(b + o_aoff); p->d_anc_rng = (KeyRange *)(b + o_arng);
    p->d_ranc_off = (int32_t *)(b + o_roff); p->d_ranc = (int32_t *)(b + o_ranc); p->d_qitems = (WorkItem *)(b + o_qt);
    p->d_pool_unit_off = (int32_t *)(b + o_puo); p->d_pool_unit_chunk = (int32_t *)(b + o_puc);
    p->d_cap_off = (int32_t *)(b + o_cap);
    p->d_chunk_rng = (KeyRange *)(b + o_crng);
    p->d_ktiles = (KTile *)(b + o_kt);
    p->d_qry_rng = (KeyRange *)(b + o_qrng);
    p->d_cand_c = (uint32_t *)(b + o_candc); p->d_lim = (int32_t *)(b + o_lim); p->d_reach = (int32_t *)(b + o_reach);
    p->d_col_chunk = (int32_t *)(b + o_colc);
    p->d_shot_chunks = (KeyRange *)(b + o_shots);
    *out = p;
    return MOC_OK;
}

extern "C" int moc_plan_destroy(moc_plan *p) {
    if (!p) return MOC_ERR_NULL;
    if (p->d_blob) cudaFree(p->d_blob);
    delete p;
    return MOC_OK;
}

extern "C" int moc_plan_set_workspace_budget(moc_plan *p, size_t max_bytes) {
    if (!p) return MOC_ERR_NULL;
    const size_t per_head = sizeof(__nv_bfloat16) * (((size_t)p->L + 127) / 128 * 128) * p->k * p->d;
    const size_t old = p->partials_budget;
    // the smallest workspace there is: one head at a time (two buffers of one head, or one if there is one head)
    p->partials_budget = p->H > 1 ? 2 * per_head : per_head;
    layout_workspace(p);
    const size_t rest = p->ws.fwd_end - p->partials_budget;
    if (p->ws.fwd_end > max_bytes) {
        p->partials_budget = old;
        layout_workspace(p);
        return MOC_ERR_TOO_LARGE;
    }
    p->partials_budget = std::max(p->partials_budget, max_bytes - rest - 65536);
    layout_workspace(p);
    if (p->ws.fwd_end > max_bytes) return MOC_ERR_TOO_LARGE;       // cannot happen: the partials only shrank
    return MOC_OK;
}

extern "C" int moc_workspace_bytes(const moc_plan *p, int with_bwd, size_t *bytes) {
    if (!p || !bytes) return MOC_ERR_NULL;
    *bytes = with_bwd ? p->ws.bwd_end : p->ws.fwd_end;
    return MOC_OK;
}

static int check_dev_ptrs(std::initializer_list<const void *> ptrs, size_t a) {
    for (const void *q : ptrs) {
        if (!q) return MOC_ERR_NULL;
        if (!aligned(q, a)) return MOC_ERR_ALIGN;
    }
    return MOC_OK;
}

static int enter(const moc_plan *p) {
    if (!p) return MOC_ERR_NULL;
    int dev = -1;
    MOC_CUDA_TRY(cudaGetDevice(&dev));
    if (dev != p->device) return MOC_ERR_ARCH;
    return MOC_OK;
}

extern "C" int moc_chunk_pool(const moc_plan *p, const void *K, float *desc, void *ws, void *stream) {
    moc::NvtxRange nvtx_range("moc_chunk_pool");
    if (int r = enter(p)) return r;
    if (int r = check_dev_ptrs({K, desc}, 16)) return r;
    if (!ws) return MOC_ERR_WORKSPACE;
    if (!aligned(ws, 256)) return MOC_ERR_ALIGN;
    return launch_chunk_pool(p, (const __nv_bfloat16 *)K, desc, ws, (cudaStream_t)stream);
}

extern "C" int moc_route(const moc_plan *p, const void *Q, const float *desc, int32_t *sel_idx, void *ws, void *stream) {
    moc::NvtxRange nvtx_range("moc_route");
    if (int r = enter(p)) return r;
    if (int r = check_dev_ptrs({Q, desc}, 16)) return r;
    if (p->k > 0) { if (int r = check_dev_ptrs({sel_idx}, 4)) return r; }
    if (!ws) return MOC_ERR_WORKSPACE;
    if (!aligned(ws, 256)) return MOC_ERR_ALIGN;
    return launch_route(p, (const __nv_bfloat16 *)Q, desc, sel_idx, ws, (cudaStream_t)stream);
}

extern "C" int moc_lists_from_sel(const moc_plan *p, int32_t *sel_idx, void *ws, void *stream) {
    moc::NvtxRange nvtx_range("moc_lists_from_sel");
    if (int r = enter(p)) return r;
    if (p->k > 0) { if (int r = check_dev_ptrs({sel_idx}, 4)) return r; }
    if (!ws) return MOC_ERR_WORKSPACE;
    if (!aligned(ws, 256)) return MOC_ERR_ALIGN;
    return launch_lists_from_sel(p, sel_idx, ws, (cudaStream_t)stream);
}

extern "C" int moc_context_drop(const moc_plan *p, int32_t *sel_idx, float p_max, float lambda, uint64_t seed, void *ws,
                                void *stream) {
    moc::NvtxRange nvtx_range("moc_context_drop");
    if (int r = enter(p)) return r;
    if (!(p_max >= 0.f && p_max <= 1.f) || !(lambda >= 0.f && lambda <= 8.f)) return MOC_ERR_SHAPE;
    if (p->k > 0) { if (int r = check_dev_ptrs({sel_idx}, 4)) return r; }
    if (!ws) return MOC_ERR_WORKSPACE;
    if (!aligned(ws, 256)) return MOC_ERR_ALIGN;
    if (int r = launch_context_drop(p, sel_idx, p_max, lambda, seed, (cudaStream_t)stream)) return r;
    return launch_lists_from_sel(p, sel_idx, ws, (cudaStream_t)stream);
}

extern "C" int moc_attend(const moc_plan *p, const void *Q, const void *K, const void *V, const int32_t *sel_idx,
                          void *O, float *lse, void *ws, void *stream) {
    moc::NvtxRange nvtx_range("moc_attend");
    if (int r = enter(p)) return r;
    if (int r = check_dev_ptrs({Q, K, V, O}, 16)) return r;
    if (int r = check_dev_ptrs({lse}, 4)) return r;
    if (p->k > 0) { if (int r = check_dev_ptrs({sel_idx}, 4)) return r; }
    if (!ws) return MOC_ERR_WORKSPACE;
    if (!aligned(ws, 256)) return MOC_ERR_ALIGN;
    auto q = (const __nv_bfloat16 *)Q, k = (const __nv_bfloat16 *)K, v = (const __nv_bfloat16 *)V;
    if (p->flags & kPrivFlagCudaCoreAttend)
        return launch_attend_scalar(p, q, k, v, sel_idx, (__nv_bfloat16 *)O, lse, ws, (cudaStream_t)stream);
    return launch_attend_tc(p, q, k, v, sel_idx, (__nv_bfloat16 *)O, lse, ws, (cudaStream_t)stream);
}

extern "C" int moc_attend_bwd(const moc_plan *p, const void *Q, const void *K, const void *V, const void *O,
                              const float *lse, const void *dO, const int32_t *sel_idx, void *dQ, void *dK, void *dV,
                              void *ws, void *stream) {
    moc::NvtxRange nvtx_range("moc_attend_bwd");
    if (int r = enter(p)) return r;
    if (int r = check_dev_ptrs({Q, K, V, O, dO, dQ, dK, dV}, 16)) return r;
    if (int r = check_dev_ptrs({lse}, 4)) return r;
    if (p->k > 0) { if (int r = check_dev_ptrs({sel_idx}, 4)) return r; }
    if (!ws) return MOC_ERR_WORKSPACE;
    if (!aligned(ws, 256)) return MOC_ERR_ALIGN;
    auto bwd = (p->flags & kPrivFlagCudaCoreAttend) ? launch_attend_bwd_scalar : launch_attend_bwd_tc;
    return bwd(p, (const __nv_bfloat16 *)Q, (const __nv_bfloat16 *)K, (const __nv_bfloat16 *)V, (const __nv_bfloat16 *)O, lse,
               (const __nv_bfloat16 *)dO, sel_idx, (__nv_bfloat16 *)dQ, (__nv_bfloat16 *)dK, (__nv_bfloat16 *)dV, ws,
               (cudaStream_t)stream);
}

extern "C" int moc_selected_pairs(const moc_plan *p, const void *ws, void *stream, int64_t *pairs) {
    if (int r = enter(p)) return r;
    if (!pairs) return MOC_ERR_NULL;
    if (!ws) return MOC_ERR_WORKSPACE;
    std::vector<int32_t> cnt((size_t)p->H * p->C);
    MOC_CUDA_TRY(cudaMemcpyAsync(cnt.data(), ws_ptr<int32_t>(ws, p->ws.cnt), cnt.size() * 4, cudaMemcpyDeviceToHost,
                                 (cudaStream_t)stream));
    MOC_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    int64_t per_head = 0;
    for (int c = 0; c < p->C; ++c) per_head += p->anc_tokens[c] * (int64_t)(p->off[c + 1] - p->off[c]);
    int64_t total = per_head * p->H;
    for (int h = 0; h < p->H; ++h)
        for (int c = 0; c < p->C; ++c) total += (int64_t)cnt[(size_t)h * p->C + c] * (p->off[c + 1] - p->off[c]);
    *pairs = total;
    return MOC_OK;
}

extern "C" int moc_get_status(const moc_plan *p, const void *ws, void *stream, int *device_status, int *detail) {
    if (int r = enter(p)) return r;
    if (!device_status) return MOC_ERR_NULL;
    if (!ws) return MOC_ERR_WORKSPACE;
    int32_t st[2] = {0, 0};
    MOC_CUDA_TRY(cudaMemcpyAsync(st, ws_ptr<int32_t>(ws, p->ws.status), sizeof st, cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    MOC_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    *device_status = st[0];
    if (detail) *detail = st[1];
    return MOC_OK;
}

extern "C" int moc_debug_use_cuda_core_attention(moc_plan *p, int on) {
    if (!p) return MOC_ERR_NULL;
    p->flags = on ? (p->flags | kPrivFlagCudaCoreAttend) : (p->flags & ~kPrivFlagCudaCoreAttend);
    return MOC_OK;
}

extern "C" int moc_debug_set_wait_limit_us(moc_plan *p, unsigned us) {
    if (!p) return MOC_ERR_NULL;
    p->wait_us = us;
    return MOC_OK;
}

extern "C" int moc_debug_shared_key_tiles(const moc_problem *pr, int n_sm, int cap, int *n_tiles, int *query_tiles, int *blocks,
                                           size_t *counter_room) {
    if (!pr || !n_tiles || !query_tiles || !blocks || !counter_room) return MOC_ERR_NULL;
    if (int r = check_problem(pr)) return r;
    if (n_sm < 1) return MOC_ERR_SHAPE;
    moc_plan p;
    DeviceTables tab;
    if (int r = derive_plan(&p, pr, n_sm, tab)) return r;
    const int most = dkv_split(&p);
    *n_tiles = p.n_long_ktiles;
    *counter_room = p.ws.queue - p.ws.pool_done;
    for (int x = 0; x < std::min(cap, p.n_long_ktiles); ++x) {
        query_tiles[x] = p.ktiles[x].n_anc;
        blocks[x] = std::min(p.ktiles[x].parts, most);
    }
    return MOC_OK;
}

extern "C" int64_t moc_launch_count(void) { return (int64_t)g_launches.load(); }

extern "C" const char *moc_strerror(int s) {
    switch (s) {
        case MOC_OK: return "ok";
        case MOC_ERR_NULL: return "a required pointer is NULL";
        case MOC_ERR_SHAPE: return "unsupported shape or parameter";
        case MOC_ERR_CHUNK_TABLE: return "invalid chunk table";
        case MOC_ERR_ALIGN: return "misaligned device pointer";
        case MOC_ERR_WORKSPACE: return "workspace missing, or it does not hold this plan's routing";
        case MOC_ERR_ARCH: return "device is not sm_100 or differs from the plan's device";
        case MOC_ERR_CUDA: return "CUDA runtime error";
        case MOC_ERR_TIMEOUT: return "a bounded device-side wait ran out";
        case MOC_ERR_TOO_LARGE: return "problem exceeds the fixed scratch of the no-allocation entry point, or the workspace budget";
        case MOC_ERR_INDEX: return "debug build: an index taken from the workspace was out of range";
        default: return "unknown status";
    }
}

extern "C" const char *moc_last_cuda_error(void) {
    static thread_local std::string copy;
    std::lock_guard<std::mutex> g(g_err_mu);
    copy = g_err;
    return copy.c_str();
}
