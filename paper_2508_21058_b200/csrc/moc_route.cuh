// What the two routing kernels share.
#pragma once
#include "moc_common.cuh"

namespace moc {

// The end of a routing kernel.  The last block to get here turns the pick counts into the running counts of attention tiles over the (head,
// chunk) pairs and marks the workspace (what route_tiles_kernel does on the paths that have no such block): one
// launch less.  Every block's counts are in place before it arrives (the atomics that made them have
// returned), and the fence orders them before the arrival.
__device__ __forceinline__ void finish_route(int *status, const int *cnt, int *tile_off, int HC, uint32_t cookie, int n_threads) {
    __shared__ int s_last, s_wsum[32];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        __threadfence();
        s_last = atomicAdd(&status[ST_ARRIVE], 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int per = (HC + n_threads - 1) / n_threads, i0 = min(t * per, HC), i1 = min(i0 + per, HC);
    int mine = 0;
    for (int i = i0; i < i1; ++i) mine += (__ldcg(cnt + i) + kQTileRows - 1) / kQTileRows;
    int incl = mine;                                     // inclusive scan over the block: warps by shuffles, then warp totals
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += up;
    }
    if (lane == 31) s_wsum[warp] = incl;
    __syncthreads();
    int at = incl - mine;
    for (int w = 0; w < warp; ++w) at += s_wsum[w];
    for (int i = i0; i < i1; ++i) {
        tile_off[i] = at;
        at += (__ldcg(cnt + i) + kQTileRows - 1) / kQTileRows;
    }
    if (t == n_threads - 1) {
        tile_off[HC] = at;
        status[ST_COOKIE] = (int)cookie;
    }
}

// Which kernel routes: a thread per row keeps its picks in a sorted list (moc_route.cu), or threads count and a warp per row sorts the scores that
// reach a threshold (moc_route_long.cu).  The lines, measured (list -> threshold, 2 heads): up to 16 picks the list is faster (168 columns,
// 14 picks 334 -> 364 us, 504: 394 -> 453), from 17 on level or slower except where one block of descriptors serves a short
// stream: 132 columns, 34k tokens, 24 picks 69 -> 81; 84 columns, 132k tokens, 24 picks 160 -> 214; but 160 columns, 264k, 24 picks 570 -> 391, 40k tokens,
// 205 columns 100 -> 86.  Beyond 32 picks a list is in no case faster (132 columns, 34k tokens, 40 picks 152 -> 90).
inline bool route_is_long(const moc_plan *p) { return p->k > 32 || (p->k > 16 && p->c_pad > 144); }
int launch_route_long(const moc_plan *p, const __nv_bfloat16 *Q, const __nv_bfloat16 *desc3, int32_t *sel, void *ws, cudaStream_t s);

}  // namespace moc
