// sm_100a building blocks in inline PTX: mbarrier with bounded waits, TMA tile loads,
// TMEM allocation, tcgen05 MMA / commit / ld / st, and the shared-memory and instruction
// descriptors the MMA consumes.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "moc_common.cuh"

namespace moc {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---- mbarrier ----
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// One poll.  The hint lets the hardware park the thread until the phase completes or the hint
// (in nanoseconds) runs out, so a waiting warp does not take issue slots from the warps at work.
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(20000u)
        : "memory");
    return ok != 0;
}

// Every wait is bounded, by a number of polls (WaitBound).  The first wait of a CTA to run out leaves its code in the CTA's abort flag, which the CTA
// reports when it leaves (report_abort); its other waits run out by themselves, so that a CTA that is stuck leaves within a few seconds.  There are
// some forty waits in a kernel, and the loops of its warps share an instruction cache: what stands behind each is as short as
// can be.  (With a clock, the limit read from the workspace and the report at every wait the forward kernels were 20 KB
// longer: 264k tokens in 256-token chunks, 2 heads, 3.89 -> 4.23 ms; 33k-token clip at d = 64 1.20 -> 1.29; its backward 3.59 -> 3.62.  With nothing but a look
// at the flag beside the limit, 6 heads in 512-token chunks, the whole forward, 18.83 -> 19.10 ms, in 256-token chunks 14.28 -> 14.56; in the
// parked waits alone 19.30 and 14.41; with 32 bits of the clock besides 19.7 and 14.95.)
__device__ __forceinline__ bool gave_up(volatile int *abort_flag, int code) {
    if (*abort_flag == 0) *abort_flag = code;
    return false;
}
__device__ __forceinline__ void report_abort(int *status, int code) {
    if (code != 0 && atomicCAS(status, 0, MOC_ERR_TIMEOUT) == 0) status[ST_DETAIL] = code;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, const WaitBound &bound, int code) {
    for (uint32_t it = 0; !mbar_try_wait(bar, parity);)
        if (++it > bound.parked) return gave_up(abort_flag, code);
    return true;
}

// One poll that never parks the thread, and the same bounded wait built on it: for the single thread
// that feeds the tensor pipe, where waking up late costs more than the issue slots of polling.
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_spin(uint32_t bar, uint32_t parity, volatile int *abort_flag, const WaitBound &bound, int code) {
    for (uint32_t it = 0; !mbar_test_wait(bar, parity);)
        if (++it > bound.polled) return gave_up(abort_flag, code);
    return true;
}

// The same for a counter in global memory that another CTA adds to.
__device__ __forceinline__ bool wait_count(const int *ctr, int need, volatile int *abort_flag, const WaitBound &bound, int code) {
    for (uint32_t it = 0; *(volatile const int *)ctr < need;) {
        __nanosleep(200);
        if (++it > bound.looks) return gave_up(abort_flag, code);
    }
    return true;
}

__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
// makes generic-proxy writes to shared memory visible to the async proxy (TMA, tensor core)
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---- TMA: 2-D tile load into this CTA's shared memory, completion on an mbarrier ----
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar)
                 : "memory");
}
// four rows of a 2-D tensor, 64 columns from column x on, into four consecutive 128-byte rows of shared memory
__device__ __forceinline__ void tma_gather4(uint32_t dst, const CUtensorMap *map, int x, int r0, int r1, int r2, int r3, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cta.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(r0), "r"(r1), "r"(r2), "r"(r3), "r"(bar)
                 : "memory");
}
// n contiguous bytes (a multiple of 16; both addresses 16-byte aligned)
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t n, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(n), "r"(bar) : "memory");
}
__device__ __forceinline__ void ld_shared_128(uint32_t addr, uint32_t (&v)[4]) {
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

// ---- TMEM ----
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// MMA and commit for a warp that stays together: every lane calls them with the same values, and the lane that elect.sync
// names issues (always the same one for a full warp).  Nothing diverges around them, so the operands live in uniform
// registers instead of being moved there, one by one, for every MMA: measured inside the forward attention kernel, a group
// of eight S MMAs leaves the issuing warp after 220 cycles instead of 730 (the pipe needs 512).
// ss: D[tmem] (+)= A[smem] B[smem]; ts: A in TMEM.  Descriptors come as (low word, high word): only the 14-bit start address
// in the low word moves between the MMAs of a tile.  The commit arrives on an mbarrier once every tcgen05 operation issued
// so far by this lane has completed.
__device__ __forceinline__ void mma_ss_elect(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                             uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_ts_elect(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t.reg .b64 db;\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_commit_elect(uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
        : "memory");
}
// A value that every lane of the warp holds, as one the compiler knows to be the same in all of them.
// The warp's number in the block is taken through it in the kernels whose warps have roles: with threadIdx.x >> 5 alone a role's
// branch counts as one that the lanes may part at, and the issuers' loops were written out with a guard around each of their
// instructions (some 33 a tcgen05.mma).  The code of the kernels is what it saves, which in these is what bounds the
// loops (a few roles' loops share the instruction cache).  Plain -> through this, with the backward's row loaders looped: the code
// of the dK/dV kernel 96 -> 55 KB, of dQ 89 -> 57 (d = 128); 24 heads of 6.7k tokens, 4 picks, backward 9.95 -> 9.69 ms, 6 heads
// 2.21 -> 2.14 ms, routing 64 -> 58 us; 2 heads of 115k tokens, 30 picks, routing 690 -> 652 us; the forward as before.
__device__ __forceinline__ int uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }

// 32 consecutive fp32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
// 64 consecutive fp32 columns of 16 TMEM lanes (from the address's lane on): of every eight columns x, this thread holds the
// two from 2 (lane % 4) on, of row lane / 4 in r[4 x], r[4 x + 1] and of row lane / 4 + 8 in r[4 x + 2], r[4 x + 3]
__device__ __forceinline__ void tmem_ld_16x256b(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
// 8 consecutive fp32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
          "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
          "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

// 16-byte asynchronous copy global -> shared; src_bytes = 0 writes zeros instead
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// ---- small arithmetic helpers of the softmax-side threads ----
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// two fp32 values in one 64-bit register pair, for the packed fp32 instructions
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// (lo, hi) -> packed bf16x2, round to nearest even
__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// ---- descriptors ----
// Shared-memory matrix descriptor, 128-byte swizzle: start address, leading / stride byte
// offsets (all in 16-byte units), descriptor version 1, layout type 2 (SWIZZLE_128B).
// K-major operand (rows of 128 bytes along K): 8-row groups are `sbo` bytes apart, lbo unused.
// MN-major operand (rows of 128 bytes along M/N): 64-element blocks along M/N are `lbo`
// bytes apart, 8-row groups along K are `sbo` bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) | ((uint64_t)(sbo_bytes >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}
// Instruction descriptor, kind::f16: fp32 accumulator, bf16 A and B, M x N tile.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N, int a_mn_major, int b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn_major << 15) | ((uint32_t)b_mn_major << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// byte offset of 16-byte chunk `c16` (0..7) of row `r` inside a 128-byte-swizzled tile of
// 128-byte rows whose base is 1024-byte aligned (the layout TMA SWIZZLE_128B produces)
__device__ __forceinline__ uint32_t sw128_offset(int r, int c16) { return (uint32_t)(r * 128 + ((c16 ^ (r & 7)) << 4)); }

// 32-byte (one sector) global load that is cached in L2 only, and 32-byte global store; addresses 32-byte aligned.
// The load where cond holds (predicated: as a branch around it, the values it leaves alone cost registers twice)
__device__ __forceinline__ void ld_cg_256_if(bool cond, const void *ptr, uint32_t (&u)[8]) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %9, 0;\n\t"
        "@p ld.global.cg.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t}"
        : "+r"(u[0]), "+r"(u[1]), "+r"(u[2]), "+r"(u[3]), "+r"(u[4]), "+r"(u[5]), "+r"(u[6]), "+r"(u[7])
        : "l"(ptr), "r"((int)cond));
}
__device__ __forceinline__ void st_256(void *ptr, const uint32_t (&u)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(ptr), "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]), "r"(u[5]), "r"(u[6]), "r"(u[7])
                 : "memory");
}

// The four lanes of a row in tmem_ld_16x256b: of its 64 columns lane i holds pairs 4 x + i (columns 8 x + 2 i, + 1) in word x.
// Afterwards words 0..3 of lane i are columns 8 i .. 8 i + 7 and words 4..7 columns 32 + 8 i .. 32 + 8 i + 7: two 16-byte pieces, of
// which the four lanes' make 64 contiguous bytes each.
__device__ __forceinline__ void quad_transpose(uint32_t (&u)[8], int i) {
#pragma unroll
    for (int z = 0; z < 8; z += 4) {
        // neighbours exchange the words off the diagonal of their 2 x 2 blocks, then lanes two apart the blocks off the diagonal
#pragma unroll
        for (int y = 0; y < 4; y += 2) {
            const uint32_t other = __shfl_xor_sync(0xffffffffu, (i & 1) ? u[z + y] : u[z + y + 1], 1);
            if (i & 1) u[z + y] = other;
            else u[z + y + 1] = other;
        }
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const uint32_t other = __shfl_xor_sync(0xffffffffu, (i & 2) ? u[z + y] : u[z + y + 2], 2);
            if (i & 2) u[z + y] = other;
            else u[z + y + 2] = other;
        }
    }
}
// what quad_transpose leaves, to a row's 64 columns at `row` (16-byte aligned: a caller's tensor promises no more)
__device__ __forceinline__ void store_quad(__nv_bfloat16 *row, int i, const uint32_t (&u)[8]) {
    uint4 *dst = reinterpret_cast<uint4 *>(row) + i;
    dst[0] = make_uint4(u[0], u[1], u[2], u[3]);
    dst[4] = make_uint4(u[4], u[5], u[6], u[7]);
}

}  // namespace tc

// host: encode a 2-D bf16 tensor map [rows][cols], box {64 cols, box_rows}, 128-byte swizzle
int make_tmap_2d_bf16(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows);

}  // namespace moc
