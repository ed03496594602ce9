// Thin wrappers over the sm_100a instructions used by the tensor-core kernels:
// mbarrier, TMA tile loads (no multicast anywhere), tcgen05 TMEM allocation, the
// kind::i8 MMA, commit and TMEM loads.  Every wait is bounded.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace q4 {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same without being suspended until the phase ends (or a time limit): a look ahead
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: gives up after `limit` polls and returns false (the caller flags the error
// and stops waiting for anything else).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t limit = (1u << 22)) {
  for (uint32_t i = 0; i < limit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if (i > 64) __nanosleep(64);
  }
  return false;
}

// One lane of a converged warp.  The loops that issue copies and MMAs are walked by a whole warp with warp-uniform values;
// the instructions themselves are predicated on the elected lane (the forms below with `on` as first argument), not branched
// over.  The next stage's barrier is tested before a chunk's MMAs are issued, so
// that the latency of the answer passes beside them (mbar_test: mbarrier.try_wait would hold the warp while that stage is still
// on its way, 13 to 20 % of a search).  Clocks per K chunk (wait, four int8 MMAs 128 x N x 32, commit; operands
// in place, all SMs), N = 32 / 64 / 128: 308 / 318 / 334 with a branch and without the test, 168 / 192 / 256 this way; the
// tensor cores take 160 / 192 / 256.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred P;\n\t.reg .b32 R;\n\t"
      "elect.sync R|P, 0xffffffff;\n\t"
      "selp.b32 %0, 1, 0, P;\n\t}"
      : "=r"(p));
  return p;
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t on, uint64_t* bar, uint32_t bytes) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t"
      "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(smem_u32(bar)), "r"(bytes), "r"(on)
      : "memory");
}
__device__ __forceinline__ int uniform_warp() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, uint32_t limit = (1u << 22)) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, limit)) != 0;
}
// the same where the barrier has been tested already
__device__ __forceinline__ bool mbar_wait_warp_tested(bool ready, uint64_t* bar, uint32_t parity, uint32_t limit = (1u << 22)) {
  return __all_sync(0xffffffffu, ready) != 0 || mbar_wait_warp(bar, parity, limit);
}

// After a wait that has run out: nobody leaves while copies are on their way into the block's memory (bounded).  The last of
// the `issued` copies into a ring of `stages`; by a producer that gave up, for those it has issued, and by a consumer that gave
// up, for all of them (if the producer has not issued them all, it waits for its own).
__device__ __forceinline__ void ring_landed(uint64_t* full, int stages, int issued) {
  for (int j = max(issued - stages, 0); j < issued; ++j)
    if (!mbar_wait_warp(&full[j % stages], (uint32_t)(j / stages) & 1u)) break;
}

// 2-D tiled TMA load into shared memory, completion counted on an mbarrier.  x is the
// innermost (contiguous) coordinate and must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_load_2d(uint32_t on, void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n\t}"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(on)
      : "memory");
}
// `bytes` (a multiple of 16) from this CTA's shared memory into the shared memory of a CTA of the cluster by
// the bulk-copy engine; counted on the mbarrier at `mbar_addr`, an address in the receiver's window.  No
// multicast: one destination per copy.
__device__ __forceinline__ void bulk_copy_to_cluster(uint32_t dst_addr, uint32_t src_addr, uint32_t bytes,
                                                     uint32_t mbar_addr) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst_addr), "r"(src_addr), "r"(bytes), "r"(mbar_addr)
               : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

// int8 matrix [rows, k] with row pitch `pitch` bytes; box = 128 bytes of K x box_rows rows, 128-byte swizzle (q4_mma.cu).
bool make_tmap_i8(CUtensorMap* m, const void* base, uint64_t k, uint64_t rows, uint64_t pitch, uint32_t box_rows);

// ---- sums of exponentials -------------------------------------------------------------
// The output heads and the label-free end of a search sum a row's exponentials in shares, by these two functions, so that a
// blank's log-probability is the same bits in both.
// e^x = 2^(x log2 e) on the base-2 unit (ex2.approx: relative error 2^-22); .ftz: a result below 2^-126 is 0.  For terms of a
// sum that has a term e^0 = 1 only: 2^11 entries of less than 2^-126 are 2^-115 of it, its rounding is 2^-24.
__device__ __forceinline__ float exp_of_sum(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__fmul_rn(x, 1.4426950408889634f)));
  return y;
}
// A share's sum relative to its maximum m; entries that do not count are -inf (m = -inf: a share without entries).
// No branch for one: 32 exponentials with a branch each took 2950 clocks of a head, 1690 this way.
template <int N>
__device__ __forceinline__ float exp_sum(const float (&v)[N], float m) {
  const float top = m > -INFINITY ? m : 0.0f;
  float sum = 0.0f;
#pragma unroll
  for (int i = 0; i < N; ++i) sum += exp_of_sum(v[i] - top);
  return sum;
}
// Shares (maximum, sum) relative to the maximum m of all; a share without entries adds 0.
template <int N>
__device__ __forceinline__ float exp_sum(const float (&part_m)[N], const float (&part_s)[N], float m) {
  const float top = m > -INFINITY ? m : 0.0f;
  float sum = 0.0f;
#pragma unroll
  for (int i = 0; i < N; ++i) sum += part_s[i] * exp_of_sum(part_m[i] - top);
  return sum;
}

// ---- tensor memory ------------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile written by TMA with the 128-byte
// swizzle: rows of 128 bytes, groups of 8 rows 1024 bytes apart, tile base 1024-byte aligned.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);        // start address, 16-byte units
  d |= (uint64_t)0 << 16;                               // leading byte offset (unused here)
  d |= (uint64_t)(1024u >> 4) << 32;                    // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;                               // descriptor version for sm_100
  d |= (uint64_t)2 << 61;                               // layout: 128-byte swizzle
  return d;
}
// The same for a tile whose rows are 32 bytes (one MMA's worth of K) under the 32-byte swizzle: groups of 8
// rows 256 bytes apart, the 16-byte halves of rows 4..7 of a group exchanged.
__device__ __forceinline__ uint64_t umma_desc_sw32(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(256u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)6 << 61;                               // layout: 32-byte swizzle
  return d;
}
// Tiles of at most 16 rows are multiplied as 64-row tiles: an MMA of 32, 64 or 128 weight rows takes 24 / 32 / 64 clocks
// instead of 40 / 48 / 64 (measured; the rows' way into the tensor cores bounds the narrow ones).  Row r is lane
// 32 (r / 16) + r % 16 of tensor memory there; the other lanes hold nothing and stand for the rows from 64 on.  With more rows
// than the 16 of a lane quarter the epilogue works on half-filled warps.  Networks of 1024, 1024 and 2048 cells,
// 160 frames of one utterance at beam 16 3.72 ->
// 3.60 ms, beam 1 1.89 -> 1.85, but 8 x 8 rows 3.86 -> 3.90.
__host__ __device__ constexpr int umma_rows(int tile_rows) { return tile_rows <= 16 ? 64 : 128; }
__device__ __forceinline__ int umma_lane_row(int m, int quarter, int lane) {   // row of a warp's lane, m = umma_rows()
  return m == 128 ? 32 * quarter + lane : lane < 16 ? 16 * quarter + lane : 48 + 16 * quarter + lane;
}
// Instruction descriptor: signed 8-bit A and B, both K-major, int32 accumulate, M x N tile.
__device__ __forceinline__ uint32_t umma_idesc_i8(int M, int N) {
  return (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// D[tmem] (+)= A[smem] * B[smem]^T, M x N x 32 int8 (M, N: see umma_idesc_i8), by the lane whose `on` is not 0.
__device__ __forceinline__ void umma_i8(uint32_t on, uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(on)
      : "memory");
}
// Arrive on an mbarrier when all MMAs issued so far by that lane have completed.
__device__ __forceinline__ void umma_commit(uint32_t on, uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar)), "r"(on)
      : "memory");
}
// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp receives lane (base+i).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, int (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, int (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld(uint32_t taddr, int (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld(uint32_t taddr, int (&r)[16]) { tmem_ld16(taddr, r); }
__device__ __forceinline__ void tmem_ld(uint32_t taddr, int (&r)[32]) { tmem_ld32(taddr, r); }
// 16 consecutive columns of the warp's 32 lanes written, and the wait for such writes
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float4& a, const float4& b, const float4& c, const float4& d) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w), "f"(c.x), "f"(c.y), "f"(c.z), "f"(c.w),
      "f"(d.x), "f"(d.y), "f"(d.z), "f"(d.w)
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 256-bit global accesses (32-byte aligned addresses): one instruction per 8 floats.
__device__ __forceinline__ void ld_global_v8(const float* p, float4& lo, float4& hi) {
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(lo.x), "=f"(lo.y), "=f"(lo.z), "=f"(lo.w), "=f"(hi.x), "=f"(hi.y), "=f"(hi.z), "=f"(hi.w)
               : "l"(p));
}
__device__ __forceinline__ void st_global_v8(float* p, const float4& lo, const float4& hi) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(lo.x), "f"(lo.y),
               "f"(lo.z), "f"(lo.w), "f"(hi.x), "f"(hi.y), "f"(hi.z), "f"(hi.w)
               : "memory");
}

__device__ __forceinline__ void st_global_v8_b32(int32_t* p, int a0, int a1, int a2, int a3, int a4, int a5, int a6,
                                                 int a7) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a0), "r"(a1), "r"(a2),
               "r"(a3), "r"(a4), "r"(a5), "r"(a6), "r"(a7)
               : "memory");
}

}  // namespace q4
