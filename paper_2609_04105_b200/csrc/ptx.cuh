// Thin inline-PTX wrappers for sm_100a: mbarrier, TMA (loads of this CTA only), tcgen05
// (tensor memory allocation, block-scaled FP4 MMA, scale-factor copy, TMEM loads/stores).
// Every wait is bounded: a wait that runs out returns false and the caller unwinds.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fp4attn {
namespace ptx {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile(
      "{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(pred));
  return pred != 0;
}

// ------------------------------------------------------------------ mbarrier
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// has the phase completed?  Never suspended; the whole warp, with one answer
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return __all_sync(0xffffffffu, ok != 0);
}
// Bounded waits.  The word at `abort_at` (shared memory) tells the end of the kernel that some wait ran out, and every other
// wait of the CTA, so that its roles fall out together.
//
// A wait is a bare poll loop: the instruction's own (short, hardware-chosen) suspension, a counter, nothing else.  The
// waiting warps share their schedulers with the softmax warps, whose time is instruction dispatch, so what a wait executes
// is taken from them.  Attention at B=4, H=16, N=8192, d=128 (exact | affine map): a poll with a suspend-time hint, a clock
// read, a look at the abort flag and a warp vote around it all 967 | 750 us; bare polls with the hint 923 | 687 us; without
// it 903 | 619 us; four polls per trip of the counter 916 | 620 us.
// How long the hardware suspends a poll is its own choice (measured on a barrier that nothing completes: 4 us), so a count of
// polls bounds no time: every kPolls polls the wait looks at the abort word and the clock.  Both loops are one piece of assembly and the word goes by its shared-memory
// address: the same as C++ statements after the poll loop, with a generic pointer, spilled up to 32 bytes a thread and
// took 3-6 % longer.
constexpr uint32_t kPolls = 1u << 6;           // a look every 0.25 ms
constexpr uint32_t kWaitClocks = 1u << 31;     // SM clocks, about a second; the longest wait of a healthy kernel lasts as long as one work item
__device__ __forceinline__ bool mbar_poll(uint32_t bar, uint32_t parity, uint32_t abort_at, uint32_t limit) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .u32 n, v, t;\n\t"
      "mov.u32 n, 0;\n"
      "MBAR_POLL:\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "@p bra MBAR_DONE;\n\t"
      "add.u32 n, n, 1;\n\tand.b32 v, n, %5;\n\tsetp.ne.u32 q, v, 0;\n\t@q bra MBAR_POLL;\n\t"
      "ld.volatile.shared.u32 v, [%3];\n\tsetp.ne.u32 q, v, 0;\n\t@q bra MBAR_DONE;\n\t"
      "mov.u32 v, %%clock;\n\tsetp.eq.u32 q, n, %6;\n\t@q mov.u32 t, v;\n\t"                  // t: the first look
      "sub.u32 v, v, t;\n\tsetp.lt.u32 q, v, %4;\n\t@q bra MBAR_POLL;\n"
      "MBAR_DONE:\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(abort_at), "r"(limit), "n"(kPolls - 1), "n"(kPolls) : "memory");
  return ok != 0;
}
// One thread waits by itself.
__device__ __forceinline__ bool mbar_wait_thread(uint32_t bar, uint32_t parity, uint32_t abort_at, uint32_t limit = kWaitClocks) {
  if (mbar_poll(bar, parity, abort_at, limit)) return true;
  asm volatile("st.volatile.shared.u32 [%0], 1;" ::"r"(abort_at) : "memory");
  return false;
}
// The whole warp waits and leaves as one, with one answer: a poll's answer is each thread's own, the warp may come here split
// (from an arrival of lane 0), and what follows are warp-wide instructions, which a part of a warp must not enter.
// VOTE_FIRST: a first poll with a vote of its own, which most waits end with: d = 64,
// N = 8192, NVFP4 1852 us without, 1815 with it; not in the FP8 P/V kernels (masked, N = 9600: 214 us without, 220 with it).
template <bool VOTE_FIRST = true>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t abort_at, uint32_t limit = kWaitClocks) {
  if (VOTE_FIRST && __all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  return __all_sync(0xffffffffu, mbar_wait_thread(bar, parity, abort_at, limit));
}

__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// generic-proxy writes to shared memory -> visible to the async proxy (TMA, tcgen05 operands)
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ------------------------------------------------------------------ TMA (bulk tensor loads, this CTA only)
__device__ __forceinline__ void prefetch_tensormap(const void* tmap) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(tmap) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void* tmap, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(tmap), "r"(x), "r"(y), "r"(bar) : "memory");
}
// untiled bulk copy global -> shared; both addresses 16-byte aligned, bytes a multiple of 16
__device__ __forceinline__ void bulk_load_1d(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// bulk tensor store shared -> global (this CTA's shared memory), tracked by bulk async-groups
__device__ __forceinline__ void tma_store_2d(const void* tmap, int x, int y, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
               ::"l"(tmap), "r"(x), "r"(y), "r"(src) : "memory");
}
__device__ __forceinline__ void bulk_commit_group() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// all earlier bulk groups of this thread have finished READING their shared-memory source
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// all earlier bulk groups of this thread are complete (writes to global memory done)
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// ------------------------------------------------------------------ tensor memory
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t ncols) {      // one full warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {       // one full warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// arrive on an mbarrier when every tcgen05 op issued so far by this thread has completed
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// 32 lanes x 128 bits of shared memory -> TMEM, replicated to all four lane quarters
// (the placement block-scaled MMAs read their scale factors from)
__device__ __forceinline__ void tc_cp_32x128b_warpx4(uint32_t taddr, uint64_t sdesc) {
  asm volatile("tcgen05.cp.cta_group::1.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}

// D[tmem] (+)= A[smem] * B[smem], E2M1 operands, block scales read from TMEM.
// scale_vec::2X : one scale per 32 elements along K (K = 64 -> 2 scales per row)
// scale_vec::4X : one scale per 16 elements along K (4 scales per row)
__device__ __forceinline__ void tc_mma_fp4_2x(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                              uint32_t sfa, uint32_t sfb, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::mxf4nvf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
      ::"r"(d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb) : "memory");
}
__device__ __forceinline__ void tc_mma_fp4_4x(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                              uint32_t sfa, uint32_t sfb, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::mxf4nvf4.block_scale.scale_vec::4X [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
      ::"r"(d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb) : "memory");
}

// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp receives lane (base + i)
__device__ __forceinline__ void tmem_ld_32x32b_x32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
// 16-column variants (lower register footprint)
__device__ __forceinline__ void tmem_ld_32x32b_x16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st_32x32b_x16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

__device__ __forceinline__ void tmem_st_32x32b_x8(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}
// block-scaled FP4 product whose A operand lives in tensor memory (128 lanes x 8 columns per K64 slice)
__device__ __forceinline__ void tc_mma_fp4_2x_ta(uint32_t d, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                                 uint32_t sfa, uint32_t sfb, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::mxf4nvf4.block_scale.scale_vec::2X [%0], [%1], %2, %3, [%5], [%6], p;\n\t}"
      ::"r"(d), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb) : "memory");
}

// ------------------------------------------------------------------ descriptors
// Shared-memory matrix descriptor (64-bit) of a K-major operand.
//   bits 0-13 start address >> 4 | 16-29 leading byte offset >> 4 | 32-45 stride byte offset >> 4
//   46-47 descriptor version (1 on sm_100) | 61-63 swizzle: 0 none, 2 = 128 B, 4 = 64 B, 6 = 32 B
// Swizzled K-major tiles whose K extent fits one swizzle row ignore the leading offset; the stride
// offset is the distance between consecutive groups of eight rows.
enum : uint64_t { kSwzNone = 0, kSwz128 = 2, kSwz64 = 4, kSwz32 = 6 };
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes, uint64_t swz) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) |
         ((uint64_t)(sbo_bytes >> 4) << 32) | (1ull << 46) | (swz << 61);
}

// Instruction descriptor of the block-scaled FP4 kinds (32-bit):
//   4-5 B scale id | 7-9 A format (E2M1 = 1) | 10-12 B format | 15/16 A/B major (0 = K-major)
//   17-22 N >> 3 | 23 scale format (0 = UE4M3, 1 = UE8M0) | 24-28 M >> 4 | 29-30 A scale id | 31 K (0 = 64)
// A scale id selects which byte(s) of the 4-byte scale column an instruction reads: with two
// scales per row (scale_vec::2X) ids 0 and 2 address bytes {0,1} and {2,3}.
__host__ __device__ constexpr uint32_t make_idesc_fp4(int M, int N, bool ue8m0, int a_sf_id, int b_sf_id) {
  return (uint32_t)(b_sf_id & 3) << 4 | 1u << 7 | 1u << 10 | (uint32_t)(N >> 3) << 17 |
         (ue8m0 ? 1u : 0u) << 23 | (uint32_t)(M >> 4) << 24 | (uint32_t)(a_sf_id & 3) << 29;
}

}  // namespace ptx
}  // namespace fp4attn
