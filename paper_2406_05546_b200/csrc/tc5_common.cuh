// PTX wrappers for the fifth-generation tensor-core path: mbarriers with bounded waits, TMA tile
// loads (each CTA loads its own tiles), tcgen05 MMA / commit / tensor-memory loads.
#pragma once
#include <cuda.h>
#include <stdint.h>

namespace psk {

constexpr long long WAIT_LIMIT_CYCLES = 2000000000ll;   // about one second: no wait lasts that long when all is well

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// Bounded wait for the phase with the given parity; false if the bound (in SM clock cycles) was exceeded.  The
// barrier is given by its shared-memory address; the clock is read only when the first try fails.
__device__ __forceinline__ bool mbar_try(uint32_t addr, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done) : "r"(addr), "r"(parity) : "memory");
  return done != 0;
}
__device__ __forceinline__ bool mbar_wait_addr(uint32_t addr, uint32_t parity, long long limit_cycles = WAIT_LIMIT_CYCLES) {
  if (mbar_try(addr, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
    if (mbar_try(addr, parity)) return true;
    if (clock64() - t0 > limit_cycles) return false;
  }
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit_cycles = WAIT_LIMIT_CYCLES) {
  return mbar_wait_addr(smem_u32(bar), parity, limit_cycles);
}

// A bounded wait of a whole warp that another role's abort ends too: the same answer in every lane, for the warp-wide
// tensor-memory reads behind it.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, const volatile uint32_t* abort_flag) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity) && !*abort_flag);
}

// What several warps do next: true in all of their THREADS threads if `ok` holds in every one of them, false in all otherwise.
// Every wait runs out on its own thread's clock, so threads that go on to exchange data behind a barrier of theirs settle
// first, here, whether all of them do: a warp that had given up alone would leave the others at that barrier for good.
template <int BARRIER, int THREADS>
__device__ __forceinline__ bool warps_agree(bool ok) {
  uint32_t all;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %3, 0;\n\t"
      "barrier.cta.red.and.pred q, %1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(all) : "n"(BARRIER), "n"(THREADS), "r"((uint32_t)ok) : "memory");
  return all != 0;
}

__device__ __forceinline__ void tma_load_3d(void* smem_dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2) : "memory");
}

__device__ __forceinline__ void tma_load_4d(void* smem_dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}

// MMAs, issued by a whole warp that has stayed together: one lane of it, always the same, issues.  Where a single lane's branch computes
// the operands' addresses, each of them goes from a vector register to a uniform one for every instruction; where the warp's lanes agree
// they are computed in uniform registers to begin with.  Clocks per instruction of the second convolution's products on the FP32
// path (M = 128, N = 32 .. 144, K = 16), one lane's branch -> whole warp: forward 86 -> 56, input gradient 96 -> 72.  us of kernels whose one
// issuing thread was behind: conv2_dw_tc5 85.4 -> 71.8 at 128 x 128 and 14.6 -> 12.8 at 4 x 16, tc5_fwd_narrow 17.9 -> 15.2 at 2 x 8, gemm_x3's
// weight gradient 171 -> 164 at 128 x 128, tc5_gemm's input gradient 53.7 -> 51.5; where two CTAs of an SM issue in turn (conv2_fwd_tc5,
// conv2_dx_tc5) nothing changes.
// Each descriptor is given as its two 32-bit halves: the high half (strides, version, layout) is a constant of the kernel and the low half
// is "start address / 16 + a compile-time offset", so that an unrolled issue loop costs one integer add per operand and MMA.
// BF16 / FP16 inputs: K = 16 per instruction; TF32: K = 8.  fp32 accumulation.
#define PSK_UMMA(NAME, KIND)                                                                                                       \
  __device__ __forceinline__ void NAME(uint32_t tmem_d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, \
                                       uint32_t accumulate) {                                                                      \
    asm volatile(                                                                                                                  \
        "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\t"                                                                           \
        "elect.sync _|q, 0xffffffff;\n\t"                                                                                          \
        "mov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\t"                                                                       \
        "setp.ne.b32 p, %6, 0;\n\t"                                                                                                \
        "@q tcgen05.mma.cta_group::1.kind::" KIND " [%0], da, db, %5, p;\n\t}"                                                     \
        ::"r"(tmem_d), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate) : "memory");                        \
  }
PSK_UMMA(umma_f16, "f16")
PSK_UMMA(umma_tf32, "tf32")
#undef PSK_UMMA

// Arrives on the barrier when the warp's MMAs so far are done.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar)) : "memory");
}
// A value that all lanes of the warp hold, in a form that shows it.
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}


// Plain bulk copy global -> shared (both 16-byte aligned, size a multiple of 16), completion on an mbarrier.
__device__ __forceinline__ void bulk_load(void* smem_dst, const void* gsrc, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(smem_dst)), "l"(gsrc), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// Plain bulk copy shared -> global (both 16-byte aligned, size a multiple of 16), tracked by the thread's bulk groups.
__device__ __forceinline__ void bulk_store(void* gdst, const void* smem_src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(smem_u32(smem_src)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// All of this thread's committed bulk copies have finished reading shared memory / have completed.
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Makes shared-memory writes of this thread (generic proxy) visible to the tensor core / TMA (async proxy).
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// The two halves of a shared-memory matrix descriptor without swizzle.  k contiguous: a core matrix is 8 rows of 16 bytes, stored
// contiguously (row pitch 16 bytes); `sbo` = byte distance between successive groups of 8 rows, `lbo` = byte distance between the two
// 16-byte k-chunks of one MMA.  Low = start address and leading byte offset, high = stride byte offset, version and layout type (0: no
// swizzle).  Adding n to the low half moves the start address by 16*n bytes.
__host__ __device__ constexpr uint32_t plain_desc_hi(uint32_t sbo) { return ((sbo >> 4) & 0x3FFF) | (1u << 14); }
__device__ __forceinline__ uint32_t plain_desc_lo(uint32_t addr, uint32_t lbo) {
  return ((addr & 0x3FFFF) >> 4) | (((lbo >> 4) & 0x3FFF) << 16);
}

// Host: tensor map of an fp32 tensor of `rank` dimensions (dims[0] contiguous; strides_bytes[i] = pitch of
// dimension i + 1), box as given, no swizzle, out-of-range elements read as zero.  False on failure.
bool encode_tensor_map_f32(CUtensorMap* m, const float* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes,
                           const uint32_t* box);
// The same of a BF16 tensor, with a swizzle of 64 or 128 bytes.
bool encode_tensor_map_bf16(CUtensorMap* m, const uint16_t* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes,
                            const uint32_t* box, int swizzle);

}  // namespace psk
