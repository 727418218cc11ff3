// tc_sm100.cuh -- the Blackwell (sm_100 family, built for sm_103a) primitives
// of the tensor-core kernels, as inline PTX: mbarriers with bounded waits,
// tiled TMA loads (cp.async.bulk.tensor), tensor-memory allocation, the
// 5th-generation MMA (tcgen05.mma, kind::tf32) with its shared-memory and
// instruction descriptors, and tensor-memory loads.
//
// Every wait is bounded by the global timer: a wait that has not completed
// after its limit returns false, and the caller records an error and leaves
// (after waiting, again bounded, for what it has in flight and freeing its
// tensor memory), so that no kernel of this library can spin forever.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace rpba {
namespace tc {

__device__ inline uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ inline uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ---------------------------------------------------------------------------
// mbarrier
// ---------------------------------------------------------------------------
__device__ inline void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// makes the initialised barriers visible to the async proxy (TMA, tcgen05)
__device__ inline void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ inline void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ inline bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// polls until done() or, false, until MBAR_POLLS polls and `limit_ns` nanoseconds
// are over: time alone also passes while the GPU runs another process
#define MBAR_POLLS 64
template <class F>
__device__ inline bool bounded_wait(uint64_t limit_ns, F done) {
  if (done()) return true;
  const uint64_t t0 = global_ns();
  for (uint32_t n = 1;; n++) {
    if (n >= MBAR_POLLS && global_ns() - t0 >= limit_ns) return false;
    if (done()) return true;
  }
}

// waits for the phase with the given parity to complete
__device__ inline bool mbar_wait(uint64_t *bar, uint32_t parity, uint64_t limit_ns) {
  return bounded_wait(limit_ns, [&] { return mbar_try_wait(bar, parity); });
}

// ---------------------------------------------------------------------------
// TMA: tiled 2-D load into shared memory, completion counted in bytes on an
// mbarrier. The inner coordinate x must make x * element size a multiple of
// 16 bytes (it is 0 in every use here).
// ---------------------------------------------------------------------------
__device__ inline void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

__device__ inline void prefetch_tmap(const CUtensorMap *map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)map) : "memory");
}

// ---------------------------------------------------------------------------
// tensor memory (TMEM): one warp allocates and frees; columns a power of 2 >= 32
// ---------------------------------------------------------------------------
__device__ inline void tmem_alloc(uint32_t *dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
}
__device__ inline void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ inline void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ inline void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ inline void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ---------------------------------------------------------------------------
// descriptors
// ---------------------------------------------------------------------------
// Shared-memory matrix descriptor of a K-major operand in the 128-byte
// swizzled layout that a TMA load with CU_TENSOR_MAP_SWIZZLE_128B writes:
// rows of 128 bytes, 8-row groups 1024 bytes apart (stride byte offset), the
// group base 1024-byte aligned. Fields: start address >> 4 (bits 0-13),
// leading byte offset >> 4 (16-29; unused by swizzled K-major layouts),
// stride byte offset >> 4 (32-45), the fixed value 1 (46-48), swizzle mode
// 2 = 128 B (61-63). The K position inside the 128-byte row is selected by
// advancing the start address.
__device__ inline uint64_t desc_sw128_kmajor(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Instruction descriptor of kind::tf32 with an FP32 accumulator, both
// operands K-major, no negation or sparsity: D format F32 (bits 4-5 = 1),
// A and B format TF32 (bits 7-9, 10-12 = 2), N >> 3 (bits 17-22), M >> 4
// (bits 24-28).
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// D[tmem] (+)= A[smem] * B[smem]^T, issued by one thread
__device__ inline void mma_tf32(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accum)
      : "memory");
}

// the mbarrier gets one arrival when every MMA this thread issued before has
// completed
__device__ inline void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// 32 consecutive FP32 columns of the calling lane's TMEM row (shape 32x32b,
// 32 repetitions): warp w reads lanes 32 w .. 32 w + 31, so taddr carries the
// lane offset 32 w in its upper 16 bits
__device__ inline void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; i++) v[i] = __uint_as_float(r[i]);
}

// ---------------------------------------------------------------------------
// splitting an FP32 value into TF32 pieces: the tensor core reads the top 19
// bits of each 32-bit operand (sign, exponent, 10 mantissa bits). hi keeps
// them with round-to-nearest; the remainder is exact in FP32.
// ---------------------------------------------------------------------------
__device__ inline float tf32_round(float x) {
  uint32_t u = __float_as_uint(x);
  if ((u & 0x7f800000u) == 0x7f800000u) return x;  // Inf / NaN unchanged
  u += 0x1000u;                                    // half of the dropped 13 bits
  u &= 0xffffe000u;
  return __uint_as_float(u);
}

}  // namespace tc
}  // namespace rpba
