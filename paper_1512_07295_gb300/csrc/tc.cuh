// tcgen05 building blocks (sm_100 family, inline PTX) shared by the tensor-core kernels: FP32 values
// split into two TF32 parts, shared-memory matrix descriptors of K-major operands without swizzle,
// the kind::tf32 instruction descriptor, bounded mbarrier waits, TMEM allocation, MMA issue, commit
// and the 32x32b loads and stores of TMEM (A operands, accumulators with compensated sums in registers).
//
// Operand layout (K-major, no swizzle): core matrices of 8 rows x 16 bytes (4 TF32 values along K),
// rows 16 B apart inside a core matrix; K-adjacent core matrices LBO = 128 B apart, 8-row groups
// SBO = (K per stage / 4) x 128 B apart. One MMA k-step (K = 8) covers two K-adjacent core matrices.
#pragma once

#include <stdint.h>

namespace pk {
namespace tc {

// x = big + small: big is x rounded to TF32 (ties away from zero), small = x - big is exact in FP32.
// Three products big.big + big.small + small.big then err by about 3 x 2^-22 of |a b|.
__device__ __forceinline__ void split(float x, float& big, float& small) {
  big = __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
  small = x - big;
}

// Byte offset of element (row, k) in a K-major operand holding kk values of K per row.
__device__ __forceinline__ uint32_t off(int row, int k, int kk) {
  return uint32_t(((row >> 3) * (kk / 4) + (k >> 2)) * 128 + (row & 7) * 16 + (k & 3) * 4);
}

// Shared-memory descriptor: start address, LBO = 128 B, SBO, version 1 (sm_100 family), no swizzle.
// A k-step advances the start address by 256 B, i.e. adds 16 to the descriptor.
__device__ __forceinline__ uint64_t desc(uint32_t saddr, uint32_t sbo) {
  return uint64_t((saddr >> 4) & 0x3FFF) | (uint64_t((128u >> 4) & 0x3FFF) << 16) | (uint64_t((sbo >> 4) & 0x3FFF) << 32) |
         (uint64_t(1) << 46);
}

// kind::tf32 instruction descriptor: FP32 accumulator, TF32 A and B, both K-major, N and M.
__host__ __device__ constexpr uint32_t idesc_tf32(int n, int m) {
  return (1u << 4) | (2u << 7) | (2u << 10) | (uint32_t(n >> 3) << 17) | (uint32_t(m >> 4) << 24);
}

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ bool try_wait(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
// Waits for the phase of the given parity of the mbarrier at shared address bar, at most limit_ns, and
// gives up early when another wait of the block has (*stop, if given). The timer is read only once the
// first polls, which cover the ordinary case, have found the phase open.
__device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity, uint64_t limit_ns, const volatile int* stop) {
  for (int i = 0; i < 64; ++i)
    if (try_wait(bar, parity)) return true;
  const uint64_t t0 = now_ns();
  for (;;) {
    if (try_wait(bar, parity)) return true;
    if (now_ns() - t0 > limit_ns || (stop && *stop)) return false;
  }
}

// Bulk copy of bytes (a multiple of 16; both addresses 16-byte aligned) from global to shared memory,
// completing on the mbarrier at bar.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
               "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Registers per thread of the calling warpgroup from here on (all four of its warps call it).
template <int N>
__device__ __forceinline__ void regs_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void regs_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Warp-wide: allocates ncols TMEM columns, the address written to shared memory at slot.
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// D (TMEM) = A B (+ D when accumulate), A in TMEM (row = lane, one column per K value), B in shared
// memory; single issuing thread.
__device__ __forceinline__ void mma_tf32_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Four consecutive columns of this warp's 32 TMEM lanes from registers; wait_st before they are used.
__device__ __forceinline__ void store4(uint32_t taddr, const float (&v)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3])
               : "memory");
}
__device__ __forceinline__ void wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// The mbarrier at bar completes a phase when every MMA issued so far by this thread has completed.
__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ uint64_t pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// N consecutive accumulator columns of this warp's 32 TMEM lanes, added to the compensated sums (value s,
// compensation c, two columns per 64-bit register) by TwoSum, which keeps the rounding of s + v whichever of the two is
// larger: t = s + v, b = t - s, c += (s - (t - b)) + (v - b), s = t; the total is s + c. (Kahan's
// summation, four operations instead of seven, loses the small running sum when a large total arrives: weights of
// both signs. 64^3 particles on N = 64: 1.58 against 1.48 ms per call.) Differences as fma(b, -1, a), which
// rounds a - b once.
template <int N>
__device__ __forceinline__ void twosum_acc(uint32_t taddr, uint64_t (&s)[N / 2], uint64_t (&c)[N / 2]) {
  static_assert(N % 8 == 0, "columns are read in eights");
  const uint64_t m1 = pack(-1.0f, -1.0f);
  auto add = [](uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
  };
  auto sub = [m1](uint64_t a, uint64_t b) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(b), "l"(m1), "l"(a));
    return r;
  };
#pragma unroll
  for (int g = 0; g < N / 8; ++g) {
    float v[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "r"(taddr + 8 * g)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint64_t& ss = s[4 * g + j];
      uint64_t& cc = c[4 * g + j];
      const uint64_t x = pack(v[2 * j], v[2 * j + 1]);
      const uint64_t t = add(ss, x), b = sub(t, ss);
      cc = add(cc, add(sub(ss, sub(t, b)), sub(x, b)));
      ss = t;
    }
  }
}

}  // namespace tc
}  // namespace pk
