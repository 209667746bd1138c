// Thin wrappers over the fifth-generation tensor core instructions (tcgen05)
// used by the network kernels: BF16 operands in shared memory without
// swizzling, FP32 accumulators in tensor memory (TMEM).
//
// Operand layout. Both operands are stored as [chunk][row][8] BF16: a chunk
// is 8 values of 16 bytes, consecutive rows are 16 bytes apart, chunks are a
// plane apart. This one layout serves as
//  - K-major operand (rows = M or N, chunks along K): the 8-row groups are
//    128 bytes apart, the K chunks a plane apart;
//  - MN-major operand (chunks = M or N, rows along K): the M/N chunks are a
//    plane apart, the 8-row K groups 128 bytes apart.
// Rows are equally spaced, so a convolution tap is only another start address
// (16 bytes per pixel), and the distance of two K chunks may just as well be
// the distance of two taps.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace umma {

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Descriptor of an operand at shared address `addr`: `lead` and `stride` are
// the leading- and stride-dimension byte offsets, no swizzle.
__device__ __forceinline__ uint64_t desc(uint32_t addr, uint32_t lead, uint32_t stride) {
  return (uint64_t)((addr >> 4) & 0x3fff) | ((uint64_t)((lead >> 4) & 0x3fff) << 16) |
         ((uint64_t)((stride >> 4) & 0x3fff) << 32) | (1ull << 46);
}
// K-major: 8-row groups 128 bytes apart, K chunks `chunk` bytes apart.
__device__ __forceinline__ uint64_t desc_k(uint32_t addr, uint32_t chunk) { return desc(addr, chunk, 128); }
// MN-major: M/N chunks `chunk` bytes apart, 8-row K groups 128 bytes apart.
__device__ __forceinline__ uint64_t desc_mn(uint32_t addr, uint32_t chunk) { return desc(addr, 128, chunk); }

// Instruction descriptor: BF16 x BF16 -> FP32, both operands K-major or both MN-major.
constexpr uint32_t idesc(int m, int n, bool mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn_major ? (3u << 15) : 0u) | ((uint32_t)(n / 8) << 17) |
         ((uint32_t)(m / 16) << 24);
}

// D (TMEM) (+)= A B for one K = 16 step; one thread issues it.
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t id, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"((uint32_t)accumulate)
      : "memory");
}
// One lane of a converged warp. The MMA's operands live in uniform registers:
// behind `lane == 0` they are moved there one by one (244 cycles per MMA
// measured), behind this election the compiler knows the warp is uniform.
__device__ __forceinline__ bool elect() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0;
}
// The barrier completes once all MMAs issued so far by this thread have.
__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}

// TMEM columns (a power of two >= 32), by one whole warp; the address lands in *slot (shared memory).
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols));
}
// 16 (8) columns of the warp's 32 lanes (warp w of its warpgroup reads lanes 32 w ..): lane in bits 16.. of addr.
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld8(uint32_t addr, float* v) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\ttcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(addr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Shared-memory writes of this thread become visible to the tensor core.
__device__ __forceinline__ void fence_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void bar_init(uint64_t* bar, uint32_t count = 1) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t* bar) {
  asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.shared::cta.b64 t, [%0];\n\t}" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void bar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

constexpr uint32_t WAIT_NS = 1000000000;  // limit of a wait: a second
__device__ __forceinline__ unsigned long long clock_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool bar_try(uint32_t bar, uint32_t phase) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(bar), "r"(phase)
      : "memory");
  return __all_sync(0xffffffffu, done);
}
// Waits for a barrier phase, for `limit` ns of the global timer (read every 16
// attempts); false if it did not complete, and at once for a limit of 0. Whole
// warps call it.
__device__ __forceinline__ bool bar_wait(uint64_t* bar, uint32_t phase, uint32_t limit) {
  if (limit == 0) return false;
  const uint32_t a = smem_addr(bar);
  unsigned long long t0 = 0;
#pragma unroll 1
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 16; ++i)
      if (bar_try(a, phase)) return true;
    const unsigned long long t = __shfl_sync(0xffffffffu, clock_ns(), 0);
    if (t0 == 0) t0 = t;
    else if (t - t0 > limit) return false;
  }
}
// After a wait that ran out: the warp that issued MMAs waits for them all, so
// that their operands and accumulators may be written and freed. `bar` is a
// barrier of its own, in its first phase.
__device__ __forceinline__ void drain(uint64_t* bar) {
  if (elect()) commit(bar);
  __syncwarp();
  bar_wait(bar, 0, WAIT_NS);
}

// x as a sum of three BF16 values (exact: 24 significant bits in pieces of 8,
// each cut towards zero; an infinity keeps zero lower pieces), for pairs.
__device__ __forceinline__ void split2(float x, float y, uint32_t* hi, uint32_t* mid, uint32_t* lo) {
  const uint32_t M = 0xffff0000u, INF2 = 0xff000000u;
  const uint32_t ux = __float_as_uint(x), uy = __float_as_uint(y);
  // a NaN stays one whatever its payload
  const uint32_t hx = (ux & M) | ((ux << 1) > INF2 ? 0x00400000u : 0u);
  const uint32_t hy = (uy & M) | ((uy << 1) > INF2 ? 0x00400000u : 0u);
  const float rx = (ux << 1) >= INF2 ? 0.0f : x - __uint_as_float(hx);
  const float ry = (uy << 1) >= INF2 ? 0.0f : y - __uint_as_float(hy);
  const uint32_t mx = __float_as_uint(rx) & M, my = __float_as_uint(ry) & M;
  const uint32_t lx = __float_as_uint(rx - __uint_as_float(mx)), ly = __float_as_uint(ry - __uint_as_float(my));
  *hi = __byte_perm(hx, hy, 0x7632);
  *mid = __byte_perm(mx, my, 0x7632);
  *lo = __byte_perm(lx, ly, 0x7632);
}
// 8 values as the three pieces' 16-byte chunks.
__device__ __forceinline__ void split8(const float* v, uint4* p) {
  uint32_t h[4], m[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) split2(v[2 * i], v[2 * i + 1], h + i, m + i, l + i);
  p[0] = make_uint4(h[0], h[1], h[2], h[3]);
  p[1] = make_uint4(m[0], m[1], m[2], m[3]);
  p[2] = make_uint4(l[0], l[1], l[2], l[3]);
}

}  // namespace umma
