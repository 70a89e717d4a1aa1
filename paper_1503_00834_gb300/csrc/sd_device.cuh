// Device helpers of the spectral-difference kernels: bulk-copy / mbarrier primitives, index and layout
// helpers.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace chorus {

// ------------------------------------------------------------------ async-copy helpers

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}

// 1D bulk copy global -> shared, completion signalled on the mbarrier (byte count).
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// Bulk prefetch into L2 of the 16-byte units that lie wholly in [p, p + bytes).
__device__ __forceinline__ void prefetch_l2(const void* p, size_t bytes) {
  const uintptr_t a = ((uintptr_t)p + 15) & ~(uintptr_t)15, b = ((uintptr_t)p + bytes) & ~(uintptr_t)15;
  if (b > a) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((uint32_t)(b - a)) : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Programmatic dependent launch: let the next kernel of the stream start; wait until the kernel before it
// has completed (both do nothing in a launch without the attribute).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Load of a value that another kernel, or another phase of the same launch, has written since this kernel
// started.  __ldg is for data that no one writes while the kernel runs: the compiler may move it above
// pdl_wait or a grid barrier, and its cache line may be stale.  The volatile asm keeps its place.
__device__ __forceinline__ float ld_written(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ int ld_written(const int* p) {
  int v;
  asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double ld_written(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}

// Polls of a bounded mbarrier wait when the mesh sets no limit of its own (about a second with the
// back-off below).
constexpr uint32_t kDefaultWaitPolls = 1u << 24;

// Bounded wait for the completion of the barrier's phase of the given parity (0 for a barrier's first
// use): at most `polls` polls.  Returns false if they ran out.
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity, uint32_t polls) {
  const uint32_t a = smem_addr(bar);
  for (uint32_t it = 0; it < polls; ++it) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.b32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
    if (it > 64) __nanosleep(64);
  }
  return false;
}

// The device control block of a mesh: err[0] error flags, err[1] the wait limit (0: the default,
// k + 1: k polls).  Returns the number of polls of a kernel's staging waits.
__device__ __forceinline__ uint32_t wait_polls(const unsigned* err) {
  if (err == nullptr) return kDefaultWaitPolls;
  const uint32_t lim = *(const volatile unsigned*)(err + 1);
  return lim == 0u ? kDefaultWaitPolls : lim - 1u;
}

// Bounded wait for the bulk copies of a staging barrier.  If `polls` run out, sets bit 0 of *err
// and waits once more (default limit) for the copies still in flight, so that no copy writes into
// the shared memory of a CTA that has given up; returns false.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, unsigned* err, uint32_t polls) {
  if (mbar_try(bar, parity, polls)) return true;
  if (err) atomicOr(err, 1u);
  mbar_try(bar, parity, kDefaultWaitPolls);
  return false;
}

// One rounding, in the operands' own type.
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// ------------------------------------------------------------------ index helpers

// neighbour face-point index of own face point t under the orientation bits (swap, flip1, flip2)
template <int N>
__device__ __forceinline__ int map_face_pt(int t, int orient) {
  const int t1 = t % N, t2 = t / N;
  int a = (orient & 4) ? t2 : t1;
  int b = (orient & 4) ? t1 : t2;
  if (orient & 2) a = N - 1 - a;
  if (orient & 1) b = N - 1 - b;
  return a + N * b;
}

// ------------------------------------------------------------------ layout helpers

// Count of R words padded to a multiple of 16 bytes whose byte size is 64 mod 128.
template <class R>
constexpr int pad_stride(int count) {
  int bytes = (count * (int)sizeof(R) + 15) / 16 * 16;
  const int r = bytes % 128;
  bytes += (64 - r + 128) % 128;
  return bytes / (int)sizeof(R);
}

// Shared-memory index of solution point (i,j,k) within one component array of the computed arrays.
template <int N, class R>
__device__ __forceinline__ int sidx(int i, int j, int k) {
  if (N == 4 && sizeof(R) == 4) return i + 4 * ((j ^ k) & 3) + 16 * k;
  return i + N * j + N * N * k;
}

// (i,j,k) of position s on line ln of direction D
template <int N, int D>
__device__ __forceinline__ void line_ijk(int ln, int s, int& i, int& j, int& k) {
  const int a = ln % N, b = ln / N;
  if (D == 0) {
    i = s; j = a; k = b;
  } else if (D == 1) {
    i = a; j = s; k = b;
  } else {
    i = a; j = b; k = s;
  }
}

template <int N, int D>
__device__ __forceinline__ int line_pt(int ln, int s) {
  int i, j, k;
  line_ijk<N, D>(ln, s, i, j, k);
  return i + N * j + N * N * k;
}

template <int N, int D, class R>
__device__ __forceinline__ int line_sidx(int ln, int s) {
  int i, j, k;
  line_ijk<N, D>(ln, s, i, j, k);
  return sidx<N, R>(i, j, k);
}

// Index of position s along line ln of direction D in the background tables' point order.
template <int N, int D, class R>
__device__ __forceinline__ int line_bg(int ln, int s) {
  if constexpr (bg_swizzle(N) && sizeof(R) == 4) return line_sidx<N, D, R>(ln, s);
  else return line_pt<N, D>(ln, s);
}

template <int N, int EPB>
__host__ __device__ constexpr int warps_per_cta() { return (EPB * N * N + 31) / 32; }

}  // namespace chorus
