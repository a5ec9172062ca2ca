// Device-side helpers shared by the factorization and solve kernels:
// memory-model primitives for the task ring and dependency counters, and the
// control block layout.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace spchol {

// Control block (int32 words) of one persistent launch.
enum CtrlWord : int {
  kHead = 0,     // next ring slot to claim (the factorization's normal-priority ring)
  kTail = 1,     // next ring slot to fill
  kErr = 2,      // 0, or an SPCHOL_E* code (timeout, internal check)
  kInfo = 3,     // smallest failing pivot column + 1, INT32_MAX if none
  kWhere = 5,    // diagnostic: task id where a wait gave up
  kWarpNext = 6, // the next warp-level subtree task (FactorArgs::wsub; the solves' forward launch)
  kWarpNextB = 7, // the solves' backward launch's next warp-level subtree
  kHiHead = 32,  // the high-priority ring, in its own 128-byte line
  kHiTail = 33,
  kDone = 64,    // tasks completed, updated by every task, in a line of its own
  kFin = 96,     // 1 once a CTA has seen every task completed: the end test of the idle ones, in a line of its own
  kCtrlWords = 128
};

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Release and acquire by fences.  A signal -- a counter lowered, a ring slot
// filled -- is a relaxed operation after fence_gpu() of the same thread, and a
// thread that learns from one fences before it passes it on.  Measured on one
// SM (clocks): fence 555; atom relaxed 1150, eight in a row 1964; atom.acq_rel
// 1931, eight 12,048; eight st.release 6455, eight st.relaxed 540: acquiring
// or releasing operations wait for one another, relaxed ones overlap.
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void st_relaxed(int* p, int v) {
  asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int atom_add_relaxed(int* p, int v) {
  int old;
  asm volatile("atom.relaxed.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
// Lower a dependency counter; true for the thread that brought it to zero,
// which then has acquired what every other thread signalled with it.  The
// calling thread has fenced after the writes it signals.
__device__ __forceinline__ bool count_down(int* p) {
  if (atom_add_relaxed(p, -1) != 1) return false;
  fence_gpu();
  return true;
}
__device__ __forceinline__ int ld_relaxed(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Two adjacent words (8-byte aligned) in one load: x = p[0], y = p[1].
__device__ __forceinline__ int2 ld_relaxed_pair(const int* p) {
  int2 v;
  asm volatile("ld.relaxed.gpu.global.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// FP32 to FP64 on the integer pipe: a conversion instruction takes the FP64
// pipe as long as two multiply-adds (119 clocks per warp and sub-partition;
// this 34).  Normal numbers and zeros; the rest by the conversion.  For the
// solves, whose every product with an FP32 panel needs one: 27-point 48^3, two
// solves 6.9 -> 6.3 ms, 35 x 31 x 38 3.5 -> 2.9 ms.  (In the factorization,
// where a block is widened once, beside other work, it was 2 % slower.)
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x), u = b & 0x7fffffffu;
  if (u - 0x00800000u < 0x7f000000u)
    return __hiloint2double((int)((b & 0x80000000u) | ((u >> 3) + 0x38000000u)), (int)(b << 29));
  return u == 0 ? __hiloint2double((int)b, 0) : (double)x;
}
__device__ __forceinline__ double widen(double x) { return x; }

// Loads of data that other CTAs of the same launch may have written: served
// from L2, never from a possibly stale L1 line.
__device__ __forceinline__ double ldcg(const double* p) { return __ldcg(p); }
__device__ __forceinline__ float ldcg(const float* p) { return __ldcg(p); }
__device__ __forceinline__ int ldcg(const int* p) { return __ldcg(p); }

__device__ __forceinline__ void red_add(double* p, double v) { atomicAdd(p, v); }

// Copy the lower triangle of a w x w column-major block (leading dimension ld)
// into shared memory as double (ld w, zeros above the diagonal).  Each thread
// issues a batch of independent loads before it stores any of them, so the
// copy costs a few memory latencies instead of one per element.
template <bool kL2Only, typename T>
__device__ __forceinline__ void stage_lower(const T* __restrict__ src, int w, int ld, double* __restrict__ dst) {
  constexpr int B = 8;
  const int total = w * w, nt = blockDim.x;
  for (int base = threadIdx.x; base < total; base += B * nt) {
    double v[B];
#pragma unroll
    for (int u = 0; u < B; ++u) {
      const int idx = base + u * nt;
      const int i = idx % w, j = idx / w;
      v[u] = 0.0;
      if (idx < total && i >= j) {
        const T* p = src + i + (size_t)j * ld;
        v[u] = kL2Only ? (double)__ldcg(p) : (double)*p;
      }
    }
#pragma unroll
    for (int u = 0; u < B; ++u) {
      const int idx = base + u * nt;
      if (idx < total) dst[idx] = v[u];
    }
  }
}

// Raise a kernel's dynamic shared-memory limit to at least `need` bytes (host).
// The limit is a per-kernel setting shared by every handle of the process; it
// only ever grows, to the largest size any handle has needed, so a launch
// never finds it lowered by another handle.  (Raising it straight to the
// device maximum would lower the occupancy the runtime reports.)
cudaError_t ensure_smem_limit(const void* fn, size_t need);
__device__ __forceinline__ void red_add(float* p, float v) { atomicAdd(p, v); }

// An update value into its destination: an atomic add into a target panel
// that other tiles update too, or a plain store into a buffer that only this
// tile writes (the fan-in mode of the factorization).
template <typename T>
__device__ __forceinline__ void scatter_put(T* p, T v, bool store) {
  if (store)
    *p = v;
  else
    red_add(p, v);
}

}  // namespace spchol
