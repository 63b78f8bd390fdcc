// Operand splitting and small tcgen05 helpers of the joint form's tensor-core kernels
// (joint_planes.cu, joint_core.cu).
#pragma once

#include <cuda_fp16.h>

#include "joint.cuh"
#include "stage.cuh"

namespace zbc {
namespace {

constexpr int kBasisShift = 10;  // basis entries (|b| <= 1) are scaled by 2^10
constexpr int kDataShift = 10;   // the other operand is brought below 2^10

// fp16 hi / lo of a scaled pair, as words (x low)
__device__ __forceinline__ void split2(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x, y);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(x - f.x, y - f.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// e with m < 2^e, at least `least` so that the scales made from it are normal floats (0 for zero and for
// values that are not finite, which go through unscaled)
__device__ __forceinline__ int exp_of(float m, int least) {
  if (!(m > 0.f) || !(m < INFINITY)) return 0;
  return max(least, (int)(__float_as_uint(m) >> 23) - 126);
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }  // -126 .. 127
// order of a chunk's 32 summed entries in a 128-byte row: entry of word w of the 16-byte chunk c, so
// that lane c's entries are two adjacent pairs and 8 lanes read 128 bytes without a gap
__host__ __device__ constexpr int entry_of(int c, int w) { return 2 * c + (w & 1) + 16 * (w >> 1); }
// max(|a|, |b|, |c|), NaN if any is
__device__ __forceinline__ float absmax_nan(float a, float b, float c) {
  float r;
  asm("{\n\t.reg .f32 t, u, v;\n\tabs.f32 t, %2;\n\tabs.f32 u, %3;\n\tmax.NaN.f32 v, t, u;\n\tmax.NaN.f32 %0, %1, v;\n\t}"
      : "=f"(r)
      : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// Tensor cores round their accumulators toward zero (Fasi, Higham, Mikaitis, Pranesh, "Numerical behavior
// of NVIDIA tensor cores", 2021), which takes a part off every sum that does not average out.  Its mean is put
// back with the scales.  One rounding takes half a unit of 2^-23 off a mantissa m in [1, 2), relatively
// 2^-24 E[1/m] = 2^-24 / (2 ln 2) = 4.3e-8 for mantissas spread evenly over their logarithm, and the partial
// sum after step s of S is s/S of the whole in the mean.  96^3 head coil, 16 right-hand sides: with lo terms
// first everywhere and nothing put back, the mean (signed) errors of the forward and the adjoint are -4.4e-7
// and -2.0e-7; as it is, within 1e-7.
//  - lo terms first, onto an accumulator of their own size; the hi hi terms alone round the full sum:
__host__ __device__ constexpr float lo_first_gain(int steps) { return 1.f + 4.3e-8f * (0.5f * (float)(steps + 1)); }
//  - lo and hi terms of a step together, which lets consecutive MMAs share an operand (the forward's
//    planes, 160 x 160 x 128 with 32 right-hand sides: 0.697 ms, lo first 0.718): two more additions onto
//    the sum before the step, each of small terms and measured at 3/4 of a rounding.  Two such chains:
__host__ __device__ constexpr float mixed_gain(int s1, int s2) {
  return 1.f + 4.3e-8f * (0.5f * (float)(s1 + 1 + s2 + 1) + 0.75f * (float)(s1 - 1 + s2 - 1));
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\t"
               "tcgen05.wait::ld.sync.aligned;"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

// the adjoint's eight worker warps and a ninth that issues the MMAs: an issue occupies its thread for
// about 100 cycles, and a worker that did it held the others up at the next barrier (2.34 -> 1.80 ms,
// 320 x 320 x 256, 8 right-hand sides)
constexpr int kThreads = 288;
__device__ __forceinline__ void worker_barrier() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
// a warp's shared-memory writes, visible to the MMAs of whoever waits on `bar`
__device__ __forceinline__ void warp_publish(uint64_t* bar) {
  tc::fence_proxy_async();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive1(bar);
}

// The bounded waits of a kernel: once one gave up (after `polls` tries of about a microsecond) its thread waits no
// more; the barriers are still passed, and the thread that issues the MMAs ends with drain2() / drain1().
struct Waits {
  int* err;
  uint32_t polls;
  bool ok = true;
  __device__ void one(uint64_t* bar, uint32_t parity) {
    if (ok && !tc::mbar_wait_idle(bar, parity, polls)) {
      ok = false;
      atomicOr(err, kErrTimeout);
    }
  }
  // by all lanes of a warp, each of which may give up by itself: what needs the whole warp after it (tcgen05.ld)
  // is run whatever `ok` says, and only what a lane does alone asks for it
  __device__ void warp(uint64_t* bar, uint32_t parity) {
    one(bar, parity);
    __syncwarp();
  }
};
// The n-th commit (from 1) to a pair of barriers, or to one, has completed: whatever was issued no longer reads
// shared memory or writes tensor memory when the CTA gives them up.
__device__ __forceinline__ void drain2(uint64_t* bar, int n) {
  if (n > 0) tc::mbar_wait_idle(bar + ((n - 1) & 1), ((n - 1) >> 1) & 1);
}
__device__ __forceinline__ void drain1(uint64_t* bar, int n) {
  if (n > 0) tc::mbar_wait_idle(bar, (n - 1) & 1);
}

}  // namespace
}  // namespace zbc
