// The FP32 decision rule of real-valued couplings (Eq. 4) and its shortcut, shared by the kernels
// that evaluate it:
//   x = b_t I, tau = tanh(x) (or the L-level staircase), delta = (tau + xi s) + eta_t z(key),
//   s' = +1 iff delta >= 0.
// The shortcut takes tanh from the hardware's approximation and the sign of its sum; where that
// sum lies within a margin of zero or is NaN (an infinite b_t times a zero field), settle_chunk
// evaluates the rule itself, so every decision is the rule's.  A NaN is no sum >= 0: the spin is -1.
#pragma once
#include <cmath>
#include <cstdint>

#include "philox.cuh"
#include "sm100_ptx.cuh"

namespace pim {

// Largest |tanh.approx(x) - tanhf(x)| on sm_103a: 7.99e-6 over every float, which a test measures (the
// documentation promises 2^-11 relative).
constexpr float kTanhGap = 8.0e-6f;

// Five times the gap, and the FP32 roundings of xi s + eta z and of the rule's own sums, each below
// 1e-6 (1 + xi) near zero.  A staircase goes by the rule alone.
__device__ __forceinline__ float rule_margin(int act, float xi) {
  return act == 0 ? 5.0f * kTanhGap + 4e-6f * (1.0f + fabsf(xi)) : INFINITY;
}

__device__ __forceinline__ float tanh_approx(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The lesser of two values, NaN if either is (fminf would drop it).
__device__ __forceinline__ float min_nan(float a, float b) {
  float y;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
  return y;
}

// The rule with tanh for the spins of a chunk (W spins from Philox block blk0 on) that the shortcut
// leaves open, |g| <= margin or NaN: g = +1 or -1 from x = b I and the old spins ob.  Out of line: the
// common path keeps its registers.
template <int W>
__device__ __noinline__ void tanh_chunk(float* g, const float* x, uint32_t blk0, uint32_t r, uint32_t t,
                                        uint32_t q, const uint32_t* rk, uint32_t ob, float margin, float xi,
                                        float eta, const float* sZ) {
#pragma unroll
  for (int b = 0; b < W / 8; ++b) {
    const PhiloxOut o = philox4x32_10_rk(blk0 + b, r, t, q, rk);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int e = 8 * b + k;
      if (!(fabsf(g[e]) > margin)) {
        const float z = sZ[philox_half(o, k) >> 4];
        const float a = __fadd_rn(tanhf(x[e]), ((ob >> e) & 1u) ? xi : -xi);
        g[e] = __fadd_rn(a, __fmul_rn(eta, z)) >= 0.0f ? 1.0f : -1.0f;
      }
    }
  }
}

// The rule with the staircase for every spin of a chunk.
template <int W>
__device__ __noinline__ void stairs_chunk(float* g, const float* x, uint32_t blk0, uint32_t r, uint32_t t,
                                          uint32_t q, const uint32_t* rk, uint32_t ob, float xi, float eta,
                                          int levels, const float* sZ) {
#pragma unroll
  for (int b = 0; b < W / 8; ++b) {
    const PhiloxOut o = philox4x32_10_rk(blk0 + b, r, t, q, rk);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int e = 8 * b + k;
      const float z = sZ[philox_half(o, k) >> 4];
      const float a = __fadd_rn(staircase(x[e], levels), ((ob >> e) & 1u) ? xi : -xi);
      g[e] = __fadd_rn(a, __fmul_rn(eta, z)) >= 0.0f ? 1.0f : -1.0f;
    }
  }
}

// Decides again the spins of a chunk that the shortcut leaves open (some lane has a g that is not
// beyond the margin; with a staircase all of them).
template <int W>
__device__ __forceinline__ void settle_chunk(float (&g)[W], const float (&x)[W], uint32_t blk0, uint32_t r,
                                             uint32_t t, uint32_t q, const uint32_t* rk, uint32_t ob,
                                             float margin, float xi, float eta, int act, int levels,
                                             const float* sZ) {
  float gm[W], xm[W];
#pragma unroll
  for (int e = 0; e < W; ++e) gm[e] = g[e], xm[e] = x[e];
  if (act == 0)
    tanh_chunk<W>(gm, xm, blk0, r, t, q, rk, ob, margin, xi, eta, sZ);
  else
    stairs_chunk<W>(gm, xm, blk0, r, t, q, rk, ob, xi, eta, levels, sZ);
#pragma unroll
  for (int e = 0; e < W; ++e) g[e] = gm[e];
}

}  // namespace pim
