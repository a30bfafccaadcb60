// The integer decision rule (Eq. 2 and 4) on a chunk of W spins of one replica: fields from tensor
// memory as exactly integral FP32 values, 16-bit draws, and a threshold per (spin, field) from a
// step's table in shared memory.  Used by the fused, latency and mid-N kernels.
//
// The chunk costs issue slots and two of the pipes: the Philox products fill the one FP32/integer
// pipe that runs integer multiply-adds, the shifts and logic fill the other integer pipe.  So what
// can be is done in FP32 arithmetic, which both FP32 pipes run: an integer below 2^23 is the subnormal
// float of the same bits, multiply-adds on those are exact, and subnormals run at full rate.  Against
// integer arithmetic, us per sweep of runs of 100 (with a bias) to 1000 sweeps, launch included: SK
// N = 200, 100 instances x 1024 replicas 13.14 -> 12.85 (12.3 over 2000 sweeps), Max-Cut N = 100, 100 x
// 1024 7.19 -> 6.84, one SK N = 200 x 128 1.48 -> 1.36; with a bias N = 256, 200 x 256 19.0 -> 13.4,
// N = 400, 80 x 256 30.2 -> 17.1 (16.7 with two spin images).
#pragma once
#include <cstdint>

namespace pim {

// An integer D, |D| < 2^22, held exactly in FP32 stands in the low mantissa bits of D + kMagic.
constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
constexpr uint32_t kMagicBits = 0x4B400000u;

// Shared-memory addresses of the 16-bit table entries of two exactly integral fields: base + 2 D.
__device__ __forceinline__ void entry_address2(uint32_t d0, uint32_t d1, uint32_t base, uint32_t& a0,
                                               uint32_t& a1) {
  uint64_t d, b, r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(d0), "r"(d1));
  asm("mov.b64 %0, {%1, %1};" : "=l"(b) : "r"(base));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(d), "l"(0x0000000200000002ull), "l"(b));
  asm("mov.b64 {%0, %1}, %2;" : "=r"(a0), "=r"(a1) : "l"(r));
}

// Word whose sign bit says that the 16-bit draw lies below 16 x threshold (threshold <= 4096), that is
// that the draw's 12-bit key lies below the threshold and the new spin is -1.  Every other spin of a
// chunk takes the FP32 form, which shares the work between the pipes: SK N = 200, 100 x 1024, 12.88 us
// per sweep all FP32, 12.69 none, 12.85 half; Max-Cut N = 100 6.90, 6.98, 6.84; one instance of N = 200
// x 128 1.365, 1.377, 1.365.
__device__ __forceinline__ uint32_t draw_below(uint32_t draw, uint32_t threshold, bool fp) {
  return fp ? __float_as_uint(__fmaf_rn(__uint_as_float(threshold), -16.0f, __uint_as_float(draw)))
            : draw - 16u * threshold;
}

__device__ __forceinline__ uint32_t table_entry(uint32_t at) {
  uint32_t m;
  asm volatile("ld.shared.u16 %0, [%1];" : "=r"(m) : "r"(at));
  return m;
}

// Draw of spin e of the chunk: two per Philox word.
__device__ __forceinline__ uint32_t draw_of(const uint32_t* rw, int e) {
  return (e & 1) ? (rw[e >> 1] >> 16) : (rw[e >> 1] & 0xFFFFu);
}

// Diagonal-encoded couplings: D = I + dk s with |I| < dk, no bias.  The threshold of (s, I) is the
// 16-bit entry of D, at shared address base + 2 D, and |D| = s I + dk sums into esum.  Returns the new
// spins as bits.  decide = false: the energy only.
template <int W>
__device__ __forceinline__ uint32_t diag_rule(const uint32_t (&v)[W], const uint32_t* rw, uint32_t base,
                                              float& esum, bool decide = true) {
  // The sign bits are shifted in from the top; two shift chains from 16 spins on and two energy sums
  // keep the dependent sequences short.
  uint32_t neg_hi = 0, neg_lo = 0, at_pair = 0;
  float e_a = 0.0f, e_b = 0.0f;
#pragma unroll
  for (int e = W - 1; e >= 0; --e) {
    if (decide) {
      uint32_t at = at_pair;
      if (e & 1) entry_address2(v[e - 1], v[e], base, at_pair, at);
      const uint32_t below = draw_below(draw_of(rw, e), table_entry(at), e & 1);
      if (W > 8 && e >= W / 2)
        neg_hi = __funnelshift_l(below, neg_hi, 1);
      else
        neg_lo = __funnelshift_l(below, neg_lo, 1);
    }
    if (e & 1)
      e_a += fabsf(__uint_as_float(v[e]));
    else
      e_b += fabsf(__uint_as_float(v[e]));
  }
  esum += e_a + e_b;
  return ~((neg_hi << (W / 2)) | neg_lo) & ((1u << W) - 1u);
}

// Plain couplings with a bias: I = D + h (h: the chunk's W values in shared memory, on 16 bytes).  The
// threshold of (s, I) is the 16-bit entry at shared address base + 4 I + 2 s (s = 0 or 1, bit e of
// `bits`); sum_i s_i (I_i + h_i) goes into esum: at most 16 terms below 2^13 here, exact.
template <int W>
__device__ __forceinline__ uint32_t bias_rule(const uint32_t (&v)[W], const uint32_t* rw, uint32_t bits,
                                              const float* h, uint32_t base, float& esum,
                                              bool decide = true) {
  uint32_t neg_hi = 0, neg_lo = 0;
  float e_a = 0.0f, e_b = 0.0f;
  float hv[W];
#pragma unroll
  for (int e = 0; e < W; e += 4) {
    const float4 x = *reinterpret_cast<const float4*>(h + e);
    hv[e] = x.x, hv[e + 1] = x.y, hv[e + 2] = x.z, hv[e + 3] = x.w;
  }
#pragma unroll
  for (int e = W - 1; e >= 0; --e) {
    const float field = __uint_as_float(v[e]) + hv[e];
    const uint32_t top = bits << (31 - e);  // s in the sign bit
    const float term = __uint_as_float(__float_as_uint(field + hv[e]) ^ (top & 0x80000000u));  // -s (I + h)
    if (e & 1)
      e_a += term;
    else
      e_b += term;
    if (decide) {
      const float at = __fmaf_rn(field, __uint_as_float(4u), __uint_as_float(base));
      const uint32_t at_s = __float_as_uint(__fmaf_rn(__uint_as_float(top >> 31), 2.0f, at));
      const uint32_t below = draw_below(draw_of(rw, e), table_entry(at_s), e & 1);
      if (W > 8 && e >= W / 2)
        neg_hi = __funnelshift_l(below, neg_hi, 1);
      else
        neg_lo = __funnelshift_l(below, neg_lo, 1);
    }
  }
  esum -= e_a + e_b;
  return ~((neg_hi << (W / 2)) | neg_lo) & ((1u << W) - 1u);
}

}  // namespace pim
