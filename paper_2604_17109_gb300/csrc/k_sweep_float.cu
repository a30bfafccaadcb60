// Fused PIMI sweep kernel for real-valued couplings (n <= 256): BF16 operands on the
// tcgen05 tensor path (kind::f16, FP32 accumulation), decision in FP32.
//
// One CTA = one instance x a tile of 32, 64 or 128 replicas, all sweeps inside.  What it
// computes per sweep:
//   operands  A = spins as BF16 +-1 (exact), B = J rounded to BF16, both K-major with the
//             128-byte swizzle; K advances 16 elements (32 bytes) per MMA.
//   decision  Eq. 4: x = b_t (I + h), tau = tanh(x) (or the L-level staircase of Algorithm
//             "LUT-based tanh approximation"), delta = (tau + xi s) + eta_t z(key),
//             s' = +1 iff delta >= 0, in FP32, with the same Philox draws and 4096 noise
//             levels as the integer path.
//   energy    H = -1/2 sum_i s_i (I_i + h_i), summed in FP32 column by column over each half
//             of the spins.
//
// The sweep is a chain of dependent steps (MMA, decision, spin write-back, MMA), and a
// serving batch puts few replicas on few SMs, so the kernel is bound by the length of that
// chain, not by any unit's rate.  The layout shortens it:
//  - TMEM lane = replica, and a warp can only read the 32 lanes of its quadrant.  A tile of
//    32 replicas is therefore written into all four lane quadrants of the A operand (64: into
//    two each), so that every quadrant's warps hold the fields of every replica and the
//    columns of one replica are split over 4x as many threads: CAP / W decision warps, each
//    thread one replica and rows / 32 chunks of W spins.
//  - Roles run in their own warps: decision warps, energy warps (one per 32 replicas and half
//    of the columns) and one MMA warp, coupled by mbarriers; two accumulators, so that the
//    energy of s(t) is summed while s(t+1) is decided and multiplied.
//  - The noise is drawn while the MMAs run.
//  - tanh is the hardware's approximation first: where the sum it gives lies within a margin of
//    zero, the decision is taken by the rule above instead (about one spin in 30 000), so every
//    decision is the rule's own.
// Measured (GB300, us per sweep) against 128-lane tiles with the rule unrolled for every column
// of one thread, which was bound by instruction fetch:
//   1 instance x 32 replicas      n = 64  7.94 -> 0.97   n = 128  28.3 -> 1.68   n = 256  37.9 -> 3.26
//   152 instances x 128 replicas  n = 64  8.39 -> 2.67   n = 256  38.1 -> 9.1 (5.5e11 spin updates/s)
// Fixed-point datapath (P.fix_w > 0, n <= 128): the couplings are Q(c J) in
// ap_fixed<W, W - F> (supplementary quantization section), held as two BF16 images whose sum
// is exact (high part + low part), so the two MMA chains give the exact field I in FP32
// (|I| 2^F < 2^24).  The decision then follows the datapath on integers in units of 2^-F:
//   u = sat(I), x = Q(fl32(beta_t) u), tau = table(x), a = sat(tau + s Q(xi)),
//   n = sat(trunc(Q(eta_t) Q(z) / 2^F)), s' = +1 iff sat(a + n) >= 0,
// and the energy is summed exactly in integers.
#include <cfloat>

#include "kernels.h"
#include "philox.cuh"
#include "real_rule.cuh"
#include "sm100_ptx.cuh"

namespace pim {
namespace {

enum FloatMode : int { kPlain = 0, kServing = 1, kFixedPoint = 2 };

constexpr int kTileM = 128;

// Fixed-point decision of one spin (see the header): integers in units of 2^-F.
__device__ __forceinline__ uint32_t fixed_decide(float I, uint32_t s, float beta, int eta_q,
                                                 int z_q, int xi_q, int F, int half_range,
                                                 const int32_t* __restrict__ tau_tab) {
  const int lo = -half_range, hi = half_range - 1;
  const int mI = __float2int_rz(__fmul_rn(I, __int_as_float((127 + F) << 23)));  // I 2^F, exact
  const int mu = min(max(mI, lo), hi);
  // Q(beta u): the product of a 24-bit and a 16-bit integer is exact in double
  long long mx = static_cast<long long>(__dmul_rn(static_cast<double>(beta), static_cast<double>(mu)));
  mx = mx < lo ? lo : (mx > hi ? hi : mx);
  const int mt = __ldg(tau_tab + (mx + half_range));
  const int ma = min(max(mt + (s ? xi_q : -xi_q), lo), hi);
  const int mn = min(max((eta_q * z_q) / (1 << F), lo), hi);  // truncation toward zero
  const int md = min(max(ma + mn, lo), hi);
  return md >= 0 ? 1u : 0u;
}

__device__ __forceinline__ uint32_t ld_acquire_sys(const unsigned int* p) {
  uint32_t v;
  asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release_sys(unsigned int* p, uint32_t v) {
  asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Serving kernel, one thread: the next request of the queue, or -1 when the queue stayed
// empty for Q.idle_ns or the host asked the kernel to stop (the reason goes to exit_status).
__device__ int serve_claim(const ServeQueue& Q) {
  const uint64_t t0 = global_ns();
  for (;;) {
    const uint32_t h = *reinterpret_cast<volatile unsigned int*>(Q.head);
    const uint32_t tl = ld_acquire_sys(Q.tail);
    if (h < tl) {
      if (atomicCAS(Q.head, h, h + 1) == h) return static_cast<int>(h);
      continue;
    }
    if (*reinterpret_cast<const volatile unsigned int*>(Q.stop) != 0) {
      atomicCAS(Q.exit_status, 0, 2);
      return -1;
    }
    if (global_ns() - t0 > Q.idle_ns) {
      atomicCAS(Q.exit_status, 0, 1);
      return -1;
    }
    __nanosleep(256);
  }
}

// Threads, shared memory and launch limits of a CTA for up to CAP spins and `rows` replicas.
// W: spins per decision thread and chunk.  8 (one Philox block) halves the chain of a sweep
// where the warps for it fit; CAP = 256 would need 32 decision warps.
template <int CAP>
struct FloatCfg {
  static constexpr int W = CAP == 256 ? 16 : 8;
  static constexpr int kWarps = CAP / W;             // decision warps
  static constexpr int kChunks = CAP / 16;           // 16-bit spin words per replica
  static constexpr int kRowBytes = 2 * CAP;          // operand row of CAP BF16 values
  // Energy warps: two of one half each for 32 replicas, where a sweep is shortest; else one
  // per 32 replicas for both halves (with 8 of them the register cap would cause spills).
  static constexpr int threads(int rows) { return 32 * (kWarps + (rows == 128 ? 4 : 2) + 1); }
  // launch bound: for CAP = 64 that of two CTAs of 32 replicas (11 warps each) per SM
  static constexpr int kBoundThreads = CAP == 64 ? 32 * 22 : threads(128);
  static constexpr int kJBytes = CAP * kRowBytes;    // one coupling image
  static constexpr int kFixed = 1024 + kTileM * kRowBytes + 4096 * 4 + CAP * 4 +
                                3 * kChunks * kTileM * 2 + 2 * 2 * 32 * 4 + 128 +
                                static_cast<int>(sizeof(Problem));
};
template <int CAP>
int float_smem_bytes(bool fixed) {
  return FloatCfg<CAP>::kFixed + (fixed ? 2 : 1) * FloatCfg<CAP>::kJBytes;
}

// kPlain / kFixedPoint: CTA b runs work item b of L (one instance x L.rows replicas).
// kServing: persistent CTAs take requests from the queue Q one after another (each a whole
// instance of at most L.rows replicas, initial spins from Philox, float32 decisions); the
// request's descriptor, couplings and bias are read from mapped host memory with loads that
// bypass the caches (a slot is rewritten for later requests), and the results go back there
// before the slot's done flag.
template <int CAP, int MODE>
__global__ void __launch_bounds__(FloatCfg<CAP>::kBoundThreads, 1)
    sweep_float_kernel(const __grid_constant__ Launch L, const __grid_constant__ ServeQueue Q) {
  using Cfg = FloatCfg<CAP>;
  constexpr int W = Cfg::W, G = Cfg::kChunks, NW = Cfg::kWarps, kRowBytes = Cfg::kRowBytes;
  constexpr bool SERVE = MODE == kServing, FIXED = MODE == kFixedPoint;
  constexpr int kJParts = FIXED ? 2 : 1;
  constexpr int kImgRows = CAP <= 128 ? 128 : 256;  // rows of the staged image's K-blocks
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* sJ = smem;                                             // kJParts coupling images
  uint8_t* sA = sJ + kJParts * Cfg::kJBytes;                      // 128 x kRowBytes
  float* sZ = reinterpret_cast<float*>(sA + kTileM * kRowBytes);  // 4096 noise levels
  float* sH = sZ + 4096;                                          // CAP
  float* sPart = sH + CAP;                                        // [2][2][32] energy halves
  uint16_t* sBits = reinterpret_cast<uint16_t*>(sPart + 2 * 2 * 32);  // [2][G][128] spins
  uint16_t* sBest = sBits + 2 * G * kTileM;                       // [G][128] best state
  uint64_t* bars = reinterpret_cast<uint64_t*>(sBest + G * kTileM);
  uint32_t* sTmem = reinterpret_cast<uint32_t*>(bars + 8);
  volatile int* sAbort = reinterpret_cast<volatile int*>(sTmem + 1);  // [0] abort, [1] request
  Problem* sProb = reinterpret_cast<Problem*>(bars + 12);         // serving: the request

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nrg = L.rows >> 5;                 // replica groups of 32: 1, 2 or 4
  const int ewarps = nrg == 4 ? 4 : 2;         // energy warps
  const int quad = warp & 3;
  const int grp = quad & (nrg - 1);            // replica group of this warp's TMEM lanes
  const int rep = grp * 32 + lane;             // replica inside the tile
  const bool decides = warp < NW, sums = warp >= NW && warp < NW + ewarps;
  const bool multiplies = warp == NW + ewarps;
  // decision warps: (warp / 4, copy of the replica group) is the slot; chunks slot + j NW / nrg
  const int lg = nrg >> 1;           // log2(nrg)
  const int step = NW >> lg, slot = (warp >> 2) * (4 >> lg) + (quad >> lg);
  const uint32_t bar_mma0 = smem_u32(&bars[0]);  // [2]: fields in accumulator 0 / 1
  const uint32_t bar_ready = smem_u32(&bars[2]);  // spins written by every decision warp
  const uint32_t bar_sum0 = smem_u32(&bars[3]);   // [2]: energy of state m & 1 summed
  const uint32_t bar_j = smem_u32(&bars[5]);

  if (multiplies) {
    tmem_alloc(smem_u32(sTmem), 2 * CAP);
    tmem_relinquish();
    if (lane == 0) {
      mbar_init(bar_mma0, 2);
      mbar_init(bar_mma0 + 8, 2);
      mbar_init(bar_ready, NW);
      mbar_init(bar_sum0, ewarps);
      mbar_init(bar_sum0 + 8, ewarps);
      mbar_init(bar_j, 1);
      fence_mbar_init();
      sAbort[0] = 0;
    }
  }
  if constexpr (SERVE)
    for (int k = tid; k < 4096; k += blockDim.x) sZ[k] = Q.zlev[k];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *sTmem;
  const uint32_t tmem_warp = tmem + (static_cast<uint32_t>(quad * 32) << 16);
  uint32_t m = 0;  // MMAs done before this unit: MMA m fills accumulator m & 1
  bool j_pending = false;
  auto give_up = [&]() {
    atomicOr(L.err, kDevErrTimeout);
    sAbort[0] = 1;
  };

  for (int unit = 0;; ++unit) {
    // ---- unit: this CTA's work item, or the next request of the queue -----------------
    int req = 0;
    if constexpr (SERVE) {
      if (tid == 0) sAbort[1] = serve_claim(Q);
      __syncthreads();
      req = sAbort[1];
      if (req < 0) break;
      const volatile int* src = reinterpret_cast<const volatile int*>(
          Q.slots + static_cast<size_t>(req % Q.nslots) * Q.slot_bytes);
      for (int k = tid; k < static_cast<int>(sizeof(Problem) / 4); k += blockDim.x)
        reinterpret_cast<int*>(sProb)[k] = src[k];
      __syncthreads();
    } else {
      if (unit > 0) break;
    }
    const WorkItem wk = SERVE ? WorkItem{0, 0} : L.work[blockIdx.x];
    const Problem& P = SERVE ? *sProb : L.probs[wk.prob];
    const int n = P.n, R = P.R;
    const uint32_t q = P.q;
    const int rg = wk.rbase + rep;
    const bool row_valid = rg < R;
    const bool grp_active = wk.rbase + grp * 32 < R;
    const int nch = (n + 15) >> 4;           // 16-spin chunks = 16-value K-steps
    const int mma_n = nch * 16;
    const int t_begin = L.t_begin, t_end = L.t_begin + L.sweeps;
    const int half_words = P.words * 2;      // 16-bit words per row of the caller's bit arrays

    // ---- prologue: zeroed A operand, noise levels, bias, coupling image -----------------
    for (int k = tid; k < kTileM * kRowBytes / 16; k += blockDim.x)
      reinterpret_cast<uint4*>(sA)[k] = make_uint4(0, 0, 0, 0);
    if constexpr (SERVE) {
      for (int k = tid; k < CAP; k += blockDim.x)
        sH[k] = (P.hf != nullptr && k < n) ? __ldcv(P.hf + k) : 0.0f;
      for (int kb = 0; kb < CAP / 64; ++kb)
        for (int k = tid; k < CAP * 8; k += blockDim.x)
          reinterpret_cast<uint4*>(sJ + kb * CAP * 128)[k] =
              __ldcv(reinterpret_cast<const uint4*>(P.jimg + kb * kImgRows * 128) + k);
    } else {
      if (multiplies && lane == 0) {
        mbar_expect_tx(bar_j, kJParts * Cfg::kJBytes);
        for (int part = 0; part < kJParts; ++part)
          for (int kb = 0; kb < CAP / 64; ++kb)
            bulk_g2s(smem_u32(sJ + part * Cfg::kJBytes + kb * CAP * 128),
                     (part ? P.jimg_lo : P.jimg) + kb * kImgRows * 128, CAP * 128, bar_j);
      }
      j_pending = multiplies;
      const float* lev = FIXED ? reinterpret_cast<const float*>(P.fix_z) : P.zlev;
      for (int k = tid; k < 4096; k += blockDim.x) sZ[k] = __ldg(lev + k);
      for (int k = tid; k < CAP; k += blockDim.x) sH[k] = (P.hf != nullptr && k < n) ? P.hf[k] : 0.0f;
    }
    fence_proxy_async_smem();  // this thread's zeros (and, serving, couplings)
    __syncthreads();  // the zeroed operand is complete before any warp writes its spins

    if (decides) {
      // ---- decision warps -------------------------------------------------------------
      const float xi = P.xi;
      const int act = P.act, levels = P.lut_levels;
      const float margin = rule_margin(act, xi);
      float* const fields = SERVE ? nullptr : P.fields_out;
      const int nchw = nch * (16 / W);
      uint8_t* bits8 = reinterpret_cast<uint8_t*>(sBits);
      const int copies = 4 >> lg, copy_bytes = 4096 * nrg;
      // spins c W .. c W + W - 1 of this thread's replica in state buffer b
      auto bits_at = [&](uint32_t b, int c) {
        return bits8 + ((b * G + c * W / 16) * kTileM + rep) * 2 + (W == 8 ? (c & 1) : 0);
      };
      // new spins of chunk c: bits (those past n cleared) for the next state, and operand
      // bytes (words of two BF16) into every copy of the replica's row
      auto put_chunk = [&](uint32_t b, int c, uint32_t nb, const uint32_t (&wd)[W / 2]) {
        const int valid = n - c * W;
        if (valid < W) nb &= valid > 0 ? (1u << valid) - 1u : 0u;
        if constexpr (W == 16)
          *reinterpret_cast<uint16_t*>(bits_at(b, c)) = static_cast<uint16_t>(nb);
        else
          *bits_at(b, c) = static_cast<uint8_t>(nb);
#pragma unroll
        for (int k = 0; k < W / 8; ++k) {
          uint8_t* at = sA + sw128_offset(rep, c * 2 * W + 16 * k, kTileM);
#pragma unroll
          for (int i = 0; i < 4; ++i)  // rows rep + 32 nrg i: 4 KB per 32 rows, the same swizzle
            if (i < copies)
              *reinterpret_cast<uint4*>(at + i * copy_bytes) =
                  make_uint4(wd[4 * k], wd[4 * k + 1], wd[4 * k + 2], wd[4 * k + 3]);
        }
      };
      // s(t_begin)
      if (grp_active)
        for (int c = slot; c < nchw; c += step) {
          uint32_t nb = 0;
          if (row_valid) {
            if constexpr (SERVE) {
              // bit 15 of the draw at step field 0xFFFFFFFF (one Philox block per 8)
#pragma unroll
              for (int g = 0; g < W / 8; ++g) {
                const PhiloxOut o = philox4x32_10_rk(c * W / 8 + g, static_cast<uint32_t>(rg), 0xFFFFFFFFu,
                                                     q, L.round_keys);
#pragma unroll
                for (int e = 0; e < 8; ++e) nb |= ((philox_half(o, e) >> 15) & 1u) << (8 * g + e);
              }
            } else {
              const size_t at = static_cast<size_t>(rg) * half_words * 2 + c * W / 8;  // byte of the bit rows
              const uint8_t* in = reinterpret_cast<const uint8_t*>(P.cur_bits) + at;
              nb = W == 16 ? *reinterpret_cast<const uint16_t*>(in) : *in;
            }
          }
          uint32_t wd[W / 2];
#pragma unroll
          for (int k = 0; k < W / 8; ++k) {
            const uint4 x = bf16x8_from_bits((nb >> (8 * k)) & 0xFFu);
            wd[4 * k] = x.x, wd[4 * k + 1] = x.y, wd[4 * k + 2] = x.z, wd[4 * k + 3] = x.w;
          }
          put_chunk(m & 1, c, nb, wd);
        }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_ready);

      // the next sweep's schedule values are loaded a sweep ahead
      const float *sb = P.sched_b, *se = P.sched_eta;
      float b_next = t_begin < t_end ? __ldg(sb + t_begin) : 0.0f;
      float eta_next = t_begin < t_end ? __ldg(se + t_begin) : 0.0f;
      for (int t = t_begin; t < t_end; ++t, ++m) {
        const float b = b_next, eta = eta_next;
        if (t + 1 < t_end) {
          b_next = __ldg(sb + t + 1);
          eta_next = __ldg(se + t + 1);
        }
        const int eta_q = FIXED ? P.fix_eta[t] : 0;
        const bool dumps = !SERVE && fields != nullptr && t == t_begin;  // diagnostics
        const uint32_t acc = tmem_warp + (m & 1) * CAP;
        bool waited = false, ok = true;
        auto wait_fields = [&]() {
          if (waited) return;
          waited = true;
          // the fields of s(t), and the energy of s(t-1), whose bits the new ones replace
          ok = mbar_wait_fast(bar_mma0 + 8 * (m & 1), (m >> 1) & 1, L.wait_ns) &&
               (m == 0 || mbar_wait_fast(bar_sum0 + 8 * ((m - 1) & 1), ((m - 1) >> 1) & 1, L.wait_ns));
          ok = __all_sync(0xFFFFFFFFu, ok);  // the same answer on every lane
          tc_fence_after();
        };
        if (grp_active)
#pragma unroll 1
          for (int c = slot; c < nchw; c += step) {
            const uint32_t ob = W == 16 ? *reinterpret_cast<const uint16_t*>(bits_at(m & 1, c)) : *bits_at(m & 1, c);
            uint32_t rw[W / 2];
#pragma unroll
            for (int g = 0; g < W / 8; ++g) {
              const PhiloxOut o = philox4x32_10_rk(c * W / 8 + g, static_cast<uint32_t>(rg),
                                                   static_cast<uint32_t>(t), q, L.round_keys);
              rw[4 * g] = o.x0, rw[4 * g + 1] = o.x1, rw[4 * g + 2] = o.x2, rw[4 * g + 3] = o.x3;
            }
            auto level = [&](int e) {  // z of spin e's key
              const uint32_t word = rw[e >> 1];
              return sZ[(e & 1) ? (word >> 20) : ((word >> 4) & 0xFFFu)];
            };
            auto inertia = [&](int e) { return ((ob >> e) & 1u) ? xi : -xi; };
            float g[W];  // sign: the new spin
            uint32_t v[W];
            if constexpr (!FIXED) {
#pragma unroll
              for (int e = 0; e < W; ++e) g[e] = __fmaf_rn(eta, level(e), inertia(e));
            }
            wait_fields();
            if constexpr (W == 16)
              tmem_ld16(acc + c * W, v);
            else
              tmem_ld8(acc + c * W, v);
            tmem_wait_ld(v);
            float x[W];
#pragma unroll
            for (int e = 0; e < W; ++e) x[e] = __fadd_rn(__uint_as_float(v[e]), sH[c * W + e]);
            if (dumps && row_valid)
#pragma unroll
              for (int e = 0; e < W; ++e)
                if (c * W + e < n) fields[static_cast<size_t>(rg) * n + c * W + e] = x[e];
            if constexpr (FIXED) {
#pragma unroll
              for (int e = 0; e < W; ++e)
                g[e] = fixed_decide(x[e], (ob >> e) & 1u, b, eta_q, __float_as_int(level(e)), P.fix_xi,
                                    P.fix_f, 1 << (P.fix_w - 1), P.fix_tau)
                           ? 1.0f
                           : -1.0f;
            } else {
              float least = 8.0f;
#pragma unroll
              for (int e = 0; e < W; ++e) {
                x[e] = __fmul_rn(b, x[e]);
                g[e] = __fadd_rn(tanh_approx(x[e]), g[e]);
                least = min_nan(least, fabsf(g[e]));
              }
              if (__any_sync(0xFFFFFFFFu, !(least > margin)))
                settle_chunk<W>(g, x, c * W / 8, static_cast<uint32_t>(rg), static_cast<uint32_t>(t), q,
                                L.round_keys, ob, margin, xi, eta, act, levels, sZ);
            }
            // the sign of g is the sign of the BF16 spin
            uint32_t neg = 0, wd[W / 2];
#pragma unroll
            for (int e = W - 1; e >= 0; --e) neg = __funnelshift_l(__float_as_uint(g[e]), neg, 1);
#pragma unroll
            for (int k = 0; k < W / 2; ++k)
              wd[k] = (__byte_perm(__float_as_uint(g[2 * k]), __float_as_uint(g[2 * k + 1]), 0x7632) &
                       0x80008000u) |
                      0x3F803F80u;
            put_chunk((m + 1) & 1, c, ~neg & ((1u << W) - 1u), wd);
          }
        wait_fields();  // a warp without a chunk stays in step
        if (!ok) {
          if (lane == 0) give_up();
          break;
        }
        fence_proxy_async_smem();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_ready);
      }
    } else if (sums) {
      // ---- energy warps: sum_i s_i (I_i + h_i) over each half's columns, in column order ---
      const bool both = nrg > 1;                  // this warp sums both halves
      const int half = both ? 0 : warp - NW;      // else this one
      const int split = (n + 16) >> 5;
      const int cb = half == 0 ? 0 : split, ce = half == 0 && !both ? split : nch;  // its chunks
      const float scale = FIXED ? __int_as_float((127 + P.fix_f) << 23) : 1.0f;  // 2^F
      double best_E = DBL_MAX;  // float32 energies, or exact ones (fixed point)
      int best_t = -1, first_hit = -1;
      const bool has_target = P.has_target != 0;
      const double target = P.target_f;
      const bool cont = !SERVE && L.cont;
      if (cont && row_valid) {
        best_E = P.best_E[rg];
        best_t = P.best_t[rg];
        first_hit = P.first_hit[rg];
        const uint16_t* best_in = reinterpret_cast<const uint16_t*>(P.best_bits) + static_cast<size_t>(rg) * half_words;
        for (int c = cb; c < ce; ++c) sBest[c * kTileM + rep] = best_in[c];
      }
      double E = 0.0;
      for (int t = t_begin; t <= t_end; ++t, ++m) {
        bool ok = __all_sync(0xFFFFFFFFu, mbar_wait_fast(bar_mma0 + 8 * (m & 1), (m >> 1) & 1, L.wait_ns));
        tc_fence_after();
        const uint16_t* bits = sBits + (m & 1) * G * kTileM + rep;
        // sum over chunks [c0, c1): FP32, or units of 2^-F as integer bits (fixed point, exact)
        auto sum_chunks = [&](int c0, int c1) -> float {
          float eacc = 0.0f;
          int ieacc = 0;
          const uint32_t acc = tmem_warp + (m & 1) * CAP;
#pragma unroll 1
          for (int c = c0; c < c1; ++c) {
            uint32_t v[16];
            tmem_ld16(acc + c * 16, v);
            const uint32_t ob = bits[c * kTileM];
            tmem_wait_ld(v);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const float hv = sH[c * 16 + e];
              const float term = __fadd_rn(__fadd_rn(__uint_as_float(v[e]), hv), hv);
              const bool up = (ob >> e) & 1u;
              if constexpr (FIXED) {
                const int it = __float2int_rz(__fmul_rn(term, scale));
                ieacc += up ? it : -it;
              } else {
                eacc += up ? term : -term;
              }
            }
          }
          return FIXED ? __int_as_float(ieacc) : eacc;
        };
        float mine = 0.0f, other = 0.0f;
        if (grp_active) {
          mine = sum_chunks(cb, both ? split : ce);
          if (both) other = sum_chunks(split, nch);
        }
        if (!both) {
          float* part = sPart + (m & 1) * 64;
          part[half * 32 + lane] = mine;
          ok = !bar_sync_or(1, 64, !ok);
          other = part[(half ^ 1) * 32 + lane];
        }
        if (!ok) {
          if (lane == 0) give_up();
          break;
        }
        // the quadratic form is even in units of 2^-F: symmetric couplings, zero diagonal
        E = FIXED ? -static_cast<double>((__float_as_int(mine) + __float_as_int(other)) / 2) / scale
                  : static_cast<double>(-0.5f * (mine + other));
        const bool better = E < best_E;
        if (better) {
          best_E = E;
          best_t = t;
        }
        if (better || (t == t_begin && !cont))
          for (int c = cb; c < ce; ++c) sBest[c * kTileM + rep] = bits[c * kTileM];
        if (has_target && first_hit < 0 && E <= target) first_hit = t;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_sum0 + 8 * (m & 1));
      }
      if (row_valid && sAbort[0] == 0) {
        const uint16_t* bits = sBits + ((m - 1) & 1) * G * kTileM + rep;
        uint16_t* cur_out = reinterpret_cast<uint16_t*>(P.cur_bits) + static_cast<size_t>(rg) * half_words;
        uint16_t* best_out = reinterpret_cast<uint16_t*>(P.best_bits) + static_cast<size_t>(rg) * half_words;
        for (int c = cb; c < ce; ++c) {
          cur_out[c] = bits[c * kTileM];
          best_out[c] = sBest[c * kTileM + rep];
        }
        if (half == 0) {
          for (int c = nch; c < half_words; ++c) best_out[c] = 0;  // no spins there
          P.best_E[rg] = best_E;
          P.best_t[rg] = best_t;
          P.first_hit[rg] = first_hit;
          P.final_E[rg] = E;
        }
      }
    } else {
      // ---- MMA warp: D = S J^T for s(t_begin) .. s(t_end) ----------------------------------
      const uint32_t idesc = idesc_bf16(kTileM, mma_n);
      const uint64_t a_desc = sw128_desc(smem_u32(sA)), b_desc = sw128_desc(smem_u32(sJ));
      bool ok = true;
      if (j_pending) {
        ok = mbar_wait_bounded(bar_j, 0, L.wait_ns);
        j_pending = !__all_sync(0xFFFFFFFFu, ok);
      }
      for (int t = t_begin; t <= t_end; ++t, ++m) {
        ok = __all_sync(0xFFFFFFFFu, ok && mbar_wait_fast(bar_ready, m & 1, L.wait_ns));
        // injected fault: nothing is multiplied, so the first wait for fields cannot complete
        if (!ok || L.inject == 1) break;
        tc_fence_after();
        const uint32_t d = tmem + (m & 1) * CAP;
        if (elect_one()) {
          for (int part = 0; part < kJParts; ++part)  // fixed point: high part, then low part
            for (int kb = 0; kb * 4 < nch; ++kb) {
              const uint64_t a = a_desc + kb * (kTileM * 128 >> 4);
              const uint64_t bj = b_desc + (part * Cfg::kJBytes >> 4) + kb * (CAP * 128 >> 4);
#pragma unroll
              for (int ks = 0; ks < 4; ++ks)
                if (kb * 4 + ks < nch)
                  mma_bf16(d, a + 2 * ks, bj + 2 * ks, idesc, (kb > 0 || ks > 0 || part > 0) ? 1u : 0u);
            }
          mma_commit(bar_mma0 + 8 * (m & 1));
          mbar_arrive(bar_mma0 + 8 * (m & 1));  // passes the decision warps' writes on
        }
        __syncwarp();
      }
      if (!ok && lane == 0) give_up();
    }
    __syncthreads();
    if (sAbort[0] != 0) break;
    if (decides) ++m;  // the state after the last decision
    if constexpr (SERVE) {
      // every thread's results are written: make them visible to the host, then the flag
      __threadfence_system();
      __syncthreads();
      if (tid == 0) st_release_sys(Q.done + (req % Q.nslots), static_cast<uint32_t>(req) + 1u);
    }
  }
  if (multiplies && lane == 0) {
    // A wait gave up: give a copy or an MMA in flight a bounded chance to land before shared
    // and tensor memory are released.
    if (j_pending) mbar_wait_bounded(bar_j, 0, L.wait_ns);
    if (sAbort[0] != 0 && m > 0) mbar_wait_bounded(bar_mma0 + 8 * ((m - 1) & 1), ((m - 1) >> 1) & 1, L.wait_ns);
  }
  tc_fence_before();
  __syncthreads();
  if (multiplies) tmem_dealloc(tmem, 2 * CAP);
}

template <int CAP, int MODE>
cudaError_t launch_float_variant(const Launch& L, const ServeQueue& Q, int blocks, cudaStream_t st) {
  const int smem = float_smem_bytes<CAP>(MODE == kFixedPoint);
  cudaError_t e = cudaFuncSetAttribute(sweep_float_kernel<CAP, MODE>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  sweep_float_kernel<CAP, MODE><<<blocks, FloatCfg<CAP>::threads(L.rows), smem, st>>>(L, Q);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sweep_float(const Launch& L, int nmax, bool fixed, int blocks, cudaStream_t st) {
  const ServeQueue none{};
  if (fixed) return nmax <= 128 ? launch_float_variant<128, kFixedPoint>(L, none, blocks, st) : cudaErrorInvalidValue;
  if (nmax <= 64) return launch_float_variant<64, kPlain>(L, none, blocks, st);
  return nmax <= 128 ? launch_float_variant<128, kPlain>(L, none, blocks, st)
                     : launch_float_variant<256, kPlain>(L, none, blocks, st);
}

cudaError_t launch_serve_float(const Launch& L, const ServeQueue& Q, int nmax, int blocks,
                               cudaStream_t st) {
  if (nmax <= 64) return launch_float_variant<64, kServing>(L, Q, blocks, st);
  return nmax <= 128 ? launch_float_variant<128, kServing>(L, Q, blocks, st)
                     : launch_float_variant<256, kServing>(L, Q, blocks, st);
}

// J (BF16 bits, row-major n x n) -> BF16 operand image (rows npad, K = npad values, 2 bytes
// each, K-major with the 128-byte swizzle); zero outside n x n.  One thread per element.
// chunk_major: the 16 KB blocks (128 rows x one K-block) ordered [row block][K-block].
__global__ void stage_bf16_image_kernel(const uint16_t* __restrict__ J, int n, int npad,
                                        int chunk_major, uint8_t* __restrict__ img) {
  const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= static_cast<uint32_t>(npad) * npad) return;
  const int i = e / npad, j = e % npad;
  const uint16_t v = (i < n && j < n) ? J[static_cast<size_t>(i) * n + j] : 0;
  uint32_t off = sw128_offset(i, 2 * j, npad);  // K-block-major position
  if (chunk_major) {
    const uint32_t kblocks = static_cast<uint32_t>(npad) * 2u / 128u, block_bytes = npad * 128u;
    const uint32_t kb = off / block_bytes, rem = off % block_bytes;
    off = ((rem >> 14) * kblocks + kb) * 16384u + (rem & 16383u);
  }
  *reinterpret_cast<uint16_t*>(img + off) = v;
}

cudaError_t launch_stage_bf16_image(const uint16_t* d_J, int n, int npad, uint8_t* d_img,
                                    cudaStream_t st, bool chunk_major) {
  if (chunk_major && npad % 128 != 0) return cudaErrorInvalidValue;
  const uint32_t total = static_cast<uint32_t>(npad) * npad;
  stage_bf16_image_kernel<<<(total + 255) / 256, 256, 0, st>>>(d_J, n, npad, chunk_major ? 1 : 0, d_img);
  return cudaGetLastError();
}

}  // namespace pim
