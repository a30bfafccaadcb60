// Fused PIMI sweep kernel for integer couplings (n <= 256) when a launch has fewer replica
// tiles than the GPU has SMs: the same sweep as k_sweep_tc.cu with the shortest chain of
// dependent steps instead of the most work per SM.
//
// One CTA = one instance x a tile of 32, 64 or 128 replicas, all sweeps inside.  Per sweep t (Box 1;
// Eq. 2 then Eq. 4): fields D = S J^T by tcgen05.mma (FP8, exact), decision by the step's
// exact threshold table, spins written back into the A operand, energy of s(t) from the same
// fields.  A lone CTA is bound by latency (MMA, TMEM load, lookups, write-back, barrier, one after
// the other), so:
//  - a tile of 32 (64) replicas is written into all four (into two) lane quadrants of the A
//    operand, because a warp reads only the 32 TMEM lanes of its quadrant: the columns of a
//    replica are then split over CAP / W decision warps, each thread one replica and rows / 32
//    chunks of W spins;
//  - roles have their own warps, coupled by mbarriers: decision warps (noise is drawn while the MMAs
//    run), one bookkeeping warp per 32 replicas (energy, best state, first hit of s(t) while
//    s(t+1) is multiplied) and one MMA warp, which also streams the threshold tables through a
//    ring of four;
//  - two accumulators, so a CTA never waits for a reader of the old fields.
// Measured (GB300, us per sweep of 500-sweep runs, one instance of 128 replicas: 4 CTAs of 32;
// k_sweep_tc.cu before):
//   h = 0  n = 64  1.19 -> 0.78   n = 128  1.94 -> 1.12   n = 256  4.28 -> 1.65
//   h != 0 n = 64  1.94 -> 0.81   n = 128  3.50 -> 1.24   n = 256  7.24 -> 1.93
// What is left at n = 64 (cycles of 1650): MMA with its barriers 870, lookups 320, write-back 370.
// Measured slower: waits that spin without suspending (+8 %), the bookkeeping wait ahead of the
// noise (+18 %), the MMAs issued by a decision warp after a named barrier (+11 %).
#include <climits>

#include "int_rule.cuh"
#include "kernels.h"
#include "philox.cuh"
#include "sm100_ptx.cuh"

namespace pim {
namespace {

constexpr int kTileM = 128;
constexpr int kTabs = 4;            // threshold tables in flight
constexpr int kDiagWords = 512;     // one diagonal-encoded table: 1024 16-bit entries
constexpr int kDiagOffset = 256;

template <int CAP>
struct LatCfg {
  static constexpr int W = CAP == 256 ? 16 : 8;   // spins per decision thread and chunk
  static constexpr int kWarps = CAP / W;          // decision warps
  static constexpr int kChunks = CAP / 16;        // 16-bit spin words per replica
  static constexpr int kKB = CAP <= 128 ? 1 : 2;  // 128-byte K-blocks of an operand row
  static constexpr int kJBlock = CAP * 128;       // one K-block of the couplings
  static constexpr int kABlock = kTileM * 128;    // one K-block of the spins
  static constexpr int threads(int rows) { return 32 * (kWarps + rows / 32 + 1); }
  static constexpr int kFixed = 1024 + kKB * (kJBlock + kABlock) + CAP * 4 + 2 * kTileM * 4 +
                                3 * kChunks * kTileM * 2 + 160;
};

// DIAG: the image carries 256 on the diagonal and the table is indexed by D = I + 256 s (h = 0);
// else the table is indexed by I = D + h and holds both spins' thresholds.
template <int CAP, bool DIAG>
__global__ void __launch_bounds__(LatCfg<CAP>::threads(128), 1)
    sweep_lat_kernel(const __grid_constant__ Launch L) {
  using Cfg = LatCfg<CAP>;
  constexpr int W = Cfg::W, NW = Cfg::kWarps, G = Cfg::kChunks, KB = Cfg::kKB;
  constexpr int kImgRows = CAP <= 128 ? 128 : 256;  // rows of the staged image's K-blocks
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int tab_words = DIAG ? kDiagWords : L.stride_words_max;
  uint8_t* sJ = smem;
  uint8_t* sA = sJ + KB * Cfg::kJBlock;
  uint32_t* sTab = reinterpret_cast<uint32_t*>(sA + KB * Cfg::kABlock);  // [kTabs][tab_words]
  float* sH = reinterpret_cast<float*>(sTab + kTabs * tab_words);         // [CAP]
  int* sE = reinterpret_cast<int*>(sH + CAP);                                                 // [2][128] energy sums
  uint16_t* sBits = reinterpret_cast<uint16_t*>(sE + 2 * kTileM);        // [2][G][128] spins
  uint16_t* sBest = sBits + 2 * G * kTileM;                              // [G][128] best state
  uint64_t* bars = reinterpret_cast<uint64_t*>(sBest + G * kTileM);
  uint32_t* sTmem = reinterpret_cast<uint32_t*>(bars + 12);
  volatile int* sAbort = reinterpret_cast<volatile int*>(sTmem + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nrg = L.rows >> 5;       // replica groups of 32: 1, 2 or 4
  const int quad = warp & 3;
  const int grp = quad & (nrg - 1);  // replica group of this warp's TMEM lanes
  const int rep = grp * 32 + lane;   // replica inside the tile
  const bool decides = warp < NW, keeps = warp >= NW && warp < NW + nrg, multiplies = warp == NW + nrg;
  // decision warps: (warp / 4, copy of the replica group) is the slot; chunks slot + j NW / nrg
  const int lg = nrg >> 1;           // log2(nrg)
  const int step = NW >> lg, slot = (warp >> 2) * (4 >> lg) + (quad >> lg);
  const uint32_t bar_mma0 = smem_u32(&bars[0]);   // [2]: fields in accumulator 0 / 1
  const uint32_t bar_ready = smem_u32(&bars[2]);  // spins of a state written by every decision warp
  const uint32_t bar_kept0 = smem_u32(&bars[3]);  // [2]: state 0 / 1 mod 2 booked
  const uint32_t bar_sum0 = smem_u32(&bars[5]);   // [2]: energy of state 0 / 1 mod 2 summed
  const uint32_t bar_tab0 = smem_u32(&bars[7]);   // [kTabs]
  const uint32_t bar_j = smem_u32(&bars[11]);

  const WorkItem wk = L.work[blockIdx.x];
  const Problem& P = L.probs[wk.prob];
  const int n = P.n, R = P.R;
  const uint32_t q = P.q;
  const int stride = DIAG ? kDiagWords : P.stride_words;
  const uint32_t* thr = DIAG ? P.thr_diag : P.thr;
  const int rg = wk.rbase + rep;
  const bool row_valid = rg < R;
  const bool grp_active = wk.rbase + grp * 32 < R;
  const int nch = (n + 15) >> 4;
  const int sweeps = L.sweeps, t_begin = L.t_begin;
  const int half_words = P.words * 2;  // 16-bit words per row of the caller's bit arrays
  auto load_table = [&](int i) {       // one lane: table of sweep t_begin + i into its slot
    const uint32_t bar = bar_tab0 + 8 * (i & (kTabs - 1));
    mbar_expect_tx(bar, stride * 4);
    bulk_g2s(smem_u32(sTab) + (i & (kTabs - 1)) * tab_words * 4, thr + static_cast<size_t>(t_begin + i) * stride,
             stride * 4, bar);
  };
  auto give_up = [&]() {
    atomicOr(L.err, kDevErrTimeout);
    sAbort[0] = 1;
  };

  if (multiplies) {
    tmem_alloc(smem_u32(sTmem), 2 * CAP);
    tmem_relinquish();
    if (lane == 0) {
      mbar_init(bar_mma0, 2);
      mbar_init(bar_mma0 + 8, 2);
      mbar_init(bar_ready, NW);
      mbar_init(bar_kept0, nrg);
      mbar_init(bar_kept0 + 8, nrg);
      mbar_init(bar_sum0, NW);
      mbar_init(bar_sum0 + 8, NW);
      for (int k = 0; k < kTabs; ++k) mbar_init(bar_tab0 + 8 * k, 1);
      mbar_init(bar_j, 1);
      fence_mbar_init();
      sAbort[0] = 0;
      mbar_expect_tx(bar_j, KB * Cfg::kJBlock);
      for (int kb = 0; kb < KB; ++kb)
        bulk_g2s(smem_u32(sJ + kb * Cfg::kJBlock), P.jimg + kb * kImgRows * 128, Cfg::kJBlock, bar_j);
      for (int i = 0; i < kTabs - 1 && i < sweeps; ++i) load_table(i);
    }
  }
  for (int k = tid; k < KB * Cfg::kABlock / 16; k += blockDim.x)
    reinterpret_cast<uint4*>(sA)[k] = make_uint4(0, 0, 0, 0);
  for (int k = tid; k < CAP; k += blockDim.x)
    sH[k] = (!DIAG && P.h != nullptr && k < n) ? static_cast<float>(P.h[k]) : 0.0f;
  for (int k = tid; k < 2 * kTileM; k += blockDim.x) sE[k] = 0;
  fence_proxy_async_smem();  // this thread's zeros
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *sTmem;
  const uint32_t tmem_warp = tmem + (static_cast<uint32_t>(quad * 32) << 16);

  // State m = s(t_begin + m); MMA m fills accumulator m & 1 with its fields.
  if (decides) {
    const int copies = 4 >> lg, copy_bytes = 4096 * nrg;  // rows rep + 32 nrg i
    const int nchw = nch * (16 / W);
    uint8_t* bits8 = reinterpret_cast<uint8_t*>(sBits);
    auto bits_at = [&](uint32_t b, int c) {
      return bits8 + ((b * G + c * W / 16) * kTileM + rep) * 2 + (W == 8 ? (c & 1) : 0);
    };
    // new spins of chunk c as bits for state buffer b and as operand bytes in every copy of the row
    auto put_chunk = [&](uint32_t b, int c, uint32_t nb) {
      const int valid = n - c * W;
      if (valid < W) nb &= valid > 0 ? (1u << valid) - 1u : 0u;
      uint8_t* at = sA + sw128_offset(rep, c * W, kTileM);
      if constexpr (W == 16) {
        *reinterpret_cast<uint16_t*>(bits_at(b, c)) = static_cast<uint16_t>(nb);
        const uint4 x = fp8x16_from_bits(nb);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i < copies) *reinterpret_cast<uint4*>(at + i * copy_bytes) = x;
      } else {
        *bits_at(b, c) = static_cast<uint8_t>(nb);
        const uint2 x = make_uint2(fp8x4_from_bits(nb & 0xFu), fp8x4_from_bits(nb >> 4));
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i < copies) *reinterpret_cast<uint2*>(at + i * copy_bytes) = x;
      }
    };
    if (grp_active)
      for (int c = slot; c < nchw; c += step) {
        uint32_t nb = 0;
        if (row_valid) {
          const uint8_t* in = reinterpret_cast<const uint8_t*>(P.cur_bits) +
                              static_cast<size_t>(rg) * half_words * 2 + c * W / 8;
          nb = W == 16 ? *reinterpret_cast<const uint16_t*>(in) : *in;
        }
        put_chunk(0, c, nb);
      }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar_ready);

    for (int m = 0; m <= sweeps; ++m) {
      const bool last = m == sweeps;
      const uint32_t acc = tmem_warp + (m & 1) * CAP;
      const uint32_t tab = smem_u32(sTab) + (m & (kTabs - 1)) * tab_words * 4;
      // byte address of the entry of D = 0, or of the one of s = -1 and I = 0
      const uint32_t base = tab + (DIAG ? 2u * 512u : 4u * static_cast<uint32_t>(P.imax));
      bool waited = false, ok = true;
      auto wait_fields = [&]() {
        if (waited) return;
        waited = true;
        // the fields and the table of this sweep, and the bookkeeping of the state before, whose
        // bits the new ones replace
        ok = mbar_wait_fast(bar_mma0 + 8 * (m & 1), (m >> 1) & 1, L.wait_ns) &&
             (m == 0 || mbar_wait_fast(bar_kept0 + 8 * ((m - 1) & 1), ((m - 1) >> 1) & 1, L.wait_ns)) &&
             (last || mbar_wait_fast(bar_tab0 + 8 * (m & (kTabs - 1)), (m / kTabs) & 1, L.wait_ns));
        ok = __all_sync(0xFFFFFFFFu, ok);  // the same answer on every lane
        tc_fence_after();
      };
      float esum = 0.0f;
      if (grp_active)
#pragma unroll 1
        for (int c = slot; c < nchw; c += step) {
          uint32_t rw[W / 2];
#pragma unroll
          for (int g = 0; g < W / 8; ++g) {
            const PhiloxOut o = philox4x32_10_rk(c * W / 8 + g, static_cast<uint32_t>(rg),
                                                 static_cast<uint32_t>(t_begin + m), q, L.round_keys);
            rw[4 * g] = o.x0, rw[4 * g + 1] = o.x1, rw[4 * g + 2] = o.x2, rw[4 * g + 3] = o.x3;
          }
          const uint32_t ob = W == 16 ? *reinterpret_cast<const uint16_t*>(bits_at(m & 1, c)) : *bits_at(m & 1, c);
          wait_fields();
          if (!ok) break;  // no table to read
          uint32_t v[W];
          if constexpr (W == 16)
            tmem_ld16(acc + c * W, v);
          else
            tmem_ld8(acc + c * W, v);
          tmem_wait_ld(v);
          // The last state's energy alone counts.  Chunks of 16 decide all the same, on a stale table,
          // and the result goes nowhere: 1.365 us per sweep against 1.396 (one instance of N = 200 x 128),
          // but chunks of 8 1.08 against 0.94 (Max-Cut N = 100 x 64).
          const bool decide = W == 16 || !last;
          uint32_t nb;
          if constexpr (DIAG)
            nb = diag_rule<W>(v, rw, base, esum, decide);
          else
            nb = bias_rule<W>(v, rw, ob, sH + c * W, base, esum, decide);
          if (!last) put_chunk((m + 1) & 1, c, nb);
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
      // the energy share after the arrival the MMAs wait for
      if (grp_active) atomicAdd(&sE[(m & 1) * kTileM + rep], static_cast<int>(esum));
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_sum0 + 8 * (m & 1));
    }
  } else if (keeps) {
    // ---- bookkeeping: energy, best state and first hit of every state ---------------------
    int best_E = INT_MAX, best_t = -1, first_hit = -1, E = 0;
    const long long target = P.target;
    const bool has_target = P.has_target != 0;
    if (L.cont && row_valid) {
      best_E = static_cast<int>(P.best_E[rg]);
      best_t = P.best_t[rg];
      first_hit = P.first_hit[rg];
      const uint16_t* in = reinterpret_cast<const uint16_t*>(P.best_bits) + static_cast<size_t>(rg) * half_words;
      for (int c = 0; c < nch; ++c) sBest[c * kTileM + rep] = in[c];
    }
    bool ok = true;
    for (int m = 0; m <= sweeps; ++m) {
      ok = __all_sync(0xFFFFFFFFu, mbar_wait_fast(bar_sum0 + 8 * (m & 1), (m >> 1) & 1, L.wait_ns));
      if (!ok) {
        if (lane == 0) give_up();
        break;
      }
      int* sum = sE + (m & 1) * kTileM + rep;
      E = DIAG ? -((*sum - kDiagOffset * n) / 2) : -(*sum / 2);
      *sum = 0;
      const uint16_t* bits = sBits + (m & 1) * G * kTileM + rep;
      const bool better = E < best_E;
      if (better) {
        best_E = E;
        best_t = t_begin + m;
      }
      if (better || (m == 0 && !L.cont))
        for (int c = 0; c < nch; ++c) sBest[c * kTileM + rep] = bits[c * kTileM];
      if (has_target && first_hit < 0 && E <= target) first_hit = t_begin + m;
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_kept0 + 8 * (m & 1));
    }
    if (row_valid && ok && sAbort[0] == 0) {
      const uint16_t* bits = sBits + (sweeps & 1) * G * kTileM + rep;
      uint16_t* cur_out = reinterpret_cast<uint16_t*>(P.cur_bits) + static_cast<size_t>(rg) * half_words;
      uint16_t* best_out = reinterpret_cast<uint16_t*>(P.best_bits) + static_cast<size_t>(rg) * half_words;
      for (int c = 0; c < half_words; ++c) best_out[c] = c < nch ? sBest[c * kTileM + rep] : 0;
      for (int c = 0; c < nch; ++c) cur_out[c] = bits[c * kTileM];
      P.best_E[rg] = static_cast<double>(best_E);
      P.best_t[rg] = best_t;
      P.first_hit[rg] = first_hit;
      P.final_E[rg] = static_cast<double>(E);
    }
  } else {
    // ---- MMA warp (converged, one elected lane): fields of every state, tables ahead ---------
    const uint32_t idesc = idesc_e4m3(kTileM, nch * 16);
    const int ksteps = (n + 31) >> 5;
    const uint64_t a_desc = sw128_desc(smem_u32(sA)), j_desc = sw128_desc(smem_u32(sJ));
    bool ok = __all_sync(0xFFFFFFFFu, mbar_wait_bounded(bar_j, 0, L.wait_ns));
    int issued = 0;
    for (int m = 0; m <= sweeps; ++m) {
      ok = __all_sync(0xFFFFFFFFu, ok && mbar_wait_fast(bar_ready, m & 1, L.wait_ns));
      // injected fault: nothing is multiplied, so the first wait for fields cannot complete
      if (!ok || L.inject == 1) break;
      tc_fence_after();
      const uint32_t d = tmem + (m & 1) * CAP;
      if (elect_one()) {
#pragma unroll
        for (int ks = 0; ks < CAP / 32; ++ks)
          if (ks < ksteps)
            mma_e4m3(d, a_desc + (ks >> 2) * (Cfg::kABlock >> 4) + 2 * (ks & 3),
                     j_desc + (ks >> 2) * (Cfg::kJBlock >> 4) + 2 * (ks & 3), idesc, ks > 0 ? 1u : 0u);
        mma_commit(bar_mma0 + 8 * (m & 1));
        mbar_arrive(bar_mma0 + 8 * (m & 1));  // passes the decision warps' writes on
        // every decision of sweep m - 1 is taken, so the slot of table m - 2 is free
        if (m > 0 && m + kTabs - 2 < sweeps) load_table(m + kTabs - 2);
      }
      __syncwarp();
      issued = m + 1;
    }
    if (!ok && lane == 0) give_up();
    // No copy or MMA may be in flight when shared and tensor memory are released.
    mbar_wait_bounded(bar_j, 0, L.wait_ns);
    if (issued > 0)
      mbar_wait_bounded(bar_mma0 + 8 * ((issued - 1) & 1), ((issued - 1) >> 1) & 1, L.wait_ns);
    const int loaded = min(sweeps, issued <= 1 ? kTabs - 1 : issued + kTabs - 2);
    for (int i = max(0, loaded - kTabs); i < loaded; ++i)
      mbar_wait_bounded(bar_tab0 + 8 * (i & (kTabs - 1)), (i / kTabs) & 1, L.wait_ns);
  }
  tc_fence_before();
  __syncthreads();
  if (multiplies) tmem_dealloc(tmem, 2 * CAP);
}

template <int CAP, bool DIAG>
cudaError_t launch_lat(const Launch& L, int blocks, cudaStream_t st) {
  const int smem = LatCfg<CAP>::kFixed + kTabs * 4 * (DIAG ? kDiagWords : L.stride_words_max);
  cudaError_t e = cudaFuncSetAttribute(sweep_lat_kernel<CAP, DIAG>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  sweep_lat_kernel<CAP, DIAG><<<blocks, LatCfg<CAP>::threads(L.rows), smem, st>>>(L);
  return cudaGetLastError();
}

}  // namespace

bool sweep_lat_fits(int stride_words_max) {
  return LatCfg<256>::kFixed + kTabs * 4 * stride_words_max <= 227 * 1024;
}

cudaError_t launch_sweep_lat(const Launch& L, int nmax, int blocks, cudaStream_t st, bool diag) {
  if (nmax <= 64) return diag ? launch_lat<64, true>(L, blocks, st) : launch_lat<64, false>(L, blocks, st);
  if (nmax <= 128) return diag ? launch_lat<128, true>(L, blocks, st) : launch_lat<128, false>(L, blocks, st);
  return diag ? launch_lat<256, true>(L, blocks, st) : launch_lat<256, false>(L, blocks, st);
}

}  // namespace pim
