// Mid-N PIMI sweep kernel (integer couplings, n <= 1024): persistent, one CTA per SM.
// Serves any integer instance with n <= 1024 (plain or diagonal-encoded FP8 image).  Each
// CTA takes (instance, 128-replica panel) units from a global counter, in the order the host
// sorted them (largest first), and runs every sweep of a unit before it takes the next, so
// instances of any size and replica count share one launch with no inter-CTA
// synchronisation.
//
// Per unit, per sweep t (Box 1, PIMI loop; Eq. 2 then Eq. 4):
//   spins    the panel's spins s(t) stay in tensor memory as the A operand of the field
//            GEMM (128 replicas = TMEM lanes, npad FP8 +-1 along the columns, four per
//            32-bit column), written by the epilogue threads that own the rows;
//   fields   the couplings stream from L2 through a 3-stage cp.async.bulk ring (four
//            K-blocks of 128 coupling rows per stage, one copy when the image is chunk-major)
//            in chunks of 128 output spins (all shared memory but the step table is ring);
//            chunk c accumulates D[r, i] = sum_j S[r, j] J[i, j] into one of two TMEM
//            buffers (tcgen05.mma kind::f8f6f4, A from TMEM), so the MMAs of chunk c+1 run
//            while the epilogue decides chunk c;
//   decision 16 epilogue warps (4 TMEM lane quadrants x 4 groups of 32 columns): each
//            thread owns one replica and 32 spins of every chunk, keeps their old / new
//            bits, draws the Philox blocks and looks the threshold up in the step's table at
//            I = D + h (int_rule.cuh); the new spins go into a second tensor-memory image
//            chunk by chunk (npad <= 512) or into the one image after the last chunk (all
//            MMAs of the sweep have completed by then);
//   energy   E(s(t)) = -1/2 sum_i s_i (I_i + h_i), exact in int32, reduced over the four
//            column groups in shared memory; best state (written to the output array when
//            it improves) and first hit per replica.
#include <climits>

#include "int_rule.cuh"
#include "kernels.h"
#include "philox.cuh"
#include "sm100_ptx.cuh"

namespace pim {
namespace {

constexpr int kNT = 128;                    // output spins per chunk (MMA N)
constexpr int kMaxNpad = 1024;
constexpr int kMaxChunks = kMaxNpad / kNT;
constexpr int kStages = 3;                  // coupling ring depth
constexpr int kBufs = 2;                    // TMEM accumulators of kNT columns
// Threshold table in shared memory.  A step's table of up to kTabHalf words (imax <= 1023, diagonal
// encoding with dk <= 1024) lies in the half of its parity: the MMA warp has copied it
// while the sweep before was decided, and no thread waits at the start of a sweep.  A larger table
// takes both halves and is loaded by the epilogue threads between two barriers; past kTabWords it is
// read from global memory.  Loading every table between barriers cost 460 - 1800 of a sweep's 15.7 k
// (N = 512) to 33 k (N = 1000) cycles: SK N = 512 x 152 15.6 -> 14.9 us per sweep, N = 1000 x 152
// 35.2 -> 32.8.
constexpr int kTabWords = 4096;
constexpr int kTabHalf = kTabWords / 2;
constexpr int kEpiWarps = 16;
constexpr int kGroups = kEpiWarps / 4;      // column groups per chunk
constexpr int kCols = kNT / kGroups;        // columns of a chunk per epilogue thread
constexpr int kWordsPT = kCols / 32;        // 32-bit spin words per thread and chunk
constexpr int kEpiThreads = kEpiWarps * 32;
constexpr int kThreads = kEpiThreads + 64;  // + producer warp + MMA warp
constexpr int kTmemA = kBufs * kNT;         // first TMEM column of the spin image (npad / 4 columns)
constexpr int kTmemCols = kTmemA + kMaxNpad / 4;
// Up to this npad two spin images fit: the new spins of a chunk go into the other image as soon as
// they are decided, and the MMAs of the next sweep's first chunk run on all K-blocks but the last
// while the last chunk is decided.  With one image the warps wrote a whole panel's spins after the last
// chunk and then waited for a chunk's MMAs: SK N = 512 x 152 14.4 -> 13.4 us per sweep, N = 400 with a
// bias, 80 x 256, 17.1 -> 16.3.
constexpr int kTwoImages = kMaxNpad / 2;
constexpr int kImageCols = kTwoImages / 4;
constexpr int kBlockBytes = kNT * 128;      // one K-block of 128 coupling rows
// K-blocks per ring stage: a bulk copy costs about the same producer and copy-engine time
// whatever its size, so fewer, larger copies stream the couplings faster (measured: 4 x 3
// stages beat 2 x 6, 3 x 4 and 6 x 2 on the uneven batch).
constexpr int kKPS = 4;
constexpr int kStageBytes = kKPS * kBlockBytes;
static_assert(kTwoImages <= kKPS * 128, "with two images a chunk's K-blocks lie in one ring stage");
constexpr int kBarCount = 2 * kStages + 2 * kBufs + 4;

// Bounded wait with the common case (phase already complete) inline; the out-of-line wait
// sleeps inside try_wait between checks.
__device__ __forceinline__ bool wait_phase(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
  return mbar_try_wait(bar, parity) || mbar_wait_sleep(bar, parity, limit_ns);
}

// 32 spins -> their FP8 bytes in the thread's TMEM lane: K index col .. col + 31 = columns
// col / 4 .. col / 4 + 7 of the spin image (four K values per 32-bit column, lowest byte
// first).  Warp-collective.
__device__ __forceinline__ void put_spins32_tm(uint32_t tlane, int col, uint32_t bits, uint32_t neg) {
  const uint4 lo = fp8x16_from_bits(bits & 0xFFFFu, neg), hi = fp8x16_from_bits(bits >> 16, neg);
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(
                   tlane + static_cast<uint32_t>(kTmemA + col / 4)),
               "r"(lo.x), "r"(lo.y), "r"(lo.z), "r"(lo.w), "r"(hi.x), "r"(hi.y), "r"(hi.z), "r"(hi.w)
               : "memory");
}

// A thread's 32 columns of one chunk (two 16-column halves): the TMEM load of each half runs while its
// two Philox blocks are drawn (DECIDE: every sweep but the final energy pass), then the rule.  Returns
// the new spins of the 32 columns as bits.
template <bool DIAG, bool DECIDE>
__device__ __forceinline__ uint32_t chunk32(uint32_t ta, uint32_t blk0, uint32_t rg, uint32_t t, uint32_t q,
                                            const uint32_t* rk, uint32_t cw32, const int* h, uint32_t base,
                                            float& esum) {
  uint32_t word = 0;
#pragma unroll
  for (int h2 = 0; h2 < 2; ++h2) {
    uint32_t v[16];
    tmem_ld16(ta + 16 * h2, v);
    PhiloxOut o0{}, o1{};
    if constexpr (DECIDE) {
      o0 = philox4x32_10_rk(blk0 + 2 * h2, rg, t, q, rk);
      o1 = philox4x32_10_rk(blk0 + 2 * h2 + 1, rg, t, q, rk);
    }
    tmem_wait_ld(v);
    const uint32_t rw8[8] = {o0.x0, o0.x1, o0.x2, o0.x3, o1.x0, o1.x1, o1.x2, o1.x3};
    if constexpr (DIAG)
      word |= diag_rule<16>(v, rw8, base, esum, DECIDE) << (16 * h2);
    else
      word |= bias_rule<16>(v, rw8, (cw32 >> (16 * h2)) & 0xFFFFu, reinterpret_cast<const float*>(h) + 16 * h2,
                            base, esum, DECIDE)
              << (16 * h2);
  }
  return word;
}

// The same columns with the table in global memory (imax >= 2048), or of a diagonal-encoded image
// without its table, sixteen table reads in flight.  Returns the spins; the energy sum is added to eacc.
__device__ __forceinline__ uint32_t table_chunk32(uint32_t ta, int col0, int n, const int* sH, int dg, uint32_t cw32,
                                               const uint16_t* tab16, bool last, uint32_t rg, uint32_t t,
                                               uint32_t q, const uint32_t* rk, int& eacc) {
  uint32_t word = 0;
#pragma unroll 1
  for (int h2 = 0; h2 < 2; ++h2) {
    uint32_t v[16];
    tmem_ld16(ta + 16 * h2, v);
    const uint32_t blk = static_cast<uint32_t>(col0 >> 3) + 2 * h2;
    const PhiloxOut o0 = philox4x32_10_rk(blk, rg, t, q, rk), o1 = philox4x32_10_rk(blk + 1, rg, t, q, rk);
    tmem_wait_ld(v);
    const uint32_t rw8[8] = {o0.x0, o0.x1, o0.x2, o0.x3, o1.x0, o1.x1, o1.x2, o1.x3};
    const uint32_t cw16 = cw32 >> (16 * h2);
    uint32_t th[16], neg = 0;
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const int col = col0 + 16 * h2 + e;
      const int s = static_cast<int>((cw16 >> e) & 1u);
      const int hv = sH[col];
      const int dgc = col < n ? (s ? dg : -dg) : 0;  // image diagonal inside n only
      // exact float -> int of the integer-valued field (|D| < 2^22)
      const int I = static_cast<int>(__float_as_uint(__fadd_rn(__uint_as_float(v[e]), kMagic)) - kMagicBits) +
                    hv - dgc;
      const int term = I + hv;
      eacc += s ? term : -term;
      th[e] = last ? 0 : __ldg(tab16 + 2 * I + s);
    }
#pragma unroll
    for (int e = 15; e >= 0; --e) neg = __funnelshift_l(draw_below(draw_of(rw8, e), th[e], true), neg, 1);
    word |= (~neg & 0xFFFFu) << (16 * h2);
  }
  return word;
}

// One variant per MidMode keeps the register allocation of each to the path that it runs.  One kernel
// for both general tables took 30.2 us per sweep at N = 400 with a bias (80 instances x 256 replicas)
// and 23.7 at N = 700 with couplings of +-9 and a bias (60 x 256); these take 16.7 and 20.1 (runs of 100
// sweeps; 15.6 and 19.2 a sweep without the launch), and the bias units of N = 400 beside one with a
// larger table, on the variant for global memory, 24.7.
template <int MODE>
__global__ void __launch_bounds__(kThreads, 1) sweep_mid_kernel(const __grid_constant__ Launch L) {
  constexpr bool DIAG = MODE == kMidDiag;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* sRing = smem;
  uint32_t* sTab = reinterpret_cast<uint32_t*>(sRing + kStages * kStageBytes);
  int* sRed = reinterpret_cast<int*>(sTab + kTabWords);  // [2][kGroups][128 rows]
  int* sH = sRed + 2 * kGroups * 128;                     // [kMaxNpad]
  uint64_t* bars = reinterpret_cast<uint64_t*>(sH + kMaxNpad);
  uint32_t* sTmem = reinterpret_cast<uint32_t*>(bars + kBarCount);
  volatile int* sUnit = reinterpret_cast<volatile int*>(sTmem + 1);
  volatile int* sAbort = sUnit + 1;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool epi = warp >= 2;
  const int quad = warp & 3;                    // TMEM lane quadrant of this warp
  // Group of kCols columns inside a chunk.  The shuffles here and for P.q tell the compiler that the
  // value is the same on every lane: what the noise blocks need of it then lives in uniform registers
  // and the 96-register cap no longer spills (SK N = 512 x 152: 16.7 -> 15.6 us per sweep).
  const int grp = __shfl_sync(0xFFFFFFFFu, epi ? (warp - 2) >> 2 : 0, 0);
  const int row = quad * 32 + lane;             // replica row inside the panel
  const uint32_t full0 = smem_u32(&bars[0]);
  const uint32_t empty0 = smem_u32(&bars[kStages]);
  const uint32_t tfull0 = smem_u32(&bars[2 * kStages]);
  const uint32_t tempty0 = smem_u32(&bars[2 * kStages + kBufs]);
  const uint32_t aready = smem_u32(&bars[2 * kStages + 2 * kBufs]);
  const uint32_t drain = aready + 8;
  const uint32_t bar_tab0 = aready + 16;  // [2]

  if (warp == 1) {
    tmem_alloc(smem_u32(sTmem), kTmemCols);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < kBufs; ++b) {
      mbar_init(tfull0 + 8 * b, 1);
      mbar_init(tempty0 + 8 * b, kEpiWarps);
    }
    mbar_init(aready, 1);
    mbar_init(drain, 1);
    mbar_init(bar_tab0, 1);
    mbar_init(bar_tab0 + 8, 1);
    fence_mbar_init();
    *sAbort = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *sTmem;
  const uint32_t tlane = tmem + (static_cast<uint32_t>(quad * 32) << 16);  // this warp's TMEM lanes

  // Role counters, continued across units so every mbarrier phase is tracked exactly.
  uint32_t loads = 0, mmas = 0, cpass = 0, apass = 0;
  uint32_t tabs_copied = 0;  // MMA warp: every table copy it has issued
  uint32_t tabs = 0;  // tables copied ahead in earlier units (table k lies in half k & 1)
  bool first_unit = true;
  const uint32_t idesc = idesc_e4m3(128, kNT);

  for (;;) {
    if (tid == 0) *sUnit = static_cast<int>(atomicAdd(L.next, 1u));
    __syncthreads();
    const int u = *sUnit;
    if (__syncthreads_or(*sAbort != 0) || u >= L.nwork) break;  // also orders the sUnit reads

    const WorkItem wk = L.work[u];
    const Problem& P = L.probs[wk.prob];
    const int n = P.n, npad = P.npad, R = P.R;
    const int nchunks = npad / kNT, kblocks = npad / 128;
    const int t_begin = L.t_begin, t_end = L.t_begin + L.sweeps;
    const int dk = DIAG ? P.dk : 0;
    const int stride = dk > 0 ? 2 * dk : P.stride_words;  // table words per step
    const uint32_t* thr = dk > 0 ? P.thr_diag : P.thr;
    const bool tab_ahead = MODE != kMidTable && stride <= kTabHalf;
    const bool two_images = npad <= kTwoImages;

    if (warp == 0) {
      // ---- producer (converged warp, one elected lane): coupling K-blocks into the ring ---
      bool ok = true;
      for (int t = t_begin; t <= t_end && ok; ++t) {
        if (L.inject == 1 && first_unit && t == t_begin) continue;  // injected fault
        for (int c = 0; c < nchunks && ok; ++c)
          for (int kb0 = 0; kb0 < kblocks; kb0 += kKPS) {
            const int nk = kblocks - kb0 < kKPS ? kblocks - kb0 : kKPS;
            const uint32_t s = loads % kStages, use = loads / kStages;
            if (!__all_sync(0xFFFFFFFFu, (use == 0 || wait_phase(empty0 + 8 * s, (use - 1) & 1, L.wait_ns)) &&
                                             *sAbort == 0)) {
              ok = false;
              break;
            }
            if (elect_one()) {
              mbar_expect_tx(full0 + 8 * s, nk * kBlockBytes);
              if (npad > 256) {
                // images of n > 256 (npad >= 512) are chunk-major: the stage's K-blocks of chunk
                // c are contiguous, one copy
                bulk_g2s(smem_u32(sRing) + s * kStageBytes,
                         P.jimg + (static_cast<size_t>(c) * kblocks + kb0) * kBlockBytes, nk * kBlockBytes,
                         full0 + 8 * s);
              } else {
                for (int j = 0; j < nk; ++j)
                  bulk_g2s(smem_u32(sRing) + s * kStageBytes + j * kBlockBytes,
                           P.jimg + static_cast<size_t>(kb0 + j) * npad * 128 + static_cast<size_t>(c) * kNT * 128,
                           kBlockBytes, full0 + 8 * s);
              }
            }
            __syncwarp();
            ++loads;
          }
      }
      if (!ok && lane == 0) {
        atomicOr(L.err, kDevErrTimeout);
        *sAbort = 1;
      }
    } else if (warp == 1) {
      // ---- MMA issuer (converged warp, one elected lane): per sweep, wait for s(t) in the A
      // image, then every chunk --------------------------------------------------------------
      const uint32_t idesc_u = P.e5m2 ? idesc_e5m2(128, kNT) : idesc;
      const uint64_t ring_desc = sw128_desc(smem_u32(sRing));
      bool ok = true;
      auto copy_table = [&](int t) {  // table of step t into its half
        const uint32_t k = tabs + static_cast<uint32_t>(t - t_begin), half = k & 1;
        if (elect_one()) {
          mbar_expect_tx(bar_tab0 + 8 * half, stride * 4);
          bulk_g2s(smem_u32(sTab) + half * kTabHalf * 4, thr + static_cast<size_t>(t) * stride, stride * 4,
                   bar_tab0 + 8 * half);
        }
        __syncwarp();
        tabs_copied = k + 1;
      };
      if (tab_ahead && t_begin < t_end) copy_table(t_begin);
      for (int t = t_begin; t <= t_end && ok; ++t) {
        const uint32_t a_img = tmem + kTmemA + (two_images ? (t & 1) * kImageCols : 0);
        int c = 0;
        if (two_images && t > t_begin) {
          // First chunk.  Its accumulator is free once all chunks of sweep t - 1 but the last are
          // decided, and so are all K-blocks of the new image but the last.
          const uint32_t b = cpass % kBufs, buse = cpass / kBufs, p = cpass - 1;
          const uint32_t s = mmas % kStages, use = mmas / kStages;
          ok = __all_sync(0xFFFFFFFFu, (buse == 0 || wait_phase(tempty0 + 8 * b, (buse - 1) & 1, L.wait_ns)) &&
                                           wait_phase(full0 + 8 * s, use & 1, L.wait_ns));
          if (!ok) break;
          tc_fence_after();
          const uint64_t b0 = ring_desc + s * (kStageBytes >> 4);
          const uint32_t d = tmem + b * kNT;
          auto multiply = [&](int kb) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              mma_f8_ta(d, a_img + kb * 32 + ks * 8, b0 + kb * (kBlockBytes >> 4) + 2 * ks, idesc_u,
                        (kb > 0 || ks > 0) ? 1u : 0u);
          };
          if (elect_one())
            for (int kb = 0; kb + 1 < kblocks; ++kb) multiply(kb);
          __syncwarp();
          ok = __all_sync(0xFFFFFFFFu, wait_phase(tempty0 + 8 * (p % kBufs), (p / kBufs) & 1, L.wait_ns));
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            multiply(kblocks - 1);
            mma_commit(empty0 + 8 * s);
            mma_commit(tfull0 + 8 * b);
          }
          __syncwarp();
          ++mmas;
          ++cpass;
          c = 1;
        } else {
          ok = __all_sync(0xFFFFFFFFu, wait_phase(aready, apass & 1, L.wait_ns));
          if (!ok) break;
          ++apass;
          tc_fence_after();
        }
        // sweep t - 1 is decided: its table's half takes the next step's
        if (tab_ahead && t + 1 < t_end) copy_table(t + 1);
        for (; c < nchunks && ok; ++c) {
          const uint32_t b = cpass % kBufs, buse = cpass / kBufs;
          if (!__all_sync(0xFFFFFFFFu, buse == 0 || wait_phase(tempty0 + 8 * b, (buse - 1) & 1, L.wait_ns))) {
            ok = false;
            break;
          }
          tc_fence_after();
          for (int kb0 = 0; kb0 < kblocks; kb0 += kKPS) {
            const int nk = kblocks - kb0 < kKPS ? kblocks - kb0 : kKPS;
            const uint32_t s = mmas % kStages, use = mmas / kStages;
            if (!__all_sync(0xFFFFFFFFu, wait_phase(full0 + 8 * s, use & 1, L.wait_ns))) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (elect_one()) {
              const uint64_t b0 = ring_desc + s * (kStageBytes >> 4);
              const uint32_t a0 = a_img + kb0 * 32, d = tmem + b * kNT;
#pragma unroll
              for (int j = 0; j < kKPS; ++j)
                if (j < nk) {
#pragma unroll
                  for (int ks = 0; ks < 4; ++ks)
                    mma_f8_ta(d, a0 + j * 32 + ks * 8, b0 + j * (kBlockBytes >> 4) + 2 * ks, idesc_u,
                              (kb0 > 0 || j > 0 || ks > 0) ? 1u : 0u);
                }
              mma_commit(empty0 + 8 * s);
              if (kb0 + kKPS >= kblocks) mma_commit(tfull0 + 8 * b);
            }
            __syncwarp();
            ++mmas;
          }
          if (!ok) break;
          ++cpass;
        }
      }
      if (!ok && lane == 0) {
        atomicOr(L.err, kDevErrTimeout);
        *sAbort = 1;
      }
    } else if (epi) {
      // ---- epilogue ---------------------------------------------------------------------
      const int etid = tid - 64;
      const int rg = wk.rbase + row;
      const bool row_valid = rg < R;
      const bool warp_active = wk.rbase + quad * 32 < R;
      // Spins of this thread's 32-column word w of chunk c that exist (columns >= n stay -1).
      auto valid_mask = [&](int c, int w) -> uint32_t {
        const int valid = n - (c * kNT + grp * kCols + 32 * w);
        return valid >= 32 ? 0xFFFFFFFFu : (valid > 0 ? (1u << valid) - 1u : 0u);
      };
      // Bit rows of the caller's arrays as 32-bit words: word c*4 + grp*kWordsPT + w of row
      // rg holds this thread's spins 32w .. 32w+31 of chunk c.
      const int words = P.words;
      uint32_t* cur_io = P.cur_bits + static_cast<size_t>(rg) * words;
      uint32_t* best_io = P.best_bits + static_cast<size_t>(rg) * words;
      auto word_of = [&](int c, int w) { return c * (kNT / 32) + grp * kWordsPT + w; };
      const uint32_t neg8 = P.e5m2 ? 0xBCBCBCBCu : 0xB8B8B8B8u;  // -1 in the unit's FP8 format
      uint32_t cur[kMaxChunks][kWordsPT], nxt[kMaxChunks][kWordsPT];
      int best_E = INT_MAX, best_t = -1, first_hit = -1;
#pragma unroll
      for (int c = 0; c < kMaxChunks; ++c)
#pragma unroll
        for (int w = 0; w < kWordsPT; ++w) {
          cur[c][w] = nxt[c][w] = 0;
          if (c < nchunks && row_valid && word_of(c, w) < words)
            cur[c][w] = cur_io[word_of(c, w)] & valid_mask(c, w);
        }
      if (L.cont && row_valid) {
        best_E = static_cast<int>(P.best_E[rg]);
        best_t = P.best_t[rg];
        first_hit = P.first_hit[rg];
      }
      for (int k = etid; !DIAG && k < npad; k += kEpiThreads) {
        const int hv = (P.h != nullptr && k < n) ? P.h[k] : 0;
        sH[k] = MODE == kMidBias ? __float_as_int(static_cast<float>(hv)) : hv;
      }
#pragma unroll
      for (int c = 0; c < kMaxChunks; ++c)
#pragma unroll
        for (int w = 0; w < kWordsPT; ++w)
          if (c < nchunks) {
            put_spins32_tm(tlane + (two_images ? (t_begin & 1) * kImageCols : 0), c * kNT + grp * kCols + 32 * w,
                           cur[c][w], neg8);
          }
      tmem_wait_st();
      tc_fence_before();
      bool stop = bar_sync_or(1, kEpiThreads, false);
      if (etid == 0) mbar_arrive(aready);

      // Problem fields in registers: the loops below store to global memory, which would
      // otherwise make the compiler reload them from the descriptor.
      const uint32_t q = __shfl_sync(0xFFFFFFFFu, P.q, 0);
      const int imax = P.imax;
      const long long target = P.target;
      const bool has_target = P.has_target != 0;
      const int dg = P.diag_img ? 256 : 0;  // diagonal-encoded image: D = I + 256 s
      const int e_off = DIAG ? dk * n : 0;  // sum of |D| over the n spins = sum s I + n dk
      for (int t = t_begin; t <= t_end && !stop; ++t) {
        const bool last = t == t_end;
        bool waitfail = false;
        uint32_t half = 0;
        if (tab_ahead) {
          const uint32_t k = tabs + static_cast<uint32_t>(t - t_begin);
          half = k & 1;
          if (!last && !wait_phase(bar_tab0 + 8 * half, (k >> 1) & 1, L.wait_ns)) waitfail = true;
        } else {
          if (MODE != kMidTable && !last) {
            const uint4* src = reinterpret_cast<const uint4*>(thr + static_cast<size_t>(t) * stride);
            for (int k = etid; k < stride / 4; k += kEpiThreads)
              reinterpret_cast<uint4*>(sTab)[k] = __ldg(src + k);
            fence_proxy_async_smem();  // a later unit's bulk copies may take the same words
          }
          if (bar_sync_or(1, kEpiThreads, *sAbort != 0)) break;
        }
        const uint16_t* tab16 =  // in global memory, entry of s = -1 and I = 0
            reinterpret_cast<const uint16_t*>(thr + static_cast<size_t>(last ? t_begin : t) * stride + imax);
        // byte address of the entry of D = 0, or of the one of s = -1 and I = 0
        const uint32_t base = smem_u32(sTab) + half * kTabHalf * 4 + 4u * static_cast<uint32_t>(DIAG ? dk : imax);
        int* red = sRed + (t & 1) * kGroups * 128;
        int eacc = 0;
        // Chunk c decided: with two images its new spins go into the next sweep's now; then TMEM
        // buffer b, drained by this warp, is the MMA issuer's again.
        const uint32_t next_img = tlane + ((t + 1) & 1) * kImageCols;
        auto release = [&](int c, uint32_t b, uint32_t word) {
          nxt[c][0] = word;
          if (two_images && !last && warp_active) {
            put_spins32_tm(next_img, c * kNT + grp * kCols, word, neg8);
            tmem_wait_st();
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty0 + 8 * b);
        };
#pragma unroll 1
        for (int c = 0; c < nchunks; ++c) {
          const uint32_t b = cpass % kBufs, buse = cpass / kBufs;
          ++cpass;
          if (!wait_phase(tfull0 + 8 * b, buse & 1, L.wait_ns)) waitfail = true;
          tc_fence_after();
          const uint32_t ta = tmem + (static_cast<uint32_t>(quad * 32) << 16) + b * kNT + grp * kCols;
          const uint32_t blk0 = static_cast<uint32_t>((c * kNT + grp * kCols) >> 3);
          static_assert(kCols == 32 && kWordsPT == 1, "one 32-bit spin word per thread and chunk");
          uint32_t word = 0;  // new spins; columns at or past n stay -1 (bit 0)
          const int col0 = c * kNT + grp * kCols;
          // A thread whose 32 columns all lie at or past n skips them: their fields are zero, and they
          // stay -1.
          if (warp_active && col0 < n) {
            if constexpr (MODE == kMidTable) {
              word = table_chunk32(ta, col0, n, sH, dg, cur[c][0], tab16, last, static_cast<uint32_t>(rg),
                                   static_cast<uint32_t>(t), q, L.round_keys, eacc);
            } else {
              float esum = 0.0f;
              word = last ? chunk32<DIAG, false>(ta, blk0, static_cast<uint32_t>(rg), static_cast<uint32_t>(t), q,
                                                 L.round_keys, cur[c][0], sH + col0, base, esum)
                          : chunk32<DIAG, true>(ta, blk0, static_cast<uint32_t>(rg), static_cast<uint32_t>(t), q,
                                                L.round_keys, cur[c][0], sH + col0, base, esum);
              eacc += static_cast<int>(esum);
            }
          }
          release(c, b, word & valid_mask(c, 0));
        }
        if (!last && warp_active && !two_images) {
          // Every MMA of sweep t has completed (the last chunk's commit was awaited): the A
          // image can take s(t+1).
#pragma unroll
          for (int c = 0; c < kMaxChunks; ++c)
#pragma unroll
            for (int w = 0; w < kWordsPT; ++w)
              if (c < nchunks) {
                put_spins32_tm(tlane, c * kNT + grp * kCols + 32 * w, nxt[c][w], neg8);
              }
          tmem_wait_st();
          tc_fence_before();
        }
        red[grp * 128 + row] = eacc;
        stop = bar_sync_or(1, kEpiThreads, waitfail || *sAbort != 0);
        if (stop) {
          if (etid == 0) {
            atomicOr(L.err, kDevErrTimeout);
            *sAbort = 1;
          }
          break;
        }
        if (!last && etid == 0 && !two_images) mbar_arrive(aready);
        int tot = 0;
#pragma unroll
        for (int g = 0; g < kGroups; ++g) tot += red[g * 128 + row];
        const int E = -((tot - e_off) / 2);
        if (E < best_E) {
          // the best state lives in the output array: written when it improves
          best_E = E;
          best_t = t;
          if (row_valid) {
#pragma unroll
            for (int c = 0; c < kMaxChunks; ++c)
#pragma unroll
              for (int w = 0; w < kWordsPT; ++w)
                if (c < nchunks && word_of(c, w) < words) best_io[word_of(c, w)] = cur[c][w];
          }
        }
        if (has_target && first_hit < 0 && static_cast<long long>(E) <= target) first_hit = t;
        if (last) {
          if (row_valid) {
#pragma unroll
            for (int c = 0; c < kMaxChunks; ++c)
#pragma unroll
              for (int w = 0; w < kWordsPT; ++w)
                if (c < nchunks && word_of(c, w) < words) cur_io[word_of(c, w)] = cur[c][w];
            if (grp == 0) {
              P.best_E[rg] = static_cast<double>(best_E);
              P.best_t[rg] = best_t;
              P.first_hit[rg] = first_hit;
              P.final_E[rg] = static_cast<double>(E);
            }
          }
        } else {
#pragma unroll
          for (int c = 0; c < kMaxChunks; ++c)
#pragma unroll
            for (int w = 0; w < kWordsPT; ++w) cur[c][w] = nxt[c][w];
        }
      }
    }
    first_unit = false;
    if (tab_ahead) tabs += L.sweeps;
  }

  // ---- teardown: no copy or MMA of this CTA may still be in flight ------------------------
  if (warp == 1 && elect_one()) {  // the lane that issued the MMAs: a commit covers its own thread's
    mma_commit(drain);
    wait_phase(drain, 0, L.wait_ns);
    for (uint32_t k = tabs_copied > 2 ? tabs_copied - 2 : 0; k < tabs_copied; ++k)
      wait_phase(bar_tab0 + 8 * (k & 1), (k >> 1) & 1, L.wait_ns);
  } else if (tid == 0) {
    for (uint32_t k = loads > kStages ? loads - kStages : 0; k < loads; ++k)
      wait_phase(full0 + 8 * (k % kStages), (k / kStages) & 1, L.wait_ns);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

}  // namespace

int sweep_mid_smem_bytes() {
  return 1024 + kStages * kStageBytes + kTabWords * 4 + 2 * kGroups * 128 * 4 + kMaxNpad * 4 +
         kBarCount * 8 + 32;
}

int sweep_mid_max_npad() { return kMaxNpad; }

int sweep_mid_max_blocks() {
  const int smem = sweep_mid_smem_bytes();
  if (cudaFuncSetAttribute(sweep_mid_kernel<kMidTable>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
      cudaSuccess)
    return 0;
  int per_sm = 0, dev = 0, sms = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sweep_mid_kernel<kMidTable>, kThreads, smem) !=
      cudaSuccess)
    return 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return resident_ctas(per_sm, kTmemCols) * sms;
}

int sweep_mid_table_words() { return kTabWords; }

cudaError_t launch_sweep_mid(const Launch& L, int blocks, cudaStream_t st, MidMode mode) {
  const auto kernel = mode == kMidDiag   ? sweep_mid_kernel<kMidDiag>
                      : mode == kMidBias ? sweep_mid_kernel<kMidBias>
                                         : sweep_mid_kernel<kMidTable>;
  const int smem = sweep_mid_smem_bytes();
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(L.next, 0, sizeof(unsigned int), st);
  if (e != cudaSuccess) return e;
  kernel<<<blocks, kThreads, smem, st>>>(L);
  return cudaGetLastError();
}

}  // namespace pim
