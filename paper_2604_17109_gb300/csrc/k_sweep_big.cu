// Large-N PIMI sweep kernel (N > 256): persistent, cooperative, one CTA per (128-replica
// tile, NT-spin column block), all sweeps in one launch.  Three operand variants:
//   FP8   integer couplings: FP8 E4M3 spins and couplings (tcgen05 kind::f8f6f4), the couplings
//         streamed every sweep; exact integer fields and the exact threshold-table decision;
//   BF16  real couplings: BF16 images (kind::f16), FP32 fields, Eq. 4 evaluated in FP32;
//   FP4   integer couplings in {0, +-1, +-2, +-3, +-4, +-6}, NT = 64: the CTA's coupling rows
//         stay in shared memory as packed E2M1 for the whole launch (block-scaled kind::mxf4
//         with unit scale factors, so the products and the FP32 sums stay exact integers);
//         same decision as FP8.
// NT (64 or 128 spins) and the variant are chosen per instance by the host.
//
// Per sweep t (Box 1, PIMI loop; Eq. 2 then Eq. 4):
//   fields   D[r, i] = sum_j S[r, j] J[i, j] for the CTA's 128 replicas and NT spins, over the K
//            dimension (all N spins) in stages: the spins come from the global bit image, expanded by
//            the epilogue warps into tensor memory (the MMA's A operand), the rows of J from the
//            coupling image through a shared-memory ring filled by cp.async.bulk unless they are
//            resident.  Streaming the spins as operand bytes took as much of the L2-to-SM path as J
//            itself, which bounded the K loop (about 10 TB/s over all SMs).
//   decision 16 epilogue warps (4 TMEM lane quadrants x 4 column groups); each thread owns
//            one replica and NT/4 spins for the whole anneal, keeps their old / new / best
//            bits in registers, draws the Philox blocks and decides: integer couplings by
//            the step's threshold table at field I = D + h (staged into shared memory while
//            the MMAs run, or read through L1 when it does not fit), real couplings by
//            tanh(b_t I) + xi s + eta_t z >= 0.  It writes the new spins into the other spin
//            image and adds its share of sum_i s_i (I_i + h_i) to the replica's energy
//            accumulator (global atomics, three rotating buffers; int32 for integer
//            couplings, so the energy stays exact).
//   exchange a bounded barrier of the tile's CTAs (one arrival atomic on a monotone counter); during
//            the next sweep's K-loop every CTA reads the replica energies of s(t), updates best /
//            first hit (redundantly, identically in all CTAs) and keeps its own spins of s(t)
//            as the best state when the energy improved.
// Measured (GB300, us per sweep; spins streamed as operand bytes before -> as bits -> with a barrier per
// tile, runs of 40 to 100 sweeps): BF16 N = 8192 x 256 replicas 40.1 -> 33.8 -> 32.9, x 64 29.7 -> 26.2 ->
// 26.7; BF16 N = 2000 x 256 11.3 -> 9.8 -> 9.2, N = 1000 x 128 7.9 -> 6.9 -> 6.6; FP8 N = 4800 x 128 10.5 ->
// 10.0 -> 10.0; E2M1 N = 4096 x 256 7.0 -> 6.7 -> 6.6 (N = 1201 x 200 4.3 -> 4.6 -> 4.6).
#include <algorithm>
#include <cfloat>
#include <climits>
#include <type_traits>

#include "int_rule.cuh"
#include "kernels.h"
#include "philox.cuh"
#include "real_rule.cuh"
#include "sm100_ptx.cuh"

namespace pim {
namespace {

constexpr int kTabWords = 8192;     // threshold table of one step staged in shared memory
constexpr int kEpiWarps = 16;
constexpr int kThreads = (2 + kEpiWarps) * 32;
constexpr int kSmemBudget = 227 * 1024;

// The K loop runs in stages of kPB K-blocks through a ring of kStages: the spins' operand in tensor
// memory (32 columns, i.e. 128 bytes of every row, per K-block), expanded from the bit image by the
// epilogue warps (warp group g takes K-block g of a stage), and the streamed coupling rows in shared
// memory, on one full and one empty barrier.  A wait that finds its phase complete still costs the
// MMA warp 85 cycles and a commit 25, and the tensor pipe idles meanwhile (four MMAs of N = 128 take
// 260; 377 with two waits and two commits per K-block), so a stage is as large as both memories allow.
constexpr int kPB = 4;
constexpr int kStages = 3;
constexpr int kACols = 32;
constexpr int KPS = 2;  // K-blocks that odd sweeps keep in ascending order
// Odd sweeps walk the K-blocks from the last pair to the first, so a sweep starts on the coupling
// blocks the previous one read last, which are still in L2 (BF16 Max-Cut N = 8192, whose
// 134 MB image just exceeds L2: DRAM reads 136 -> 75 MB per sweep).  The order depends on the
// absolute sweep index, so split runs and resumes sum in the same order.
constexpr bool kRev = true;
// Shared-memory and tensor-memory plan of one kernel variant: NT output spins per CTA, operand
// variant OP.
template <int NT, int OP>
struct BigCfg {
  static constexpr bool kReal = OP == kBigBf16, kFp4 = OP == kBigFp4;
  static constexpr int kSpinsPerKB = kFp4 ? 256 : (kReal ? 64 : 128);  // per 128-byte row
  static constexpr int kWPK = kSpinsPerKB / 32;  // words of the bit image per row and K-block
  static constexpr int kSPT = NT / 4;            // spins per epilogue thread
  static constexpr int kChunks = kSPT / 16;      // 16-spin chunks per thread
  static constexpr int kBBytes = kFp4 ? 0 : NT * 128;  // streamed coupling rows per K-block
  static constexpr int kRing = kStages * kPB * kBBytes;
  // Largest step table staged in shared memory (words): 8192, or what the ring leaves.
  static constexpr int kTab = OP == kBigFp8 && NT == 128 ? 7680 : kTabWords;
  static constexpr int kAux = kReal ? 4096 * 4 : kTab * 4;  // noise levels | step table
  static constexpr int kMisc = 4 * 128 * 4 + NT * 4 + 256;  // sRed, sH, barriers, flags
  static constexpr int kSmem = 1024 + kRing + kAux + kMisc;
  static constexpr int kTmemA = kFp4 ? 2 * NT : NT;  // accumulator (+ unit scale factors), then A
  static constexpr int kTmemCols = 512;
  static_assert(kTmemA + kStages * kPB * kACols <= kTmemCols, "tensor memory");
  static_assert(kFp4 || kSmem <= kSmemBudget, "shared memory");
  static_assert(!kFp4 || NT == 64, "the coupling-resident variant has 64-spin column blocks");
};

// Shared-memory plan of the coupling-resident variant for npad spins: [pad][resident couplings
// NT x npad / 2][table?][misc].
BigSmem fp4_plan(int npad, int stride_words) {
  using C = BigCfg<64, kBigFp4>;
  BigSmem out;
  if (npad % 256 != 0 || npad > 4096) return out;
  out.tab_smem = stride_words <= C::kTab ? 1 : 0;
  out.bytes = 1024 + 64 * npad / 2 + (out.tab_smem ? C::kTab * 4 : 0) + C::kMisc;
  out.ok = out.bytes <= kSmemBudget;
  return out;
}

// ---- spins as bits: the image of one replica tile is [npad / 32 words][128 rows], each 16-bit half
// holding 16 consecutive spins in the order its operand type expands with a shift and a mask:
//   BF16  bit k = spin 2 k, bit 8 + k = spin 2 k + 1     (a register = spins 2 k, 2 k + 1)
//   FP8   bit 4 b + j = spin 4 j + b                      (register j = spins 4 j .. 4 j + 3)
//   E2M1  bits 4 m + 2 j, 4 m + 2 j + 1 = spins 8 j + 2 m, 8 j + 2 m + 1   (register j = spins 8 j ..
//         8 j + 7; a pair of bits selects a byte of two nibbles)
template <int OP>
__device__ __forceinline__ uint32_t pack_spins16(uint32_t x) {
  uint32_t t;
  if constexpr (OP == kBigBf16) {
    t = (x ^ (x >> 1)) & 0x2222u, x ^= t ^ (t << 1);
    t = (x ^ (x >> 2)) & 0x0C0Cu, x ^= t ^ (t << 2);
    t = (x ^ (x >> 4)) & 0x00F0u, x ^= t ^ (t << 4);
  } else if constexpr (OP == kBigFp8) {
    t = (x ^ (x >> 3)) & 0x0A0Au, x ^= t ^ (t << 3);
    t = (x ^ (x >> 6)) & 0x00CCu, x ^= t ^ (t << 6);
  } else {
    t = (x ^ (x >> 4)) & 0x00F0u, x ^= t ^ (t << 4);
    t = (x ^ (x >> 2)) & 0x0C0Cu, x ^= t ^ (t << 2);
  }
  return x;
}

// Half h of word w -> its operand registers v[0 .. kRegs - 1] (8 BF16, 4 FP8 or 2 E2M1).
template <int OP>
__device__ __forceinline__ void expand_spins16(uint32_t w, int h, uint32_t* v) {
  if constexpr (OP == kBigBf16) {
    const uint32_t z = __byte_perm(w, 0, h ? 0x3424 : 0x1404);
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = ((z << (7 - k)) & 0x80008000u) ^ 0xBF80BF80u;
  } else if constexpr (OP == kBigFp8) {
    uint32_t z = __byte_perm(w, 0, h ? 0x4342 : 0x4140);
    z = (z | (z << 4)) & 0x0F0F0F0Fu;
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = ((z << (7 - j)) & 0x80808080u) ^ 0xB8B8B8B8u;
  } else {
#pragma unroll
    for (int j = 0; j < 2; ++j) v[j] = __byte_perm(0x222AA2AAu, 0, (w >> (16 * h + 2 * j)) & 0x3333u);
  }
}

// Barrier of the CTAs of one replica tile (its spins, energies and images are its own, so the tiles of
// a launch need not wait for one another) with a time bound, over a monotone 64-bit arrival counter
// (bar[0..1], zeroed before the launch, on a 128-byte line of its own): a CTA's k-th barrier completes
// once the counter reaches k * ncb, so no reset or generation word is needed and an arrival is one
// acq_rel atomic.  Aborting sets a high bit of the counter, which releases every present and later
// wait of the tile at once; all of them then return false (on all threads of the CTA).
// Measured against one counter for all tiles (us per sweep, launch included, 60 to 100 sweeps): FP8
// N = 512 x 20 tiles 6.60 -> 6.21, N = 1024 x 18 7.58 -> 7.17; E2M1 N = 1500 x 6 4.99 -> 4.88, N = 4096 x 2
// 6.89 -> 6.91; BF16 N = 300 x 8 5.56 -> 4.98, N = 2000 x 8 13.7 -> 12.7, N = 8192 x 2 34.2 -> 33.6.
constexpr unsigned long long kBarAbort = 1ull << 62;

__device__ __forceinline__ void tile_abort(unsigned int* bar) {
  atomicOr(reinterpret_cast<unsigned long long*>(bar), kBarAbort);
}

// Called by the epilogue threads; their first one arrives for the CTA.
__device__ bool tile_barrier(unsigned int* bar, unsigned long long target, int* err, int* sflag,
                             uint64_t limit_ns) {
  const uint64_t limit = limit_ns ? limit_ns : 2000000000ull;
  asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
  if (threadIdx.x == 64) {
    unsigned long long* cnt = reinterpret_cast<unsigned long long*>(bar);
    unsigned long long v;
    asm volatile("atom.add.acq_rel.gpu.global.u64 %0, [%1], 1;" : "=l"(v) : "l"(cnt) : "memory");
    v += 1;
    if (v < target) {
      const uint64_t t0 = global_ns();
      uint32_t polls = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(cnt) : "memory");
        if ((++polls & 31) == 0 && v < target && global_ns() - t0 > limit) {
          atomicOr(err, kDevErrTimeout);
          tile_abort(bar);
          v |= kBarAbort;
        }
      } while (v < target);
    }
    *sflag = (v & kBarAbort) ? 0 : 1;
  }
  asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
  return *sflag != 0;
}

template <int NT, int OP>
__global__ void __launch_bounds__(kThreads, 1) sweep_big_kernel(const __grid_constant__ BigLaunch L) {
  using C = BigCfg<NT, OP>;
  constexpr bool REAL = C::kReal, FP4 = C::kFp4;
  using EAcc = std::conditional_t<REAL, float, int>;  // energy partial sums
  constexpr int kBBytes = C::kBBytes;
  constexpr int kSPT = C::kSPT, kChunks = C::kChunks, kWPK = C::kWPK;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* sB = smem;                               // kStages x kPB x kBBytes (streamed couplings)
  uint8_t* sJ = sB + C::kRing;                      // resident couplings (FP4): NT x npad / 2
  const int jres_bytes = FP4 ? NT * L.P.npad / 2 : 0;
  const bool tab_smem = L.tab_smem != 0;
  uint32_t* sTab = reinterpret_cast<uint32_t*>(sJ + jres_bytes);  // [C::kTab]
  float* sZ = reinterpret_cast<float*>(sTab);       // [4096] noise levels (real)
  const int aux_bytes = REAL ? C::kAux : (FP4 && !tab_smem ? 0 : C::kAux);
  EAcc* sRed = reinterpret_cast<EAcc*>(sJ + jres_bytes + aux_bytes);  // [4][128 rows]
  uint32_t* sH = reinterpret_cast<uint32_t*>(sRed + 4 * 128);  // [NT] bias: int32 or float bits
  uint64_t* bars = reinterpret_cast<uint64_t*>(sH + NT);
  uint32_t* sTmem = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 3);
  int* sFlag = reinterpret_cast<int*>(sTmem + 1);

  const Problem& P = L.P;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ncb = L.ncb;
  const int cb = blockIdx.x % ncb, rt = blockIdx.x / ncb;
  unsigned int* const bar = L.bar + rt * kBarWords;  // this replica tile's
  const int n = P.n, npad = P.npad, R = P.R, rpad = L.rpad;
  const int kblocks = npad / C::kSpinsPerKB;
  const int t_begin = L.t_begin, t_end = L.t_begin + L.sweeps;
  const bool epi = warp >= 2;
  const int ew = warp - 2;             // epilogue warp 0..15
  const int quad = warp & 3;           // TMEM lane quadrant of this warp
  const int grp = epi ? ew >> 2 : 0;   // column group 0..3 (kSPT spins each)
  const int row = quad * 32 + lane;    // replica row inside the tile
  const int rl = rt * 128 + row;       // replica row inside this launch's images
  const int r = L.rbase + rl;          // replica index
  const int col0 = cb * NT + grp * kSPT;  // first spin of this thread's kSPT
  const bool row_valid = epi && r < R;
  const bool warp_active = epi && (L.rbase + rt * 128 + quad * 32) < R && col0 < n;
  const int valid = n - col0;            // spins of the kSPT that exist
  const uint32_t full_mask = kSPT == 32 ? 0xFFFFFFFFu : ((1u << (kSPT & 31)) - 1u);
  const uint32_t vmask = valid >= kSPT ? full_mask : (valid > 0 ? (1u << valid) - 1u : 0u);

  const uint32_t bar_full0 = smem_u32(&bars[0]);          // a stage's spins and couplings
  const uint32_t bar_empty0 = smem_u32(&bars[kStages]);
  const uint32_t bar_done = smem_u32(&bars[2 * kStages]);  // a sweep's MMAs
  const uint32_t bar_jres = bar_done + 8;                          // resident couplings
  const uint32_t bar_tab = bar_done + 16;                          // the step's table

  if (warp == 1) {
    tmem_alloc(smem_u32(sTmem), C::kTmemCols);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(bar_full0 + 8 * s, kEpiWarps + (FP4 ? 0 : 1));
      mbar_init(bar_empty0 + 8 * s, 1);
    }
    mbar_init(bar_done, 1);
    mbar_init(bar_jres, 1);
    mbar_init(bar_tab, 1);
    fence_mbar_init();
  }
  for (int k = tid; k < NT; k += kThreads) {
    const int i = cb * NT + k;
    if constexpr (REAL)
      sH[k] = __float_as_uint((P.hf != nullptr && i < n) ? P.hf[i] : 0.0f);
    else
      sH[k] = static_cast<uint32_t>((P.h != nullptr && i < n) ? P.h[i] : 0);
  }
  if constexpr (REAL)
    for (int k = tid; k < 4096; k += kThreads) sZ[k] = P.zlev[k];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *sTmem;
  if constexpr (FP4) {
    // Resident couplings: the CTA's column block (NT rows x all K-blocks, contiguous in the
    // E2M1 image) arrives once, in copies of up to 32 KB on one barrier.
    if (tid == 0) {
      const uint8_t* src = L.j4 + static_cast<size_t>(cb) * jres_bytes;
      mbar_expect_tx(bar_jres, jres_bytes);
      for (int o = 0; o < jres_bytes; o += 32768)
        bulk_g2s(smem_u32(sJ + o), src + o, jres_bytes - o < 32768 ? jres_bytes - o : 32768, bar_jres);
    }
    // Unit scale factors (UE8M0 127 = 2^0) in every TMEM column after the accumulator, so
    // whatever layout the block-scaled MMA reads them in, each scale is 1.
    if (epi && grp == 0) {
#pragma unroll
      for (int c = 0; c < NT; c += 32)
        tmem_fill32(tmem + (static_cast<uint32_t>(quad * 32) << 16) + NT + c, 0x7F7F7F7Fu);
      tmem_wait_st();
    }
    tc_fence_before();
  }

  // ---- per-thread state: this replica's kSPT spins ------------------------------------
  uint32_t cur = 0, best = 0;
  EAcc best_E;
  if constexpr (REAL)
    best_E = FLT_MAX;
  else
    best_E = INT_MAX;
  int best_t = -1, first_hit = -1;
  const int half_words = P.words * 2;  // 16-bit chunks per row in the caller's bit arrays
  const int chunk = col0 >> 4;
  const uint16_t* cur_in = reinterpret_cast<const uint16_t*>(P.cur_bits);
  const uint16_t* best_in = reinterpret_cast<const uint16_t*>(P.best_bits);
  if (row_valid) {
#pragma unroll
    for (int c = 0; c < kChunks; ++c)
      if (chunk + c < half_words) {
        const size_t o = static_cast<size_t>(r) * half_words + chunk + c;
        cur |= static_cast<uint32_t>(cur_in[o]) << (16 * c);
        if (L.cont) best |= static_cast<uint32_t>(best_in[o]) << (16 * c);
      }
    if (L.cont) {
      best_E = static_cast<EAcc>(P.best_E[r]);
      best_t = P.best_t[r];
      first_hit = P.first_hit[r];
    }
  }
  if (!L.cont) best = cur;
  const bool has_target = P.has_target != 0;

  // Bit image of s(t): this thread's spins (the rows of the tile, the CTA's NT spins).
  const size_t tile_words = static_cast<size_t>(npad / 32) * 128;
  auto write_image = [&](uint32_t* img, uint32_t bits) {
    if (!epi) return;
    uint32_t* word = img + rt * tile_words + static_cast<size_t>(col0 >> 5) * 128 + row;
    if constexpr (kSPT == 32)
      *word = pack_spins16<OP>(bits & 0xFFFFu) | (pack_spins16<OP>(bits >> 16) << 16);
    else
      reinterpret_cast<uint16_t*>(word)[(col0 >> 4) & 1] = static_cast<uint16_t>(pack_spins16<OP>(bits));
  };
  bool aborted = false;  // on every thread of the role that gave up

  {
    const uint32_t idesc = REAL ? idesc_bf16(128, NT) : (FP4 ? idesc_mxf4(128, NT) : idesc_e4m3(128, NT));
    const int nst = (kblocks + kPB - 1) / kPB;  // ring stages of a sweep
    // Stages used so far, the same count in every role: stage g lies in slot g % kStages.
    uint32_t gs = 0;
    // K-block at position p of a sweep: in order, or pair by pair from the end
    auto kb_at = [&](int p, bool rev) {
      if (!rev) return p;
      const int pairs = (kblocks + KPS - 1) / KPS, first = kblocks - (pairs - 1) * KPS;
      return p < first ? (pairs - 1) * KPS + p : (pairs - 2 - (p - first) / KPS) * KPS + (p - first) % KPS;
    };
    // Whether slot of stage g may be filled (bounded wait for the MMAs of its last use).
    auto slot_free = [&](uint32_t g) -> bool {
      return __all_sync(0xFFFFFFFFu, g < kStages || mbar_wait_fast(bar_empty0 + 8 * (g % kStages),
                                                                   (g / kStages - 1) & 1, L.wait_ns));
    };
    // Producer (warp 0, converged, one elected lane): the coupling rows of the column block.  They
    // do not depend on the spins, so it runs ahead into the next sweep as slots become free.
    auto produce = [&](bool rev) -> bool {
      // Coupling images of n > 256 are chunk-major: 16 KB blocks of 128 rows x one K-block,
      // ordered [row block][K-block], so consecutive K-blocks of a 128-row column block are
      // one copy; a 64-row column block is half of each 16 KB block (one copy per K-block).
      const uint8_t* b_src = P.jimg + static_cast<size_t>(NT == 128 ? cb : cb >> 1) * kblocks * 16384 +
                             (NT == 128 ? 0 : (cb & 1) * 8192);
      for (int si = 0; si < nst; ++si, ++gs) {
        const int p0 = si * kPB, nk = kblocks - p0 < kPB ? kblocks - p0 : kPB;
        if (!slot_free(gs)) return false;
        const uint32_t slot = gs % kStages;
        if (elect_one()) {
          const uint32_t full = bar_full0 + 8 * slot;
          mbar_expect_tx(full, nk * kBBytes);
          for (int j = 0; j < nk;) {
            const int kb = kb_at(p0 + j, rev);
            int run = 1;
            if (NT == 128)
              while (j + run < nk && kb_at(p0 + j + run, rev) == kb + run) ++run;
            bulk_g2s(smem_u32(sB) + (slot * kPB + j) * kBBytes, b_src + static_cast<size_t>(kb) * 16384,
                     run * kBBytes, full);
            j += run;
          }
        }
        __syncwarp();
      }
      return true;
    };
    // Epilogue warps: the tile's spins from the bit image into tensor memory, K-block `grp` of
    // every stage into this warp's lane quadrant.  The next stage's words are in flight meanwhile (more
    // stages ahead, 2 to 8, measured the same or slower).
    auto expand = [&](const uint32_t* img, bool rev) -> bool {
      const uint32_t* src = img + rt * tile_words + row;
      uint32_t w[kWPK];
      auto fetch = [&](int p) {
        if (p >= kblocks) return;
        const uint32_t* at = src + static_cast<size_t>(kb_at(p, rev)) * kWPK * 128;
#pragma unroll
        for (int k = 0; k < kWPK; ++k) w[k] = __ldcg(at + k * 128);
      };
      fetch(grp);
      for (int p = grp; p - grp < kblocks; p += kPB, ++gs) {
        if (!slot_free(gs)) return false;
        tc_fence_after();
        const uint32_t slot = gs % kStages;
        if (p < kblocks) {
          const uint32_t ta = tmem + (static_cast<uint32_t>(quad * 32) << 16) + C::kTmemA +
                              (slot * kPB + grp) * kACols;
          constexpr int kRegs = 16 / kWPK;  // operand registers of a 16-spin half
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            uint32_t v[16];
#pragma unroll
            for (int k = 0; k < kWPK; ++k) {
              const int hw = i * kWPK + k;  // half word of the K-block
              expand_spins16<OP>(w[hw >> 1], hw & 1, v + k * kRegs);
            }
            tmem_st16(ta + 16 * i, v);
          }
          fetch(p + kPB);
          tmem_wait_st();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_full0 + 8 * slot);
      }
      return true;
    };
    // MMA issuer (warp 1, converged, one elected lane): D = S_tile x J_block^T, stage by stage as
    // spins and couplings land; it never waits for an MMA to finish, only for data.  Each MMA
    // consumes 32 bytes of K (32 FP8, 16 BF16 or 64 E2M1 values).
    auto multiply = [&](bool rev) -> bool {
      const uint64_t b_desc = sw128_desc(smem_u32(FP4 ? sJ : sB));
      for (int si = 0; si < nst; ++si, ++gs) {
        const int p0 = si * kPB, nk = kblocks - p0 < kPB ? kblocks - p0 : kPB;
        const uint32_t slot = gs % kStages;
        if (!__all_sync(0xFFFFFFFFu, mbar_wait_fast(bar_full0 + 8 * slot, (gs / kStages) & 1, L.wait_ns)))
          return false;
        tc_fence_after();
        if (elect_one()) {
          const uint32_t a0 = tmem + C::kTmemA + slot * kPB * kACols;
#pragma unroll
          for (int j = 0; j < kPB; ++j)
            if (j < nk) {
              const uint64_t bj = b_desc + (FP4 ? kb_at(p0 + j, rev) * (NT * 128 >> 4)
                                                : (slot * kPB + j) * (kBBytes >> 4));
#pragma unroll
              for (int ks = 0; ks < 4; ++ks) {
                const uint32_t acc = (si > 0 || j > 0 || ks > 0) ? 1u : 0u;
                if constexpr (REAL)
                  mma_bf16_ta(tmem, a0 + j * kACols + 8 * ks, bj + 2 * ks, idesc, acc);
                else if constexpr (FP4)
                  mma_mxf4_ta(tmem, a0 + j * kACols + 8 * ks, bj + 2 * ks, idesc, tmem + NT, tmem + NT, acc);
                else
                  mma_f8_ta(tmem, a0 + j * kACols + 8 * ks, bj + 2 * ks, idesc, acc);
              }
            }
          if (si + 1 == nst) mma_commit(bar_done);
          mma_commit(bar_empty0 + 8 * slot);
        }
        __syncwarp();
      }
      return true;
    };
    auto give_up = [&]() {
      aborted = true;
      if (lane == 0) {
        atomicOr(L.err, kDevErrTimeout);
        tile_abort(bar);
      }
    };

    // Best / first-hit bookkeeping of state `state` = s(tt) from its replica energy, complete
    // since the barrier that ended sweep tt.  Returns that energy.
    EAcc* energy = reinterpret_cast<EAcc*>(L.energy);
    // L2 read: the accumulator was written by other SMs during sweep tt.
    auto summed = [&](int tt) { return __ldcg(&energy[((tt - t_begin) % 3) * rpad + rl]); };
    auto track = [&](int tt, uint32_t state, EAcc etot) -> EAcc {
      EAcc E;
      bool hit;
      if constexpr (REAL) {
        E = -0.5f * etot;
        hit = static_cast<double>(E) <= P.target_f;
      } else {
        E = -(etot / 2);  // s^T J s is even for symmetric integer J with zero diagonal
        hit = static_cast<long long>(E) <= P.target;
      }
      if (E < best_E) {
        best_E = E;
        best_t = tt;
        best = state;
      }
      if (has_target && first_hit < 0 && hit) first_hit = tt;
      return E;
    };

    if (warp == 0) {
      if constexpr (!FP4)
        for (int t = t_begin; t <= t_end; ++t) {
          // Injected fault: nothing is loaded in the first sweep, so the MMA warp's first
          // wait cannot complete.
          if (L.inject == 1 && t == t_begin) break;
          if (!produce(kRev && (t & 1))) {
            give_up();
            break;
          }
        }
    } else if (warp == 1) {
      bool ok = !FP4 || __all_sync(0xFFFFFFFFu, mbar_wait_fast(bar_jres, 0, L.wait_ns));
      for (int t = t_begin; t <= t_end && ok; ++t) ok = multiply(kRev && (t & 1));
      if (!ok) give_up();
    } else {  // ---- epilogue warps
    unsigned long long bar_target = ncb;  // counter value that completes the next barrier
    write_image(reinterpret_cast<uint32_t*>(L.s_img[0]), cur & vmask);
    aborted = !tile_barrier(bar, bar_target, L.err, sFlag, L.wait_ns);
    int cur_img = 0;
    uint32_t done_phase = 0;
    uint32_t prev = 0;  // s(t-1) of this thread's spins, until its energy has been tracked
    for (int t = t_begin; t <= t_end && !aborted; ++t) {
      const bool last = t == t_end;
      // The step's table (the last step's reads ended before the barrier).
      if (!REAL && tab_smem && !last && tid == 64) {
        mbar_expect_tx(bar_tab, P.stride_words * 4);
        bulk_g2s(smem_u32(sTab), P.thr + static_cast<size_t>(t) * P.stride_words, P.stride_words * 4, bar_tab);
      }
      // Zero the energy buffer that sweep t+1 will accumulate into (see header).
      if (cb == 0 && grp == 0) __stcg(&energy[((t - t_begin + 1) % 3) * rpad + rl], EAcc(0));
      EAcc eacc = 0;
      uint32_t nxt = 0;
      {
        const EAcc etot = t > t_begin ? summed(t - 1) : EAcc(0);
        bool ok = (L.inject == 1 && t == t_begin) || expand(reinterpret_cast<const uint32_t*>(L.s_img[cur_img]), kRev && (t & 1));
        // While the last MMAs run: the bookkeeping of s(t-1), whose energy the last barrier
        // completed.
        if (t > t_begin) track(t - 1, prev, etot);
        // The sweep's noise while the MMAs run: draws (integer couplings) or xi s + eta z (real).
        uint32_t rw[kSPT / 2];
        float ns[REAL ? kSPT : 1];
        float b = 0.0f, eta = 0.0f;
        if (warp_active && !last) {
          if constexpr (REAL) {
            b = P.sched_b[t];
            eta = P.sched_eta[t];
          }
#pragma unroll
          for (int k = 0; k < kSPT / 8; ++k) {
            const PhiloxOut o = philox4x32_10_rk(static_cast<uint32_t>((col0 >> 3) + k), static_cast<uint32_t>(r),
                                                 static_cast<uint32_t>(t), P.q, L.round_keys);
            rw[4 * k] = o.x0, rw[4 * k + 1] = o.x1, rw[4 * k + 2] = o.x2, rw[4 * k + 3] = o.x3;
          }
          if (REAL && P.act == 0)
#pragma unroll
            for (int e = 0; e < (REAL ? kSPT : 0); ++e) {
              const uint32_t word = rw[e >> 1];
              const uint32_t key = (e & 1) ? (word >> 20) : ((word >> 4) & 0xFFFu);
              ns[e] = __fmaf_rn(eta, sZ[key], ((cur >> e) & 1u) ? P.xi : -P.xi);
            }
        }
        ok = __all_sync(0xFFFFFFFFu, ok && mbar_wait_fast(bar_done, done_phase, L.wait_ns) &&
                                         (REAL || !tab_smem || last ||
                                          mbar_wait_fast(bar_tab, static_cast<uint32_t>(t - t_begin) & 1, L.wait_ns)));
        if (!ok && lane == 0) {
          atomicOr(L.err, kDevErrTimeout);
          tile_abort(bar);  // the barrier below returns false on every thread
        }
        tc_fence_after();
        if (warp_active && ok) {
          const bool dumps = REAL && P.fields_out != nullptr && t == t_begin && !last && row_valid;
          const uint32_t ta = tmem + (static_cast<uint32_t>(quad * 32) << 16) + grp * kSPT;
#pragma unroll
          for (int c = 0; c < kChunks; ++c) {
            uint32_t v[16];
            tmem_ld16(ta + 16 * c, v);
            tmem_wait_ld(v);
            const uint32_t cw16 = (cur >> (16 * c)) & 0xFFFFu;
            if constexpr (REAL) {
              float x[16];
#pragma unroll
              for (int e = 0; e < 16; ++e) {
                const float hv = __uint_as_float(sH[grp * kSPT + 16 * c + e]);
                x[e] = __fadd_rn(__uint_as_float(v[e]), hv);
                const float term = __fadd_rn(x[e], hv);
                eacc += ((cw16 >> e) & 1u) ? term : -term;
              }
              if (dumps)  // diagnostics: fields of the first sweep
#pragma unroll
                for (int e = 0; e < 16; ++e)
                  if (col0 + 16 * c + e < n) P.fields_out[static_cast<size_t>(r) * n + col0 + 16 * c + e] = x[e];
              if (!last) {
                float g[16], least = P.act == 0 ? 8.0f : 0.0f;
                const float margin = rule_margin(P.act, P.xi);
#pragma unroll
                for (int e = 0; e < 16; ++e) x[e] = __fmul_rn(b, x[e]);
                if (P.act == 0) {
#pragma unroll
                  for (int e = 0; e < 16; ++e) {
                    g[e] = __fadd_rn(tanh_approx(x[e]), ns[REAL ? 16 * c + e : 0]);
                    least = min_nan(least, fabsf(g[e]));
                  }
                }
                if (__any_sync(0xFFFFFFFFu, !(least > margin)))
                  settle_chunk<16>(g, x, static_cast<uint32_t>((col0 + 16 * c) >> 3), static_cast<uint32_t>(r),
                                   static_cast<uint32_t>(t), P.q, L.round_keys, cw16, margin, P.xi, eta, P.act,
                                   P.lut_levels, sZ);
                uint32_t neg = 0;
#pragma unroll
                for (int e = 15; e >= 0; --e) neg = __funnelshift_l(__float_as_uint(g[e]), neg, 1);
                nxt |= (~neg & 0xFFFFu) << (16 * c);
              }
            } else {
              // bits of (D + 1.5 * 2^23) + h = 0x4B400000 + I; the 16-bit threshold of (s, I) is
              // half s of the table's word I + imax, and key >= M <=> draw - 16 M >= 0
              uint32_t vb[16];
#pragma unroll
              for (int e = 0; e < 16; ++e) {
                const int hv = static_cast<int>(sH[grp * kSPT + 16 * c + e]);
                vb[e] = __float_as_uint(__fadd_rn(__uint_as_float(v[e]), kMagic)) + hv;
                const int term = static_cast<int>(vb[e] - kMagicBits) + hv;
                eacc += ((cw16 >> e) & 1u) ? term : -term;
              }
              if (!last) {
                uint32_t neg = 0;
                auto decide = [&](int e, uint32_t th) {
                  const uint32_t word = rw[8 * c + (e >> 1)];
                  const uint32_t d = (e & 1) ? (word >> 16) : (word & 0xFFFFu);
                  neg = __funnelshift_l(draw_below(d, th, e & 1), neg, 1);
                };
                if (tab_smem) {
                  const uint32_t tab_c = smem_u32(sTab) + 4u * static_cast<uint32_t>(P.imax) - 4u * kMagicBits;
#pragma unroll
                  for (int e = 15; e >= 0; --e) {
                    uint32_t th;
                    asm volatile("ld.shared.u16 %0, [%1];"
                                 : "=r"(th)
                                 : "r"(tab_c + 4u * vb[e] + 2u * ((cw16 >> e) & 1u)));
                    decide(e, th);
                  }
                } else {  // through L1
                  const uint16_t* tab16 = reinterpret_cast<const uint16_t*>(
                      P.thr + static_cast<size_t>(t) * P.stride_words + P.imax);
                  uint32_t th[16];
#pragma unroll
                  for (int e = 0; e < 16; ++e)
                    th[e] = __ldg(tab16 + 2 * static_cast<int>(vb[e] - kMagicBits) + static_cast<int>((cw16 >> e) & 1u));
#pragma unroll
                  for (int e = 15; e >= 0; --e) decide(e, th[e]);
                }
                nxt |= (~neg & 0xFFFFu) << (16 * c);
              }
            }
          }
          nxt &= vmask;
        }
        sRed[grp * 128 + row] = eacc;
      }
      done_phase ^= 1;
      if (!last) write_image(reinterpret_cast<uint32_t*>(L.s_img[cur_img ^ 1]), nxt);
      tc_fence_before();
      asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
      if (grp == 0) {
        const EAcc tot = sRed[row] + sRed[128 + row] + sRed[256 + row] + sRed[384 + row];
        atomicAdd(&energy[((t - t_begin) % 3) * rpad + rl], tot);
      }
      bar_target += ncb;
      aborted = !tile_barrier(bar, bar_target, L.err, sFlag, L.wait_ns);
      if (aborted) break;
      if (last) {
        const EAcc E = track(t, cur, summed(t));
        if (row_valid) {
#pragma unroll
          for (int c = 0; c < kChunks; ++c)
            if (chunk + c < half_words) {
              const size_t o = static_cast<size_t>(r) * half_words + chunk + c;
              reinterpret_cast<uint16_t*>(P.cur_bits)[o] = static_cast<uint16_t>(cur >> (16 * c));
              reinterpret_cast<uint16_t*>(P.best_bits)[o] = static_cast<uint16_t>(best >> (16 * c));
            }
          if (cb == 0 && grp == 0) {
            P.best_E[r] = static_cast<double>(best_E);
            P.best_t[r] = best_t;
            P.first_hit[r] = first_hit;
            P.final_E[r] = static_cast<double>(E);
          }
        }
      } else {
        prev = cur;
        cur = nxt;
      }
      cur_img ^= 1;
    }
    }
  }

  // A wait gave up: copies and MMAs in flight need microseconds; the other roles end on their own
  // bounded waits.
  if (aborted) __nanosleep(20000);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, C::kTmemCols);
}

template <int NT, int OP>
cudaError_t variant_setup(int smem, const void** fn, int* max_blocks) {
  *fn = reinterpret_cast<const void*>(sweep_big_kernel<NT, OP>);
  const int attr = OP == kBigFp4 ? kSmemBudget : BigCfg<NT, OP>::kSmem;
  cudaError_t e = cudaFuncSetAttribute(sweep_big_kernel<NT, OP>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, attr);
  if (e != cudaSuccess) return e;
  int per_sm = 0, dev = 0, sms = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sweep_big_kernel<NT, OP>, kThreads,
                                                    smem);
  if (e != cudaSuccess) return e;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  *max_blocks = resident_ctas(per_sm, BigCfg<NT, OP>::kTmemCols) * sms;
  return cudaSuccess;
}

cudaError_t variant(int nt, int op, int smem, const void** fn, int* max_blocks) {
  if (op == kBigFp4) return nt == 64 ? variant_setup<64, kBigFp4>(smem, fn, max_blocks)
                                     : cudaErrorInvalidValue;
  const bool real = op == kBigBf16;
  if (op != kBigFp8 && op != kBigBf16) return cudaErrorInvalidValue;
  if (nt == 64) return real ? variant_setup<64, kBigBf16>(smem, fn, max_blocks)
                            : variant_setup<64, kBigFp8>(smem, fn, max_blocks);
  if (nt == 128) return real ? variant_setup<128, kBigBf16>(smem, fn, max_blocks)
                             : variant_setup<128, kBigFp8>(smem, fn, max_blocks);
  return cudaErrorInvalidValue;
}

template <int NT, int OP>
BigSmem streamed_plan(int stride_words) {
  BigSmem out;
  out.ok = true;
  out.tab_smem = OP == kBigFp8 && stride_words <= BigCfg<NT, OP>::kTab ? 1 : 0;
  out.bytes = BigCfg<NT, OP>::kSmem;
  return out;
}

}  // namespace

BigSmem sweep_big_smem(int nt, int op, int npad, int stride_words) {
  if (op == kBigFp4) return nt == 64 ? fp4_plan(npad, stride_words) : BigSmem{};
  if (op == kBigFp8) {
    if (nt == 64) return streamed_plan<64, kBigFp8>(stride_words);
    if (nt == 128) return streamed_plan<128, kBigFp8>(stride_words);
  } else if (op == kBigBf16) {
    if (nt == 64) return streamed_plan<64, kBigBf16>(stride_words);
    if (nt == 128) return streamed_plan<128, kBigBf16>(stride_words);
  }
  return BigSmem{};
}

int sweep_big_max_blocks(int nt, int op, int npad, int stride_words) {
  const BigSmem plan = sweep_big_smem(nt, op, npad, stride_words);
  if (!plan.ok) return 0;
  const void* fn = nullptr;
  int blocks = 0;
  return variant(nt, op, plan.bytes, &fn, &blocks) == cudaSuccess ? blocks : 0;
}

cudaError_t launch_sweep_big(const BigLaunch& L, int nt, int op, int blocks, cudaStream_t st) {
  const BigSmem plan = sweep_big_smem(nt, op, L.P.npad, L.P.stride_words);
  if (!plan.ok || L.tab_smem != plan.tab_smem) return cudaErrorInvalidValue;
  if (op == kBigFp4 && L.j4 == nullptr) return cudaErrorInvalidValue;
  const void* fn = nullptr;
  int cap = 0;
  cudaError_t e = variant(nt, op, plan.bytes, &fn, &cap);
  if (e != cudaSuccess) return e;
  if (blocks > cap) return cudaErrorCooperativeLaunchTooLarge;
  void* args[] = {const_cast<BigLaunch*>(&L)};
  e = cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(kThreads), args, plan.bytes, st);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace pim
