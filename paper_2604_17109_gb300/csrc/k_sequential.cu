// Conventional PIM with sequential updates (Eq. 3; Box 1, orange path), the baseline the
// fully parallel loop is compared with.  One warp per replica; sweep k updates spins
// i = 0 .. n-1 one after another, each from the field of the current state, with the 12-bit key of
// draw (i>>3, r, k, q) and the threshold table of schedule entry k (the same exact decisions as
// the parallel path); a flip adds 2 s_i' J_i (row i of J = column i) to the fields.
//
// The chain of n dependent steps bounds a replica, so the warp walks it flip by flip instead of
// spin by spin: spins are taken 32 at a time, one per lane; every lane decides its spin from the
// current fields; the lanes before the first one that flips keep their decision (nothing before
// them changes), that flip is applied to all fields, and the lanes after it decide again.  That is
// the sequential order exactly, in (flips + n / 32) rounds of about 120 cycles a sweep rather than
// n steps of 290.  Fields live in registers (n <= 1024, else shared memory, where registers are kept
// to 64 a thread so that 32 replicas fit an SM), spins as bit words, the draws, the sweep's table (copied
// ahead) and J, where they fit, in shared memory.
// Measured (GB300, us per sweep, spin by spin with J in L2 before): SK n = 200 27.9 -> 2.3 (256
// replicas), 106 -> 9.7 (8192); n = 400 57.6 -> 4.7; n = 1000 369 -> 70.  Runs of 12 sweeps, fields of the
// first state included: n = 513 480 -> 162 (12000 replicas), n = 1024 1167 -> 1026 (12000), n = 1025 319 ->
// 100 (256), 1215 -> 613 (12000), n = 2000 961 -> 281 (256), 2307 -> 960 (6000).
//
// Energies E = -1/2 sum_i s_i (I_i + h_i) are evaluated on the state at the start of every
// sweep and on the final state, with the best-state / first-hit bookkeeping of the
// parallel kernels.  No waits between warps once J is loaded: every warp runs on its own.
#include <climits>

#include "kernels.h"
#include "philox.cuh"
#include "sm100_ptx.cuh"

namespace pim {
namespace {

constexpr int kMaxWarps = 8;                // replicas per block
constexpr int kSmemBudget = 227 * 1024;
constexpr int kTabWordsMax = 4096;          // tables up to this size are staged in shared memory

__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

__host__ __device__ inline int round16(int x) { return (x + 15) & ~15; }

// Draws of a warp in shared memory: a sweep's, or with the fields in shared memory beside them the next
// 256 spins' (one Philox block per lane).
__host__ __device__ inline int draw_bytes(int n, int kf) { return kf == 0 ? 512 : round16((n + 7) / 8 * 16); }

// Shared memory of a launch: J (when jsm), then per warp two tables (when tsm), the draws, the spin
// words and, for KF = 0, the fields.
struct SeqPlan {
  int kf = 0;      // 32-spin field registers per lane (0: fields in shared memory)
  int warps = 1;   // replicas per block
  int jsm = 0, tsm = 0;
  int warp_bytes = 0, bytes = 0;
};

SeqPlan seq_plan(int n, int words, int stride_words, int replicas, int sms) {
  SeqPlan p;
  p.kf = n <= 128 ? 4 : n <= 256 ? 8 : n <= 512 ? 16 : n <= 640 ? 20 : n <= 768 ? 24 : n <= 896 ? 28 : n <= 1024 ? 32 : 0;
  const int base = draw_bytes(n, p.kf) + round16(words * 4) + (p.kf == 0 ? round16(n * 4) : 0);
  const int tab = 2 * stride_words * 4;
  // spread the replicas over the SMs first, then share a block between up to kMaxWarps
  const int want = (replicas + sms - 1) / sms;
  p.warps = want < 1 ? 1 : want > kMaxWarps ? kMaxWarps : want;
  p.tsm = stride_words <= kTabWordsMax && base + tab <= kSmemBudget ? 1 : 0;
  if (p.kf == 0 || p.kf > 16) {
    // Without J in shared memory a replica waits for rows of J from L2, and other warps hide that:
    // tables stay out where they would keep some of the SM's replicas from running beside the others
    // (n = 1025 x 2048 replicas, 867 us per sweep with them, 679 without; n = 1500 x 6000 4320, 2471).
    if (want > kSmemBudget / (base + tab)) p.tsm = 0;
    // Registers for 1024 fields leave room for eight or nine such warps: two blocks of four let a
    // block start when four have ended (n = 1024 x 2048 325 -> 291 us per sweep).
    if (p.kf == 32 && want > kMaxWarps) p.warps = kMaxWarps / 2;
  }
  p.warp_bytes = base + (p.tsm ? tab : 0);
  const int jbytes = p.kf > 0 && p.kf <= 16 ? round16(n * n) : kSmemBudget;
  // J beside fewer than half of a block's replicas costs more than it saves (n = 470, one replica beside
  // J: 1962 us per sweep at 12000 replicas; n = 500, J in L2: 296).
  p.jsm = (kSmemBudget - jbytes) / p.warp_bytes >= (p.warps < kMaxWarps / 2 ? p.warps : kMaxWarps / 2) ? 1 : 0;
  while (p.warps > 1 && (p.jsm ? jbytes : 0) + p.warps * p.warp_bytes > kSmemBudget) --p.warps;
  p.bytes = (p.jsm ? jbytes : 0) + p.warps * p.warp_bytes;
  return p;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// JSM: J in shared memory.
template <int KF, bool JSM>
__global__ void __launch_bounds__(kMaxWarps * 32, KF == 0 ? 4 : 0) sequential_kernel(const __grid_constant__ SeqLaunch L,
                                                                    const SeqPlan plan) {
  constexpr int K = KF > 0 ? KF : 1;
  extern __shared__ __align__(16) uint8_t smem_seq[];
  const Problem& P = L.P;
  const int n = P.n, words = P.words, imax = P.imax, stride = P.stride_words;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.x * plan.warps + warp;
  const int8_t* J = JSM ? reinterpret_cast<const int8_t*>(smem_seq) : P.j8;
  uint8_t* mine = smem_seq + (JSM ? round16(n * n) : 0) + warp * plan.warp_bytes;
  if constexpr (JSM) {
    const int total = n * n;
    const uint4* src = reinterpret_cast<const uint4*>(P.j8);
    uint4* dst = reinterpret_cast<uint4*>(smem_seq);
    for (int k = threadIdx.x; k < total / 16; k += blockDim.x) dst[k] = __ldg(src + k);
    for (int k = total / 16 * 16 + threadIdx.x; k < total; k += blockDim.x)
      smem_seq[k] = static_cast<uint8_t>(P.j8[k]);
    __syncthreads();
  }
  if (r >= P.R) return;  // a whole warp; no block-level synchronisation from here on
  uint32_t* tabs = reinterpret_cast<uint32_t*>(mine);                  // [2][stride] when tsm
  uint16_t* draws = reinterpret_cast<uint16_t*>(mine + (plan.tsm ? 2 * stride * 4 : 0));
  uint32_t* sw = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(draws) + draw_bytes(n, KF));
  int* sI = reinterpret_cast<int*>(reinterpret_cast<uint8_t*>(sw) + round16(words * 4));  // KF = 0
  const int nblk32 = (n + 31) >> 5;
  uint32_t* cur_io = P.cur_bits + static_cast<size_t>(r) * words;
  uint32_t* best_io = P.best_bits + static_cast<size_t>(r) * words;
  const int32_t* h = P.h;

  for (int w = lane; w < words; w += 32) sw[w] = cur_io[w];
  __syncwarp();
  // Field of spin 32 k + lane (lanes past n keep 0).
  int F[K];
#pragma unroll
  for (int k = 0; k < K; ++k) F[k] = 0;
  auto add_row = [&](int i, int d) {  // I += d * row i of J
    const int8_t* Ji = J + static_cast<size_t>(i) * n + lane;
    if constexpr (KF > 0) {
      int v[K];  // every load before the first use
#pragma unroll
      for (int k = 0; k < K; ++k) v[k] = 32 * k + lane < n ? (JSM ? Ji[32 * k] : __ldg(Ji + 32 * k)) : 0;
#pragma unroll
      for (int k = 0; k < K; ++k) F[k] += v[k] * d;
    } else {
      for (int j0 = 0; j0 < n; j0 += 512) {  // 16 loads in flight
        int v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = j0 + 32 * k + lane < n ? __ldg(Ji + j0 + 32 * k) : 0;
#pragma unroll
        for (int k = 0; k < 16; ++k)
          if (j0 + 32 * k + lane < n) sI[j0 + 32 * k + lane] += v[k] * d;
      }
    }
  };
  // Fields of the starting state, row by row (J is symmetric); 256 at a time in registers for KF = 0.
  if constexpr (KF > 0) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (32 * k + lane < n && h) F[k] = h[32 * k + lane];
#pragma unroll 4
    for (int i = 0; i < n; ++i) add_row(i, ((sw[i >> 5] >> (i & 31)) & 1u) ? 1 : -1);
  } else {
    for (int j0 = 0; j0 < n; j0 += 256) {
      int sum[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) sum[k] = h && j0 + 32 * k + lane < n ? h[j0 + 32 * k + lane] : 0;
#pragma unroll 4
      for (int i = 0; i < n; ++i) {
        const int8_t* Ji = J + static_cast<size_t>(i) * n + j0 + lane;
        const int d = ((sw[i >> 5] >> (i & 31)) & 1u) ? 1 : -1;
#pragma unroll
        for (int k = 0; k < 8; ++k) sum[k] += (j0 + 32 * k + lane < n ? __ldg(Ji + 32 * k) : 0) * d;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (j0 + 32 * k + lane < n) sI[j0 + 32 * k + lane] = sum[k];
    }
  }

  long long best_E = LLONG_MAX;
  int best_t = -1, first_hit = -1;
  if (L.cont) {
    best_E = static_cast<long long>(P.best_E[r]);
    best_t = P.best_t[r];
    first_hit = P.first_hit[r];
  }
  // E(s) on the current state, bookkeeping at schedule index t; returns E.
  auto evaluate = [&](int t) -> long long {
    long long acc = 0;
    if constexpr (KF > 0) {
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (32 * k + lane < n) {
          const long long term = F[k] + (h ? h[32 * k + lane] : 0);
          acc += ((sw[k] >> lane) & 1u) ? term : -term;
        }
    } else {
      for (int j = lane; j < n; j += 32) {
        const long long term = static_cast<long long>(sI[j]) + (h ? h[j] : 0);
        acc += ((sw[j >> 5] >> (j & 31)) & 1u) ? term : -term;
      }
    }
    const long long E = -(warp_sum(acc) / 2);
    if (E < best_E) {
      best_E = E;
      best_t = t;
      for (int w = lane; w < words; w += 32) best_io[w] = sw[w];
    }
    if (P.has_target && first_hit < 0 && E <= P.target) first_hit = t;
    return E;
  };
  auto fetch_table = [&](int t) {  // asynchronously, into the table buffer of t
    const uint32_t dst = smem_u32(tabs + (t & 1) * stride);
    const uint32_t* src = P.thr + static_cast<size_t>(t) * stride;
    for (int k = lane; k < stride / 4; k += 32) cp_async16(dst + 16 * k, src + 4 * k);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  const int t_end = L.t_begin + L.sweeps;
  if (plan.tsm && L.t_begin < t_end) fetch_table(L.t_begin);
  for (int t = L.t_begin; t < t_end; ++t) {
    evaluate(t);
    __syncwarp();  // the last sweep's draws and table have been read
    auto draw8 = [&](int b, int at) {  // Philox block b, in spin order
      const PhiloxOut o = philox4x32_10_rk(static_cast<uint32_t>(b), static_cast<uint32_t>(r),
                                           static_cast<uint32_t>(t), P.q, L.round_keys);
      reinterpret_cast<uint4*>(draws)[at] = make_uint4(o.x0, o.x1, o.x2, o.x3);
    };
    for (int b = lane; KF > 0 && b < (n + 7) / 8; b += 32) draw8(b, b);
    const uint32_t* tab = P.thr + static_cast<size_t>(t) * stride;
    if (plan.tsm) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      if (t + 1 < t_end) fetch_table(t + 1);
      tab = tabs + (t & 1) * stride;
    }
    __syncwarp();
    // spins 32 k .. 32 k + 31, this lane's field in f (and its register / shared copy kept)
    auto block32 = [&](int k, auto field) {
      const int i = 32 * k + lane;
      uint32_t word = sw[k];
      if (KF == 0 && (k & 7) == 0) {
        __syncwarp();  // the last 256 have been read
        if (8 * (4 * k + lane) < n) draw8(4 * k + lane, lane);
        __syncwarp();
      }
      const int key = i < n ? draws[KF == 0 ? i & 255 : i] >> 4 : 0;
      uint32_t todo = n - 32 * k >= 32 ? 0xFFFFFFFFu : (1u << (n - 32 * k)) - 1u;
      for (;;) {
        const uint32_t up = (word >> lane) & 1u;
        const uint32_t w = tab[field() + imax];
        const int th = static_cast<int>(up ? (w >> 16) : (w & 0xFFFFu));
        const uint32_t flips = __ballot_sync(0xFFFFFFFFu, (key >= th ? 1u : 0u) != up) & todo;
        if (flips == 0) break;
        const int l = __ffs(static_cast<int>(flips)) - 1;
        add_row(32 * k + l, ((word >> l) & 1u) ? -2 : 2);
        word ^= 1u << l;
        todo &= l == 31 ? 0u : 0xFFFFFFFEu << l;  // the spins after it decide again
        if constexpr (KF == 0) __syncwarp();
      }
      __syncwarp();
      if (lane == 0) sw[k] = word;
    };
    if constexpr (KF > 0) {
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (k < nblk32) block32(k, [&]() { return F[k]; });
    } else {
      for (int k = 0; k < nblk32; ++k)
        block32(k, [&]() { return 32 * k + lane < n ? sI[32 * k + lane] : 0; });
    }
    __syncwarp();
  }
  const long long E = evaluate(t_end);
  for (int w = lane; w < words; w += 32) cur_io[w] = sw[w];
  if (lane == 0) {
    P.best_E[r] = static_cast<double>(best_E);
    P.best_t[r] = best_t;
    P.first_hit[r] = first_hit;
    P.final_E[r] = static_cast<double>(E);
  }
}

template <int KF, bool JSM>
cudaError_t launch_seq(const SeqLaunch& L, const SeqPlan& plan, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(sequential_kernel<KF, JSM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       plan.bytes);
  if (e != cudaSuccess) return e;
  const int blocks = (L.P.R + plan.warps - 1) / plan.warps;
  sequential_kernel<KF, JSM><<<blocks, plan.warps * 32, plan.bytes, st>>>(L, plan);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sequential(const SeqLaunch& L, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const SeqPlan plan = seq_plan(L.P.n, L.P.words, L.P.stride_words, L.P.R, sms);
  switch (plan.kf) {
    case 4: return plan.jsm ? launch_seq<4, true>(L, plan, st) : launch_seq<4, false>(L, plan, st);
    case 8: return plan.jsm ? launch_seq<8, true>(L, plan, st) : launch_seq<8, false>(L, plan, st);
    case 16: return plan.jsm ? launch_seq<16, true>(L, plan, st) : launch_seq<16, false>(L, plan, st);
    case 20: return launch_seq<20, false>(L, plan, st);
    case 24: return launch_seq<24, false>(L, plan, st);
    case 28: return launch_seq<28, false>(L, plan, st);
    case 32: return launch_seq<32, false>(L, plan, st);
    default: return launch_seq<0, false>(L, plan, st);
  }
}

}  // namespace pim
