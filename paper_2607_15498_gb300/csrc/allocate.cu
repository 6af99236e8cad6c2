// Step 2 — rank allocation (Sec. 3.2: min-max normalisation, Eq. 4 water-filling, Algorithm 1's
// water level) for every (sequence, layer), one thread-block cluster each.
//
// All float arithmetic is IEEE fp32 with explicitly rounded intrinsics (no contraction into FMA),
// so the ranks are a deterministic function of the salience bits:
//   s_hat = (s - min) / (max - min)            (1 if max == min, or in UNIFORM mode)
//   x     = fl(fl(lambda * s_hat) + r_min)
//   rank  = r_max if x >= r_max else max(r_min, floor(x))
// lambda is the largest finite fp32 value >= 0 whose ranks sum to at most B_c, searched over the
// fp32 bit patterns (the sum is non-decreasing in lambda).
//
// What bounds it: the chain of sums over all tokens, one after another. So each CTA of the cluster
// takes a contiguous share of the tokens, normalises it once into shared memory (the division is
// what a pass over the salience costs most), and each pass sums the ranks at 15 water levels at
// once, with one cluster barrier, instead of halving the bracket.
#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace vr {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kCand = 15;              // water levels per pass
static_assert(kWarps > kCand, "a warp adds the warps' sums of one level");
constexpr int kMaxCluster = 8;         // portable cluster size
constexpr int64_t kMaxCached = 49152;  // normalised saliences kept in shared memory (192 KB)

__device__ __forceinline__ float shat_of(float s, float mn, float den) {
  const float v = __fdiv_rn(__fsub_rn(s, mn), den);
  return v == v ? v : 0.f;   // NaN salience: rank r_min, as x = r_min gives
}

// floor(min(x, r_max)) + 0x4B000000 as an integer, x = fl(fl(lam * sh) + r_min) in [r_min, inf]: adding
// 2^23 with rounding toward minus infinity leaves floor(x) in the mantissa (x <= 128).
__device__ __forceinline__ uint32_t rank_bits(float lam, float sh, float r_min, float r_max) {
  const float x = fminf(__fadd_rn(__fmul_rn(lam, sh), r_min), r_max);
  return __float_as_uint(__fadd_rd(x, 8388608.f));
}
constexpr uint32_t kRankBias = 0x4B000000u;

__device__ __forceinline__ void warp_stats(float& mn, float& mx, float& sum) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
  }
}

__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Offset of the k-th of kCand levels around a guess whose error is expected within `reach` (in units of
// the bit pattern): none at the guess, then factors of four (two near the ends) on both sides.
__device__ __forceinline__ int64_t spread(int k, int64_t reach) {
  const int m = k - kCand / 2;
  const int a = m < 0 ? -m : m;
  const int64_t d = a == 0 ? 0 : reach >> (2 * (kCand / 2 - a));
  return m < 0 ? -d : d;
}

struct AllocSmem {
  float mm[kMaxCluster][3];                        // every CTA's min, max and sum
  long long tot[2][kMaxCluster][kCand + 1];        // every CTA's sums, by pass parity
  unsigned long long wsum[kCand][kWarps + 1];
  float fred[3][kWarps];
};

// grid (C B L) in clusters of C CTAs, one cluster for each (sequence, layer); CTA `rank` of it takes
// `share` tokens, the first `cached` of them held in the dynamic shared memory.
__global__ void __launch_bounds__(kThreads)
allocate_kernel(const float* __restrict__ sal, uint8_t* __restrict__ ranks,
                int64_t* __restrict__ realized, int32_t* __restrict__ dev_status, Shape s,
                int64_t share, int64_t cached) {
  extern __shared__ float sh_cache[];
  __shared__ AllocSmem sm;
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int64_t bl = blockIdx.x / C;
  const int64_t n = s.n_coded;
  const float* sl = sal ? sal + bl * n : nullptr;
  uint8_t* rk = ranks + bl * s.N;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t t0 = min(n, rank * share), cnt = min(n, t0 + share) - t0;   // this CTA's tokens

  // exact set: full rank
  if (rank == 0)
    for (int64_t t = n + tid; t < s.N; t += kThreads) rk[t] = (uint8_t)s.r_max;

  int mode_fixed = -1;    // -1: search, otherwise every coded token gets this rank
  if (n == 0) {
    mode_fixed = s.r_max;
  } else if ((int64_t)s.r_min * n > s.Bc) {
    mode_fixed = s.r_min;
    if (rank == 0 && tid == 0) raise_status(dev_status, VARRATE_FLOOR_BINDS);
  } else if (s.Bc >= (int64_t)s.r_max * n) {
    mode_fixed = s.r_max;
  } else if (sl == nullptr || s.mode == VARRATE_UNIFORM) {
    mode_fixed = (int)(s.Bc / n);   // all s_hat are 1: the largest lambda that fits gives every token floor(B_c / n)
  }
  if (mode_fixed >= 0) {   // uniform over the cluster: no barrier is skipped by part of it
    for (int64_t i = tid; i < cnt; i += kThreads) rk[t0 + i] = (uint8_t)mode_fixed;
    if (rank == 0 && tid == 0 && realized) realized[bl] = (int64_t)mode_fixed * n;
    return;
  }

  cluster.barrier_arrive();   // this CTA runs: the others may write its shared memory once they have waited
  // min / max over the coded set (exact in any order), and the sum, which only places the first levels
  float mn = INFINITY, mx = -INFINITY, sum = 0.f;
  for (int64_t i = tid; i < cnt; i += kThreads) {
    const float v = sl[t0 + i];
    if (i < cached) sh_cache[i] = v;
    mn = fminf(mn, v);
    mx = fmaxf(mx, v);
    sum += v;
  }
  warp_stats(mn, mx, sum);
  if (lane == 0) { sm.fred[0][warp] = mn; sm.fred[1][warp] = mx; sm.fred[2][warp] = sum; }
  __syncthreads();
  cluster.barrier_wait();     // every CTA of the cluster has started
  if (warp == 0) {
    mn = lane < kWarps ? sm.fred[0][lane] : INFINITY;
    mx = lane < kWarps ? sm.fred[1][lane] : -INFINITY;
    sum = lane < kWarps ? sm.fred[2][lane] : 0.f;
    warp_stats(mn, mx, sum);
    if (lane < C) {
      float* peer = cluster.map_shared_rank(&sm.mm[0][0], lane) + 3 * rank;
      peer[0] = mn;
      peer[1] = mx;
      peer[2] = sum;
    }
  }
  cluster.sync();
  mn = INFINITY; mx = -INFINITY; sum = 0.f;
  for (int c = 0; c < C; ++c) {
    mn = fminf(mn, sm.mm[c][0]);
    mx = fmaxf(mx, sm.mm[c][1]);
    sum += sm.mm[c][2];
  }
  if (!(mx > mn)) {   // a constant salience is the uniform case (the same for the whole cluster)
    const int r = (int)(s.Bc / n);
    for (int64_t i = tid; i < cnt; i += kThreads) rk[t0 + i] = (uint8_t)r;
    if (rank == 0 && tid == 0 && realized) realized[bl] = (int64_t)r * n;
    return;
  }
  const float den = __fsub_rn(mx, mn);
  // a thread normalises, and reads in every pass, the entries it loaded itself
  for (int64_t i = tid; i < min(cnt, cached); i += kThreads)   // entries past n_cached: normalised when read
    sh_cache[i] = shat_of(sh_cache[i], mn, den);
  const int n_cached = (int)min(cnt, cached);
  auto shat_far = [&](int64_t i) { return shat_of(sl[t0 + i], mn, den); };
  const float fmin_r = (float)s.r_min, fmax_r = (float)s.r_max;
  const bool wide = share >= (int64_t(1) << 24);   // a warp's sum may pass 32 bits

  // The answer is the largest b with total(b) <= B_c: total(lo) <= B_c < total(hi), where lo = 0 and the
  // pattern after the largest finite value stand in at the start. Any levels that bracket it closer give
  // the same answer. The first pass spreads them around the level that would spend the budget if no
  // rank met r_max; then the totals at both ends interpolate a guess (the total is close to linear in
  // a narrow bracket), and every third pass cuts the bracket evenly, to a sixteenth, which bounds the
  // number of passes whatever the salience looks like.
  uint32_t lo = 0, hi = 0x7F800000u;
  long long tot_lo = (long long)s.r_min * n, tot_hi = (long long)s.r_max * n;
  const float mean = (sum / (float)n - mn) / den;
  const float first = ((float)((double)s.Bc / (double)n) - fmin_r + 0.5f) / mean;
  for (int pass = 0; hi - lo > 1; ++pass) {
    const uint32_t span = hi - lo, step = (span + kCand) / (kCand + 1);
    const bool even = span <= kCand + 1 || (pass == 0 ? !(first > 0.f && first < 3e38f) : pass % 3 == 0);
    int64_t guess, reach;
    if (pass == 0) {
      guess = __float_as_uint(first);
      reach = 1 << 26;                       // eight octaves either way
    } else {
      guess = lo + (int64_t)((float)span * ((float)(s.Bc - tot_lo) / (float)(tot_hi - tot_lo)));
      reach = max(span / 4, 1u);
    }
    // level k of this pass, in (lo, hi), not decreasing in k: lane k forms it
    const int k0 = min(lane, kCand - 1);
    const int64_t near = guess + spread(k0, reach) + (k0 - kCand / 2);
    const uint32_t mine = even ? min(lo + step * (k0 + 1), hi - 1)
                               : (uint32_t)max((int64_t)lo + 1, min(near, (int64_t)hi - 1));
    float lam[kCand];
    uint32_t acc[kCand];
#pragma unroll
    for (int k = 0; k < kCand; ++k) {
      lam[k] = __uint_as_float(__shfl_sync(0xffffffffu, mine, k));
      acc[k] = 0;
    }
    uint32_t seen = 0;
    auto add = [&](float sh) {
#pragma unroll
      for (int k = 0; k < kCand; ++k) acc[k] += rank_bits(lam[k], sh, fmin_r, fmax_r);
      ++seen;
    };
    for (int i = tid; i < n_cached; i += kThreads) add(sh_cache[i]);
    for (int64_t i = n_cached + tid; i < cnt; i += kThreads) add(shat_far(i));
    // modulo 2^32 the sums themselves; lane k keeps that of level k
    unsigned long long w = 0;
    if (!wide) {
#pragma unroll
      for (int k = 0; k < kCand; ++k) {
        const uint32_t v = __reduce_add_sync(0xffffffffu, acc[k] - seen * kRankBias);
        if (lane == k) w = v;
      }
    } else {
#pragma unroll
      for (int k = 0; k < kCand; ++k) {
        const unsigned long long v = warp_sum64(acc[k] - seen * kRankBias);
        if (lane == k) w = v;
      }
    }
    if (lane < kCand) sm.wsum[lane][warp] = w;
    __syncthreads();
    if (warp < kCand) {
      w = lane < kWarps ? sm.wsum[warp][lane] : 0;
      w = wide ? warp_sum64(w) : __reduce_add_sync(0xffffffffu, (uint32_t)w);
      if (lane < C) *cluster.map_shared_rank(&sm.tot[pass & 1][rank][warp], lane) = (long long)w;
    }
    // also orders this pass's reads of wsum before the next pass's writes
    if (C > 1) cluster.sync(); else __syncthreads();
    long long total = 0;
    for (int c = 0; c < C; ++c) total += sm.tot[pass & 1][c][k0];
    // the levels do not decrease, so those that fit come first
    const int m = __popc(__ballot_sync(0xffffffffu, lane < kCand && total <= s.Bc));
    const uint32_t below = __shfl_sync(0xffffffffu, mine, max(m - 1, 0)), above = __shfl_sync(0xffffffffu, mine, min(m, kCand - 1));
    const long long t_below = __shfl_sync(0xffffffffu, total, max(m - 1, 0)), t_above = __shfl_sync(0xffffffffu, total, min(m, kCand - 1));
    if (m > 0) { lo = below; tot_lo = t_below; }
    if (m < kCand) { hi = above; tot_hi = t_above; }
  }

  const float lam = __uint_as_float(lo);
  for (int64_t i = tid; i < cnt; i += kThreads)
    rk[t0 + i] = (uint8_t)(rank_bits(lam, i < n_cached ? sh_cache[i] : shat_far(i), fmin_r, fmax_r) - kRankBias);
  if (rank == 0 && tid == 0 && realized) realized[bl] = tot_lo;
}

}  // namespace

int launch_allocate(const Shape& s, const float* sal, uint8_t* ranks, int64_t* realized,
                    int32_t* dev_status, int num_sms, cudaStream_t st) {
  // One CTA for every 2048 tokens or so (eight per thread), at most 8 to a pair, and no more than two CTAs
  // an SM over all pairs: a second wave would double the time.
  const int64_t pairs = (int64_t)s.B * s.L;
  int C = 1;
  while (C < kMaxCluster && (int64_t)C * 2048 < s.n_coded && C * pairs <= num_sms) C *= 2;
  const int64_t share = (s.n_coded + C - 1) / C;
  const int64_t cached = share < kMaxCached ? share : kMaxCached;
  const size_t smem = (size_t)cached * sizeof(float);
  if (smem > 32768 &&
      cudaFuncSetAttribute(allocate_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(kMaxCached * sizeof(float))) != cudaSuccess)
    return -1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(pairs * C));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = C; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const float* sp = s.mode == VARRATE_UNIFORM ? nullptr : sal;
  return cudaLaunchKernelEx(&cfg, allocate_kernel, sp, ranks, realized, dev_status, s, share, cached) == cudaSuccess
             ? 1 : -1;
}

}  // namespace vr
