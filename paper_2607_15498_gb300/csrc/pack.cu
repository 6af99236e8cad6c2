// Step 3 — rank-bucketed packing (layout tables) and projection (Algorithm 1's projection onto the
// basis; Eq. 5 with the anchor mean at 0).
//
// pack_tables (one thread-block cluster per (sequence, layer)):
//   count[r]           tokens of rank r;
//   base[r_min] = 0,   base[r + 1] = base[r] + r * pad8(count[r])  (element offsets);
//   pos[t]             stable position of t among the tokens of its rank;
//   perm[slot]         token of each slot, buckets in increasing rank.
// project (fp32; grid over slot chunks x (head, K/V) x (sequence, layer)): tokens are visited in
// bucketed slot order, so one coefficient of consecutive slots lands in consecutive addresses of
// its 8-slot group (layout: coef_offset in common.cuh); the same kernel zeroes the padding slots
// [count[r], pad8(count[r])) of every bucket.
#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace vr {

namespace {

constexpr int kMaxR = kHeadDim;  // r_max

constexpr int kTabThreads = 512;
constexpr int kTabWarps = kTabThreads / 32;
constexpr int kTabCluster = 8;   // portable cluster size
constexpr int kTabUnroll = 8;    // 32-token groups whose ranks are in flight together

struct TabSmem {
  int wcnt[kTabWarps][kMaxR + 1];         // tokens of each rank in each warp's share, then running positions
  int cta[kTabCluster][kMaxR + 2];        // every CTA's counts; the last entry says a rank was out of range
  int cnt[kMaxR + 1];
  int slot_start[kMaxR + 2];
  long long base[kMaxR + 2];
  int bad;
};

// grid (C B L) in clusters of C CTAs, one cluster per (sequence, layer). CTA `rank` takes `share`
// consecutive tokens and each of its warps a consecutive part of them, so a stable position is: tokens of
// that rank in earlier CTAs, in earlier warps, and before it in the warp. Counts cross the cluster once;
// the positions then need no barrier, only the warp's own running counts (match and popc within 32
// tokens). Bound by the latency of that chain: two passes over the ranks, one cluster barrier.
// One CTA that also zeroed the pads of all streams took, for 32768 tokens, 350 us with wide ranks (most of
// it the pads' 64-bit divisions, now the projection's) and 80 us with narrow ones; now 6.6 us (1 pair), 8.4
// us (32 pairs), and 17.6 us for 2 pairs of 131072 tokens.
__global__ void __launch_bounds__(kTabThreads)
pack_tables_kernel(const uint8_t* __restrict__ ranks, int32_t* __restrict__ bucket_count,
                   int64_t* __restrict__ bucket_base, int32_t* __restrict__ perm,
                   int32_t* __restrict__ pos, int32_t* __restrict__ dev_status, Shape s, int64_t share) {
  __shared__ TabSmem sm;
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int64_t bl = blockIdx.x / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t c0 = min(s.N, rank * share), c1 = min(s.N, c0 + share);
  const int64_t wshare = ((c1 - c0 + kTabThreads - 1) / kTabThreads) * 32;   // a multiple of 32 per warp
  const int64_t w0 = min(c1, c0 + warp * wshare), w1 = min(c1, w0 + wshare);
  const uint8_t* rk = ranks + bl * s.N;

  cluster.barrier_arrive();   // this CTA runs: the others may write its shared memory once they have waited
  for (int i = tid; i < kTabWarps * (kMaxR + 1); i += kTabThreads) (&sm.wcnt[0][0])[i] = 0;
  if (tid == 0) sm.bad = 0;
  __syncthreads();
  for (int64_t t = w0 + lane; t < w1; t += 32 * kTabUnroll) {
    int r[kTabUnroll];
#pragma unroll
    for (int u = 0; u < kTabUnroll; ++u) r[u] = t + 32 * u < w1 ? (int)rk[t + 32 * u] : -1;
#pragma unroll
    for (int u = 0; u < kTabUnroll; ++u) {
      if (r[u] < 0) continue;
      if (r[u] < s.r_min || r[u] > s.r_max) sm.bad = 1;
      else atomicAdd(&sm.wcnt[warp][r[u]], 1);
    }
  }
  __syncthreads();
  cluster.barrier_wait();     // every CTA of the cluster has started
  if (tid <= kMaxR + 1) {
    int v = tid > kMaxR ? sm.bad : 0;
    if (tid <= kMaxR) {
#pragma unroll
      for (int w = 0; w < kTabWarps; ++w) {
        const int x = sm.wcnt[w][tid];
        sm.wcnt[w][tid] = v;
        v += x;
      }
    }
    for (int c = 0; c < C; ++c) *cluster.map_shared_rank(&sm.cta[rank][tid], c) = v;
  }
  cluster.sync();
  int before = 0;   // tokens of rank tid in earlier CTAs
  if (tid <= kMaxR) {
    int total = 0;
    for (int c = 0; c < C; ++c) {
      if (c == rank) before = total;
      total += sm.cta[c][tid];
    }
    sm.cnt[tid] = total;
  }
  int bad = 0;
  for (int c = 0; c < C; ++c) bad |= sm.cta[c][kMaxR + 1];
  if (bad) {   // uniform over the cluster; no shared memory of another CTA is touched from here on
    if (rank == 0 && tid == 0) {
      raise_status(dev_status, VARRATE_ERR_CORRUPT);
      // poison the table so the projection and decode skip this (sequence, layer)
      bucket_base[bl * (kMaxR + 2) + kMaxR + 1] = INT64_MAX;
    }
    return;
  }
  __syncthreads();
  if (warp == 0) {   // bases and first slots: five ranks a lane, then a prefix over the lanes
    constexpr int kPer = 5;
    long long b = 0;
    int ss = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int r = lane * kPer + i;
      if (r <= kMaxR) {
        ss += sm.cnt[r];
        if (r >= s.r_min) b += (long long)r * pad8(sm.cnt[r]);
      }
    }
    long long ib = b;
    int is = ss;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long ob = __shfl_up_sync(0xffffffffu, ib, o);
      const int os = __shfl_up_sync(0xffffffffu, is, o);
      if (lane >= o) { ib += ob; is += os; }
    }
    ib -= b;
    is -= ss;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int r = lane * kPer + i;
      if (r <= kMaxR + 1) {
        sm.base[r] = ib;   // 0 up to r_min: nothing is counted before it
        sm.slot_start[r] = is;
      }
      if (r <= kMaxR) {
        is += sm.cnt[r];
        if (r >= s.r_min) ib += (long long)r * pad8(sm.cnt[r]);
      }
    }
  }
  __syncthreads();
  const bool fits = sm.base[kMaxR + 1] <= s.cap;
  if (rank == 0) {
    if (tid <= kMaxR) bucket_count[bl * (kMaxR + 1) + tid] = sm.cnt[tid];
    if (tid <= kMaxR + 1) bucket_base[bl * (kMaxR + 2) + tid] = sm.base[tid];
    if (tid == 0 && !fits) raise_status(dev_status, VARRATE_ERR_CORRUPT);
  }
  if (!fits) return;
  if (tid <= kMaxR)
#pragma unroll
    for (int w = 0; w < kTabWarps; ++w) sm.wcnt[w][tid] += before;
  __syncthreads();

  const unsigned lt_mask = (1u << lane) - 1u;
  int* run = sm.wcnt[warp];
  for (int64_t tb = w0; tb < w1; tb += 32 * kTabUnroll) {
    int r[kTabUnroll];
#pragma unroll
    for (int u = 0; u < kTabUnroll; ++u) {
      const int64_t t = tb + 32 * u + lane;
      r[u] = t < w1 ? (int)rk[t] : -1;
    }
#pragma unroll
    for (int u = 0; u < kTabUnroll; ++u) {
      if (tb + 32 * u >= w1) break;   // warp-uniform
      const int64_t t = tb + 32 * u + lane;
      const unsigned peers = __match_any_sync(0xffffffffu, r[u]);
      const int within = __popc(peers & lt_mask);
      const int p = r[u] >= 0 ? run[r[u]] + within : 0;
      __syncwarp();
      if (r[u] >= 0) {
        if (within == 0) run[r[u]] = p + __popc(peers);
        pos[bl * s.N + t] = p;
        perm[bl * s.N + sm.slot_start[r[u]] + p] = (int32_t)t;
      }
      __syncwarp();
    }
  }
}

int launch_tables(const Shape& s, const varrate_packed& out, int32_t* dev_status, int num_sms, cudaStream_t st) {
  // A CTA for every 2048 tokens, at most 8 to a pair and two CTAs an SM over all pairs.
  const int64_t pairs = (int64_t)s.B * s.L;
  int C = 1;
  while (C < kTabCluster && (int64_t)C * 2048 < s.N && C * pairs <= num_sms) C *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(pairs * C));
  cfg.blockDim = dim3(kTabThreads);
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = C; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, pack_tables_kernel, (const uint8_t*)out.ranks, out.bucket_count, out.bucket_base,
                            out.perm, out.pos, dev_status, s, (s.N + C - 1) / C) == cudaSuccess ? 1 : -1;
}

constexpr int kTile = 64;
constexpr int kLd = kHeadDim + 4;

// grid (n_chunks, G * 2, B * L), 256 threads.
template <typename T>
__global__ void __launch_bounds__(256)
project_kernel(const T* __restrict__ k, const T* __restrict__ v, const T* __restrict__ basis_k,
               const T* __restrict__ basis_v, const uint8_t* __restrict__ ranks,
               const int32_t* __restrict__ bucket_count, const int64_t* __restrict__ bucket_base,
               const int32_t* __restrict__ perm, const int32_t* __restrict__ pos,
               T* __restrict__ coef, Shape s, int64_t chunk) {
  extern __shared__ float smem[];
  float* us = smem;                         // [128][kLd]  U rows
  float* xs = us + kHeadDim * kLd;          // [64][kLd]   gathered tokens, then coefficients
  __shared__ int stok[kTile], srk[kTile], spos[kTile];
  __shared__ int s_ranks;                   // largest rank of the tile (its last valid slot's)
  __shared__ int n8s[kMaxR + 1];
  __shared__ long long bases[kMaxR + 2];
  const int64_t bl = blockIdx.z;
  const int g = blockIdx.y >> 1, kv = blockIdx.y & 1;
  const int64_t l = bl % s.L;
  const int tid = threadIdx.x;

  for (int r = tid; r <= kMaxR + 1; r += blockDim.x) {
    if (r <= kMaxR) n8s[r] = (int)pad8(bucket_count[bl * (kMaxR + 1) + r]);
    bases[r] = bucket_base[bl * (kMaxR + 2) + r];
  }
  const T* U = (kv ? basis_v : basis_k) + (l * s.G + g) * (int64_t)kHeadDim * kHeadDim;
#pragma unroll 4
  for (int i = tid; i < kHeadDim * (kHeadDim / 4); i += 256) {
    const int row = i / (kHeadDim / 4), c = i % (kHeadDim / 4) * 4;
    *reinterpret_cast<float4*>(&us[row * kLd + c]) = load4(U + 4 * i);
  }
  __syncthreads();
  if (bases[kMaxR + 1] > s.cap) return;   // corrupt tables were reported by pack_tables

  // zero the padding of each bucket of this stream: in row j they are the end of the last 8-slot group
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + tid; i < (kMaxR + 1) * kHeadDim; i += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)i / kHeadDim, j = (int)i % kHeadDim;
    if (r < s.r_min || j >= r) continue;
    const int n = bucket_count[bl * (kMaxR + 1) + r];
    for (int p = n; p < n8s[r]; ++p)
      coef[((bl * s.G + g) * 2 + kv) * s.cap + bases[r] + coef_offset(r, n8s[r], p, j)] = from_f<T>(0.f);
  }

  const T* x = (kv ? v : k) + (bl * s.G + g) * s.N * kHeadDim;
  T* out = coef + ((bl * s.G + g) * 2 + kv) * s.cap;
  const int ts = tid / 16, tj = tid % 16;
  const int64_t s_begin = blockIdx.x * chunk;
  const int64_t s_end = min(s.N, s_begin + chunk);
  for (int64_t s0 = s_begin; s0 < s_end; s0 += kTile) {
    __syncthreads();
    if (tid < kTile) {
      const int64_t sl = s0 + tid;
      int t = -1, r = 0, p = 0;
      if (sl < s_end) {
        t = perm[bl * s.N + sl];
        r = ranks[bl * s.N + t];
        p = pos[bl * s.N + t];
      }
      stok[tid] = t; srk[tid] = r; spos[tid] = p;
      if (sl < s_end && (sl + 1 == s_end || tid == kTile - 1)) s_ranks = r;
    }
    __syncthreads();
#pragma unroll
    for (int i = tid; i < kTile * (kHeadDim / 4); i += 256) {
      const int row = i / (kHeadDim / 4), c = i % (kHeadDim / 4) * 4;
      const int t = stok[row];
      *reinterpret_cast<float4*>(&xs[row * kLd + c]) =
          t >= 0 ? load4(x + (int64_t)t * kHeadDim + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    const int nj = s_ranks;   // slots come in increasing rank: rows of U from nj on are not needed
    float acc[4][8];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[a][i] = 0.f;
    if (nj <= 32) {
#pragma unroll 4
      for (int c = 0; c < kHeadDim; c += 4) {
        float4 xv[4], uv[2];
#pragma unroll
        for (int a = 0; a < 4; ++a) xv[a] = *reinterpret_cast<const float4*>(&xs[(4 * ts + a) * kLd + c]);
#pragma unroll
        for (int i = 0; i < 2; ++i) uv[i] = *reinterpret_cast<const float4*>(&us[(tj + 16 * i) * kLd + c]);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            acc[a][i] = fmaf(xv[a].x, uv[i].x, acc[a][i]);
            acc[a][i] = fmaf(xv[a].y, uv[i].y, acc[a][i]);
            acc[a][i] = fmaf(xv[a].z, uv[i].z, acc[a][i]);
            acc[a][i] = fmaf(xv[a].w, uv[i].w, acc[a][i]);
          }
      }
    } else
#pragma unroll 4
    for (int c = 0; c < kHeadDim; c += 4) {
      float4 xv[4], uv[8];
#pragma unroll
      for (int a = 0; a < 4; ++a) xv[a] = *reinterpret_cast<const float4*>(&xs[(4 * ts + a) * kLd + c]);
#pragma unroll
      for (int i = 0; i < 8; ++i) uv[i] = *reinterpret_cast<const float4*>(&us[(tj + 16 * i) * kLd + c]);
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          acc[a][i] = fmaf(xv[a].x, uv[i].x, acc[a][i]);
          acc[a][i] = fmaf(xv[a].y, uv[i].y, acc[a][i]);
          acc[a][i] = fmaf(xv[a].z, uv[i].z, acc[a][i]);
          acc[a][i] = fmaf(xv[a].w, uv[i].w, acc[a][i]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int i = 0; i < 8; ++i) xs[(4 * ts + a) * kLd + tj + 16 * i] = acc[a][i];
    __syncthreads();
    for (int i = tid; i < kTile * nj; i += blockDim.x) {
      const int slot = i % kTile, j = i / kTile;
      const int r = srk[slot];
      if (stok[slot] >= 0 && j < r)
        out[bases[r] + coef_offset(r, n8s[r], spos[slot], j)] = from_f<T>(xs[slot * kLd + j]);
    }
  }
}

}  // namespace

int launch_pack(const Shape& s, const void* k, const void* v, const void* basis_k,
                const void* basis_v, const varrate_packed& out, int32_t* dev_status, int num_sms,
                cudaStream_t st) {
  const int64_t units = (int64_t)s.B * s.L * s.G * 2;
  const int64_t want = 4LL * num_sms;
  int64_t n = (want + units - 1) / units;
  int64_t chunk = (s.N + n - 1) / n;
  chunk = ((chunk + kTile - 1) / kTile) * kTile;
  if (chunk < kTile) chunk = kTile;
  const int n_chunks = (int)((s.N + chunk - 1) / chunk);
  const size_t smem = (size_t)(kHeadDim + kTile) * kLd * sizeof(float);
  dim3 grid(n_chunks, s.G * 2, s.B * s.L);
  if (launch_tables(s, out, dev_status, num_sms, st) < 0) return -1;
  if (s.dtype == VARRATE_BF16) {
    const int np = launch_project_tc(s, k, v, basis_k, basis_v, out, dev_status, num_sms, st);
    return np < 0 ? -1 : 1 + np;
  } else {
    using T = float;
    cudaFuncSetAttribute(project_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    project_kernel<T><<<grid, 256, smem, st>>>((const T*)k, (const T*)v, (const T*)basis_k,
                                               (const T*)basis_v, out.ranks, out.bucket_count,
                                               out.bucket_base, out.perm, out.pos, (T*)out.coef, s, chunk);
  }
  return 2;
}

}  // namespace vr
