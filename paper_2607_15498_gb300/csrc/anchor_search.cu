// Joint codec, nearest-anchor search (Sec. 3.1, Eq. 2), bf16, on the 5th-generation tensor cores.
//
// Every token's joint vector z_t = [k_t of heads 0..G-1 ; v_t of heads 0..G-1] (Eq. 1, D = 2 G d)
// is compared with the anchors z_{a * stride} by squared Euclidean distance,
//   dist(t, a) = |z_t|^2 + |z_a|^2 - 2 z_t . z_a,
// with the bf16 products exact and every sum in fp32 (the paper keeps this search in fp32: its
// bf16 form cancels). Two kernels:
//   anchor_prep_kernel    one pass over K and V: |z_t|^2 of every token (a warp per token, a fixed
//                         shuffle tree, so the value is reproducible), and the anchors copied into a
//                         dense [B L][2][G][n_ap][d] block (n_ap = anchor count rounded up to 256,
//                         padding rows zero with norm +inf, so they are never chosen);
//   anchor_search_tc_kernel  a CTA pair (cta_group::2) per 256 tokens of one (sequence, layer): S = Z_tile A^T
//                         by tcgen05.mma (M = 256 tokens x N = 256 anchors per accumulator, K = D in
//                         steps of 64 columns, each step one head half of K or V fed by TMA with a
//                         128-byte swizzle: each CTA stages its own 128 tokens and half of the anchors),
//                         both TMEM accumulators in use (512 columns) so that the
//                         epilogue of one anchor tile overlaps the products of the next. Epilogue
//                         thread = token row: it turns its 256 scores into distances and keeps the
//                         8 smallest (distance, anchor) pairs in registers, in lexicographic order;
//                         the two epilogue groups (alternate anchor tiles) merge their lists at the
//                         end and the first c pairs are stored.
// What bounds the search is what each SM takes in from L2: at 64 bytes a clock, 128 tokens x 256 anchors x 64
// columns on one CTA need 48 KB, 768 clocks, for 512 clocks of products; half the anchors per CTA make it
// 32 KB. Before that the epilogue did: an insertion walked the list in a chain of compares, each warp for
// each lane that inserted. 32768 tokens, 2048 anchors, D = 2048: 387 us on single CTAs and on pairs, 206 us on
// pairs with the insertion of independent compares (61 % of the tensor pipe's time, 1.7 waves of pairs).
// A third kernel, anchor_residual_kernel, forms the residuals e_t = z_t - z_bar_t of Eq. 2 from the
// lists (Algorithm 1, third step).
// Warp roles of the search kernel: one TMA producer warp, one MMA-issuing warp, eight epilogue
// warps (lane quarter = warp % 4). Every mbarrier wait is bounded; a timeout raises
// VARRATE_ERR_TIMEOUT.
#include <cudaTypedefs.h>
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace vr {

namespace {

constexpr uint32_t kTries = 1u << 22;
constexpr int AS_TM = 128;                  // tokens per CTA (half of the pair's MMA M)
constexpr int AS_TN = 256;                  // anchors per accumulator (MMA N)
constexpr int AS_ST = 6;                    // operand stages
constexpr int AS_ABYTES = AS_TM * 128;      // 128 token rows x 64 bf16
constexpr int AS_BBYTES = AS_TN / 2 * 128;  // this CTA's 128 anchor rows x 64 bf16
constexpr int AS_SBYTES = AS_ABYTES + AS_BBYTES;
constexpr int AS_NGRP = 2;                  // epilogue groups of four warps (alternate anchor tiles)
constexpr int AS_EPI = 4 * AS_NGRP;
constexpr int AS_THREADS = (AS_EPI + 2) * 32;
constexpr int AS_LIST = 8;                  // (distance, anchor) pairs kept per token

struct AsSmem {
  uint64_t full[AS_ST], empty[AS_ST], tfull[AS_NGRP], tempty[AS_NGRP], drain;
  uint32_t tmem;
  int err;
  float md[AS_TM][AS_LIST];                 // group 1's lists, merged by group 0
  int mi[AS_TM][AS_LIST];
};

// ------------------------------------------------------------------------------ prep
// grid (ceil(N / 8), B * L), 256 threads: warp w takes token blockIdx.x * 8 + w.
__global__ void __launch_bounds__(256)
anchor_prep_kernel(const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                   __nv_bfloat16* __restrict__ anchors, float* __restrict__ anorm,
                   float* __restrict__ tnorm, int G, int64_t N, int stride, int n_a, int n_ap) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t bl = blockIdx.y;
  const int64_t t = (int64_t)blockIdx.x * 8 + warp;
  if (t < N) {
    const bool is_anchor = (t % stride) == 0;
    const int64_t a = t / stride;
    float acc = 0.f;
    for (int kvg = 0; kvg < 2 * G; ++kvg) {
      const int kv = kvg >= G, g = kvg - kv * G;
      const __nv_bfloat16* row = (kv ? v : k) + ((bl * G + g) * N + t) * kHeadDim;
      const uint2 u = __ldg(reinterpret_cast<const uint2*>(row) + lane);   // 4 bf16 per lane
      const float x0 = __uint_as_float(u.x << 16), x1 = __uint_as_float(u.x & 0xffff0000u);
      const float x2 = __uint_as_float(u.y << 16), x3 = __uint_as_float(u.y & 0xffff0000u);
      acc = fmaf(x0, x0, acc);
      acc = fmaf(x1, x1, acc);
      acc = fmaf(x2, x2, acc);
      acc = fmaf(x3, x3, acc);
      if (is_anchor)
        reinterpret_cast<uint2*>(anchors + (((bl * 2 + kv) * G + g) * n_ap + a) * kHeadDim)[lane] = u;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
      tnorm[bl * N + t] = acc;
      if (is_anchor) anorm[bl * n_ap + a] = acc;
    }
  }
  // padding anchors [n_a, n_ap): zero rows, infinite norm (never among the nearest)
  if (blockIdx.x == 0) {
    const int pad = n_ap - n_a;
    for (int idx = threadIdx.x; idx < pad * 2 * G * 32; idx += blockDim.x) {
      const int ln = idx & 31, rest = idx >> 5;
      const int a = n_a + rest % pad, kvg = rest / pad;
      reinterpret_cast<uint2*>(anchors + ((bl * 2 * G + kvg) * n_ap + a) * kHeadDim)[ln] = make_uint2(0, 0);
    }
    for (int a = n_a + threadIdx.x; a < n_ap; a += blockDim.x) anorm[bl * n_ap + a] = INFINITY;
  }
}

// Insert (d, j) where d < bd[s] into a list sorted by distance, j larger than every anchor in it: behind equal
// distances, so the order stays lexicographic on (distance, anchor). A lane whose d is not below its last
// entry keeps its list. The eight comparisons are independent: no chain through the list.
__device__ __forceinline__ void list_insert_next(float (&bd)[AS_LIST], int (&bi)[AS_LIST], float d, int j) {
  bool lt[AS_LIST];
#pragma unroll
  for (int s = 0; s < AS_LIST; ++s) lt[s] = d < bd[s];
#pragma unroll
  for (int s = AS_LIST - 1; s > 0; --s) {
    bd[s] = lt[s - 1] ? bd[s - 1] : lt[s] ? d : bd[s];
    bi[s] = lt[s - 1] ? bi[s - 1] : lt[s] ? j : bi[s];
  }
  bd[0] = lt[0] ? d : bd[0];
  bi[0] = lt[0] ? j : bi[0];
}

// Insert (d, j) into the sorted list (bd, bi): lexicographic order on (distance, anchor), so equal
// distances keep the lower anchor first whatever order the pairs arrive in.
__device__ __forceinline__ void list_insert(float (&bd)[AS_LIST], int (&bi)[AS_LIST], float d, int j) {
  float cd = d;
  int ci = j;
#pragma unroll
  for (int s = 0; s < AS_LIST; ++s) {
    const bool lt = cd < bd[s] || (cd == bd[s] && ci < bi[s]);
    const float td = bd[s];
    const int ti = bi[s];
    bd[s] = lt ? cd : td;
    bi[s] = lt ? ci : ti;
    cd = lt ? td : cd;
    ci = lt ? ti : ci;
  }
}

// ------------------------------------------------------------------------------ search
// grid (2 ceil(N / 256), B * L) in clusters of two along x. The even CTA's full and tempty barriers serve the
// pair; each CTA has its own empty and tfull barriers, which the pair's commits arrive on.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(AS_THREADS, 1)
anchor_search_tc_kernel(const __grid_constant__ CUtensorMap tk, const __grid_constant__ CUtensorMap tv,
                        const __grid_constant__ CUtensorMap ta, const float* __restrict__ tnorm,
                        const float* __restrict__ anorm, int32_t* __restrict__ idx_out,
                        float* __restrict__ dist_out, int32_t* __restrict__ dev_status, int G, int64_t N,
                        int n_ap, int c) {
  extern __shared__ __align__(1024) unsigned char raw_smem[];
  unsigned char* smem = raw_smem + ((1024 - (smem_addr(raw_smem) & 1023)) & 1023);
  AsSmem& sm = *reinterpret_cast<AsSmem*>(smem + AS_ST * AS_SBYTES);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = blockIdx.x & 1;
  const int64_t bl = blockIdx.y;
  const int64_t t0 = (int64_t)blockIdx.x * AS_TM;
  // the odd CTA of the last pair may have no tokens: it loads its partner's and stores nothing
  const int64_t t_load = t0 < N ? t0 : t0 - AS_TM;
  const int n_kb = 4 * G;                    // 64-column steps over D = 2 G d
  const int n_at = n_ap / AS_TN;
  const int total = n_at * n_kb;

  if (warp == AS_EPI + 1 && lane == 0) {
    for (int i = 0; i < AS_ST; ++i) { mbar_init(&sm.full[i], 1); mbar_init(&sm.empty[i], 1); }
    for (int i = 0; i < AS_NGRP; ++i) { mbar_init(&sm.tfull[i], 1); mbar_init(&sm.tempty[i], 8); }
    mbar_init(&sm.drain, 1);
    sm.err = 0;
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc2(&sm.tmem, AS_NGRP * AS_TN);
  tc_fence_before();
  __syncthreads();
  cluster_barrier();   // both CTAs' barriers are initialised
  tc_fence_after();
  const uint32_t tmem = sm.tmem;
  const uint32_t stage0 = smem_addr(smem);
  float bd[AS_LIST];
  int bi[AS_LIST];
#pragma unroll
  for (int s = 0; s < AS_LIST; ++s) { bd[s] = INFINITY; bi[s] = -1; }

  if (warp == AS_EPI) {
    if (lane == 0) {                                    // TMA producer: this CTA's operand halves
      int i = 0;
      for (; i < total; ++i) {
        const int at = i / n_kb, kb = i - at * n_kb, st = i % AS_ST;
        if (!mbar_wait_cluster(&sm.empty[st], ((i / AS_ST) & 1) ^ 1, kTries)) { sm.err = 1; break; }
        const int kv = kb >= 2 * G;
        const int g = (kb >> 1) - kv * G, half = kb & 1;
        const uint32_t dst = stage0 + st * AS_SBYTES, bar = cluster_addr(&sm.full[st], 0);
        if (rank == 0) mbar_arrive_expect_tx(&sm.full[st], 2 * AS_SBYTES);
        // token rows past N read the next stream's rows (or zeros past the tensor): never stored
        tma_load_2d_pair(dst, kv ? &tv : &tk, 64 * half, (int)((bl * G + g) * N + t_load), bar);
        tma_load_2d_pair(dst + AS_ABYTES, &ta, 64 * half,
                         (int)(((bl * 2 + kv) * G + g) * n_ap + at * AS_TN + (int)rank * (AS_TN / 2)), bar);
      }
      // every copy of the pair has landed before either CTA can end, also after a wait that gave up
      if (rank == 0)
        for (int j = max(0, i - AS_ST); j < i; ++j) mbar_wait_cluster(&sm.full[j % AS_ST], (j / AS_ST) & 1, kTries);
    }
  } else if (warp == AS_EPI + 1) {
    if (lane == 0 && rank == 0) {                       // MMA issuer of the pair
      constexpr uint32_t idesc = idesc_bf16_f32(2 * AS_TM, AS_TN);
      bool ok = true;
      for (int at = 0; at < n_at && ok; ++at) {
        const int b = at & 1;
        if (!mbar_wait_cluster(&sm.tempty[b], ((at >> 1) & 1) ^ 1, kTries)) { ok = false; break; }
        tc_fence_after();
        for (int kb = 0; kb < n_kb; ++kb) {
          const int i = at * n_kb + kb, st = i % AS_ST;
          if (!mbar_wait_cluster(&sm.full[st], (i / AS_ST) & 1, kTries)) { ok = false; break; }
          tc_fence_after();
          const uint32_t a0 = stage0 + st * AS_SBYTES, b0 = a0 + AS_ABYTES;
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)
            tc_mma2_bf16(tmem + b * AS_TN, sdesc_sw128(a0 + ks * 32), sdesc_sw128(b0 + ks * 32), idesc,
                         (kb | ks) != 0);
          tc_commit2(&sm.empty[st]);
        }
        if (ok) tc_commit2(&sm.tfull[b]);
      }
      if (!ok) {   // the products in flight end before TMEM is freed
        sm.err = 1;
        tc_commit2(&sm.drain);
        mbar_wait_cluster(&sm.drain, 0, kTries);
      }
    }
  } else {                                              // epilogue: one token row, alternate tiles
    const int quarter = warp & 3, eg = warp >> 2;
    const int row = quarter * 32 + lane;
    const int64_t t = t0 + row;
    const float nz = t < N ? tnorm[bl * N + t] : 0.f;
    const float* an = anorm + bl * n_ap;
    bool bad = false;
    for (int at = eg; at < n_at; at += AS_NGRP) {
      const int b = at & 1;
      if (!bad && !mbar_wait_cluster(&sm.tfull[b], (at >> 1) & 1, kTries)) { sm.err = 1; bad = true; }
      tc_fence_after();
      const uint32_t taddr = tmem + b * AS_TN + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
      for (int cb = 0; cb < AS_TN / 32; ++cb) {
        float sv[32];
        tmem_ld32(taddr + cb * 32, sv);
        const int j0 = at * AS_TN + cb * 32;
        const float4* an4 = reinterpret_cast<const float4*>(an + j0);
#pragma unroll
        for (int q4 = 0; q4 < 8; ++q4) {
          const float4 na = __ldg(an4 + q4);
          const float nav[4] = {na.x, na.y, na.z, na.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int jj = q4 * 4 + e;
            const float dd = fmaxf(fmaf(-2.f, sv[jj], nz + nav[e]), 0.f);
            // some lane's list takes it (a vote, so that the warp stays together); no-op for the others
            if (__any_sync(0xffffffffu, dd < bd[AS_LIST - 1])) list_insert_next(bd, bi, dd, j0 + jj);
          }
        }
        __syncwarp();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(cluster_addr(&sm.tempty[b], 0));
    }
    if (eg == 1) {
#pragma unroll
      for (int s = 0; s < AS_LIST; ++s) { sm.md[row][s] = bd[s]; sm.mi[row][s] = bi[s]; }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp < 4) {                                       // group 0 merges and stores
    const int row = warp * 32 + lane;
    const int64_t t = t0 + row;
#pragma unroll
    for (int s = 0; s < AS_LIST; ++s)
      if (sm.mi[row][s] >= 0) list_insert(bd, bi, sm.md[row][s], sm.mi[row][s]);
    if (t < N && !sm.err) {
#pragma unroll
      for (int s = 0; s < AS_LIST; ++s) {
        if (s < c) {
          idx_out[(bl * N + t) * c + s] = bi[s];
          if (dist_out != nullptr) dist_out[(bl * N + t) * c + s] = bd[s];
        }
      }
    }
  }
  if (tid == 0 && sm.err) raise_status(dev_status, VARRATE_ERR_TIMEOUT);
  __syncwarp();
  cluster_barrier();   // no CTA leaves, or frees TMEM, while the other may still signal it or use the pair's TMEM
  if (warp == 0) tmem_dealloc2(tmem, AS_NGRP * AS_TN);
}

size_t search_smem_bytes() { return 1024 + (size_t)AS_ST * AS_SBYTES + sizeof(AsSmem); }

// ------------------------------------------------------------------------------ residual
// Eq. 2: e_t = z_t - mean of the anchors listed for t. The listed anchors are summed in list order in
// fp32 (bf16 values are exact in fp32), divided by their count (IEEE division; by a power of two the
// product with its exact reciprocal is the same number), subtracted from z_t and rounded to bf16.
// The list of a token: rows[s] = anchor, or n_a (a row of zeros) for a skipped entry; returns the number of valid
// entries, 0 when there is none or an entry is out of [-1, n_a). K entries are formed, of which c are in the list
// (K = c = 2 or 4: one load, aligned to the list).
template <int K>
__device__ __forceinline__ int load_list(const int32_t* __restrict__ p, int c, int n_a, uint32_t (&rows)[K]) {
  int x[K];
  if constexpr (K == 4) {
    const int4 q = __ldg(reinterpret_cast<const int4*>(p));
    x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
  } else if constexpr (K == 2) {
    const int2 q = __ldg(reinterpret_cast<const int2*>(p));
    x[0] = q.x; x[1] = q.y;
  } else {
#pragma unroll
    for (int s = 0; s < K; ++s) x[s] = s < c ? __ldg(p + s) : -1;
  }
  int m = K;
  uint32_t worst = 0;
#pragma unroll
  for (int s = 0; s < K; ++s) {
    worst = max(worst, (uint32_t)(x[s] + 1));   // -1 .. n_a - 1 -> 0 .. n_a; anything else is above
    m += x[s] >> 31;
    rows[s] = min((uint32_t)x[s], (uint32_t)n_a);
  }
  return worst > (uint32_t)n_a ? 0 : m;
}

// acc + x with x a bf16 (exact in fp32): one mixed-precision add per element, rounded to nearest.
__device__ __forceinline__ void add8(float (&acc)[8], uint4 u) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i)
    asm("{\n .reg .b16 l, h;\n mov.b32 {l, h}, %2;\n add.rn.f32.bf16 %0, l, %0;\n add.rn.f32.bf16 %1, h, %1;\n}\n"
        : "+f"(acc[2 * i]), "+f"(acc[2 * i + 1]) : "r"(w[i]));
}

__device__ __forceinline__ uint4 residual8(uint4 z, float (&acc)[8], int m) {
  if ((m & (m - 1)) == 0) {
    const float inv = m == 1 ? 1.f : m == 2 ? 0.5f : m == 4 ? 0.25f : 0.125f;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = __fmul_rn(acc[i], inv);
  } else {
    const float fm = (float)m;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = __fdiv_rn(acc[i], fm);
  }
  const uint32_t w[4] = {z.x, z.y, z.z, z.w};
  uint32_t o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    o[i] = pack_bf16(__fsub_rn(__uint_as_float(w[i] << 16), acc[2 * i]),
                     __fsub_rn(__uint_as_float(w[i] & 0xffff0000u), acc[2 * i + 1]));
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// Slab form: a CTA keeps CW columns of every anchor of one (sequence, layer, head, K-or-V) in shared memory
// (plus a zero row for skipped entries) and streams its share of the tokens past them, 16 bytes a thread.
// Read straight from L2 the c listed anchors of every token are c times the bytes of K and V themselves;
// from shared memory K and V are read once and the residuals written once. Bound by shared-memory reads (rows
// of 64 bytes: two of them share a wavefront when their parities differ) and instructions: the length of the lists
// C is a constant (any length in one form, eight entries tested each, took 72 to 102 us at lengths 1 to 8 where this
// takes 56 to 86). 2 layers x 8 heads x 32768 tokens, 4 of 2048 anchors each (538 MB): a warp per token
// reading L2 248 us, this 117 us.
// grid (column blocks x splits x 2 G, B L).
constexpr int RS_THREADS = 1024;
constexpr int RS_TOK = 2;                    // tokens per thread whose loads are in flight together
constexpr size_t RS_SMEM = 208 * 1024;       // most shared memory for a slab

template <int CW, int C>
__global__ void __launch_bounds__(RS_THREADS, 1)
anchor_residual_slab_kernel(const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                            const int32_t* __restrict__ idx, __nv_bfloat16* __restrict__ e,
                            int32_t* __restrict__ dev_status, int G, int64_t N, int stride, int n_a,
                            int splits, int64_t share) {
  constexpr int TPT = CW / 8, TOKS = RS_THREADS / TPT, NCB = kHeadDim / CW;   // threads a token, tokens a step
  extern __shared__ uint4 slab[];            // [n_a + 1][TPT]
  const int tid = threadIdx.x, part = tid % TPT;
  const int cb = blockIdx.x % NCB, rest = blockIdx.x / NCB, split = rest % splits, kvg = rest / splits;
  const int64_t bl = blockIdx.y;
  const int kv = kvg >= G, g = kvg - kv * G;
  const __nv_bfloat16* base = (kv ? v : k) + (bl * G + g) * N * kHeadDim + cb * CW;
#pragma unroll 4
  for (int i = tid; i < n_a * TPT; i += RS_THREADS)
    slab[i] = __ldg(reinterpret_cast<const uint4*>(base + (int64_t)(i / TPT) * stride * kHeadDim) + part);
  if (tid < TPT) slab[n_a * TPT + tid] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  const int64_t t_end = min(N, (split + 1) * share);
  for (int64_t t0 = split * share + tid / TPT; t0 < t_end; t0 += TOKS * RS_TOK) {
    uint4 z[RS_TOK];
    uint32_t rows[RS_TOK][C];
    int m[RS_TOK];
#pragma unroll
    for (int u = 0; u < RS_TOK; ++u) {
      const int64_t t = t0 + u * TOKS;
      if (t < t_end) {
        z[u] = __ldcs(reinterpret_cast<const uint4*>(base + t * kHeadDim) + part);
        m[u] = load_list<C>(idx + (bl * N + t) * C, C, n_a, rows[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < RS_TOK; ++u) {
      const int64_t t = t0 + u * TOKS;
      if (t >= t_end) break;
      if (m[u] == 0) {
        raise_status(dev_status, VARRATE_ERR_CORRUPT);
        continue;
      }
      float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int s = 0; s < C; ++s) add8(acc, slab[rows[u][s] * TPT + part]);
      __stcs(reinterpret_cast<uint4*>(e + ((bl * N + t) * 2 * G + kvg) * kHeadDim + cb * CW) + part,
             residual8(z[u], acc, m[u]));
    }
  }
}

// Direct form, for more anchors or fewer tokens than the slab form is for: a warp per token, half a warp per head row
// (16 bytes a lane), the listed anchors read from L2, all of a row's in flight together. Bound by that latency: at 64
// registers four CTAs share an SM; at 78 (three) 8 heads x 32768 tokens, lists of 7 at stride 5, took 127 us, now 93 (134
// with a whole warp per head row, 8 bytes a lane). grid (ceil(N / 8), B L), 256 threads.
__global__ void __launch_bounds__(256, 4)
anchor_residual_kernel(const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                       const int32_t* __restrict__ idx, __nv_bfloat16* __restrict__ e,
                       int32_t* __restrict__ dev_status, int G, int64_t N, int stride, int c, int n_a) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l16 = lane & 15;
  const int64_t bl = blockIdx.y;
  const int64_t t = (int64_t)blockIdx.x * 8 + warp;
  if (t >= N) return;
  uint32_t rows[AS_LIST];
  const int m = load_list<AS_LIST>(idx + (bl * N + t) * c, c, n_a, rows);
  if (m == 0) {                                      // warp-uniform: every lane read the same list
    if (lane == 0) raise_status(dev_status, VARRATE_ERR_CORRUPT);
    return;
  }
#pragma unroll 2
  for (int kvg = lane >> 4; kvg < 2 * G; kvg += 2) {
    const int kv = kvg >= G, g = kvg - kv * G;
    const __nv_bfloat16* base = (kv ? v : k) + (bl * G + g) * N * kHeadDim;
    const uint4 z = __ldg(reinterpret_cast<const uint4*>(base + t * kHeadDim) + l16);
    uint4 u[AS_LIST];
#pragma unroll
    for (int s = 0; s < AS_LIST; ++s) {
      u[s] = make_uint4(0, 0, 0, 0);
      if (rows[s] < (uint32_t)n_a) u[s] = __ldg(reinterpret_cast<const uint4*>(base + (int64_t)rows[s] * stride * kHeadDim) + l16);
    }
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int s = 0; s < AS_LIST; ++s)
      if (rows[s] < (uint32_t)n_a) add8(acc, u[s]);
    reinterpret_cast<uint4*>(e + ((bl * N + t) * 2 * G + kvg) * kHeadDim)[l16] = residual8(z, acc, m);
  }
}

}  // namespace

bool make_tmap_rows_bf16(CUtensorMap* map, const void* base, uint64_t rows, uint32_t box_rows);

int anchor_count(int64_t N, int stride) { return (int)((N + stride - 1) / stride); }
int anchor_count_padded(int64_t N, int stride) {
  return (anchor_count(N, stride) + AS_TN - 1) / AS_TN * AS_TN;
}

size_t anchor_search_ws_bytes(const Shape& s, int stride) {
  const size_t n_ap = (size_t)anchor_count_padded(s.N, stride);
  const size_t bl = (size_t)s.B * s.L;
  auto a256 = [](size_t x) { return (x + 255) & ~size_t(255); };
  return a256(bl * 2 * s.G * n_ap * kHeadDim * 2) + a256(bl * n_ap * 4) + a256(bl * (size_t)s.N * 4);
}

bool anchor_residual_supported(const Shape& s, int stride, int c) {
  return s.dtype == VARRATE_BF16 && stride >= 1 && stride <= s.N && c >= 1 && c <= AS_LIST &&
         (int64_t)s.B * s.L <= 65535;
}

namespace {

template <int CW, int C>
int launch_residual_slab(const Shape& s, const void* k, const void* v, int stride, const int32_t* idx,
                         void* e_out, int32_t* dev_status, int num_sms, cudaStream_t st) {
  const int n_a = anchor_count(s.N, stride);
  const size_t smem = (size_t)(n_a + 1) * CW * 2;
  auto kernel = anchor_residual_slab_kernel<CW, C>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RS_SMEM) != cudaSuccess) return -1;
  // splits of the tokens that make waves x (steps of a CTA + its slab, read at about twice a step's rate) least
  constexpr int64_t kStep = RS_THREADS / (CW / 8) * RS_TOK;
  const int64_t units = (int64_t)s.B * s.L * 2 * s.G * (kHeadDim / CW), steps = (s.N + kStep - 1) / kStep;
  const double setup = 1.0 + (double)n_a / (2.0 * kStep);
  int64_t n = 1;
  double best = 1e300;
  for (int64_t i = 1; i <= steps && i <= 2 * num_sms; ++i) {
    const double cost = (double)((units * i + num_sms - 1) / num_sms) * ((double)((steps + i - 1) / i) + setup);
    if (cost < best * 0.999) { best = cost; n = i; }
  }
  const int64_t share = (steps + n - 1) / n * kStep;
  n = (s.N + share - 1) / share;
  const dim3 grid((unsigned)(kHeadDim / CW * n * 2 * s.G), (unsigned)((size_t)s.B * s.L));
  kernel<<<grid, RS_THREADS, smem, st>>>(
      (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, idx, (__nv_bfloat16*)e_out, dev_status, s.G, s.N, stride, n_a,
      (int)n, share);
  return 1;
}

}  // namespace

int launch_anchor_residual(const Shape& s, const void* k, const void* v, int stride, int c,
                           const int32_t* idx, void* e_out, int32_t* dev_status, int num_sms, cudaStream_t st) {
  // Slabs where 32 columns of all anchors (and the zero row) fit and there are some 24 thousand rows of K to stream
  // past them; at 32 columns, lists of 8 read too many rows of shared memory. Slab / direct in us, 8 heads: 32768
  // tokens, stride 64 (128 columns) lists of 1 52 / 75, 4 55 / 79, 8 64 / 83; stride 16 (32 columns) 1 56 / 76, 3 64 / 89,
  // 4 62 / 81, 7 86 / 89, 8 95 / 83; 2000 tokens 4 12.7 / 10.0, 4000 tokens 12.4 / 14.7. With 16 columns (stride 5 to 8)
  // slabs took 79 to 170 us where direct takes 76 to 94.
  const size_t rows = (size_t)anchor_count(s.N, stride) + 1;
  const int cw = rows * 256 <= RS_SMEM ? 128 : rows * 128 <= RS_SMEM ? 64 : rows * 64 <= RS_SMEM ? 32 : 0;
  if (cw && !(cw == 32 && c == AS_LIST) && (int64_t)s.B * s.L * s.G * s.N >= 24576) {
    auto launch = [&](auto C) {
      return cw == 128 ? launch_residual_slab<128, C()>(s, k, v, stride, idx, e_out, dev_status, num_sms, st)
             : cw == 64 ? launch_residual_slab<64, C()>(s, k, v, stride, idx, e_out, dev_status, num_sms, st)
                        : launch_residual_slab<32, C()>(s, k, v, stride, idx, e_out, dev_status, num_sms, st);
    };
    switch (c) {
      case 1: return launch(std::integral_constant<int, 1>());
      case 2: return launch(std::integral_constant<int, 2>());
      case 3: return launch(std::integral_constant<int, 3>());
      case 4: return launch(std::integral_constant<int, 4>());
      case 5: return launch(std::integral_constant<int, 5>());
      case 6: return launch(std::integral_constant<int, 6>());
      case 7: return launch(std::integral_constant<int, 7>());
      default: return launch(std::integral_constant<int, 8>());
    }
  }
  anchor_residual_kernel<<<dim3((unsigned)((s.N + 7) / 8), (unsigned)((size_t)s.B * s.L)), 256, 0, st>>>(
      (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, idx, (__nv_bfloat16*)e_out, dev_status, s.G, s.N,
      stride, c, anchor_count(s.N, stride));
  return 1;
}

bool anchor_search_supported(const Shape& s, int stride, int c) {
  if (s.dtype != VARRATE_BF16 || stride < 1 || stride > s.N || c < 1 || c > AS_LIST) return false;
  if ((int64_t)s.B * s.L > 65535 || s.G > 64) return false;
  const uint64_t rows_kv = (uint64_t)s.B * s.L * s.G * s.N;
  const uint64_t rows_a = (uint64_t)s.B * s.L * 2 * s.G * anchor_count_padded(s.N, stride);
  return rows_kv + AS_TM <= (uint64_t)INT32_MAX && rows_a <= (uint64_t)INT32_MAX;
}

int launch_anchor_search(const Shape& s, const void* k, const void* v, int stride, int c, int32_t* idx_out,
                         float* dist_out, int32_t* dev_status, void* ws, cudaStream_t st) {
  const int n_a = anchor_count(s.N, stride), n_ap = anchor_count_padded(s.N, stride);
  const size_t bl = (size_t)s.B * s.L;
  auto a256 = [](size_t x) { return (x + 255) & ~size_t(255); };
  char* w = static_cast<char*>(ws);
  __nv_bfloat16* anchors = reinterpret_cast<__nv_bfloat16*>(w);
  float* anorm = reinterpret_cast<float*>(w + a256(bl * 2 * s.G * n_ap * kHeadDim * 2));
  float* tnorm = reinterpret_cast<float*>(reinterpret_cast<char*>(anorm) + a256(bl * n_ap * 4));
  const uint64_t rows_kv = (uint64_t)s.B * s.L * s.G * s.N;
  const uint64_t rows_a = (uint64_t)bl * 2 * s.G * n_ap;
  CUtensorMap tk, tv, ta;
  if (!make_tmap_rows_bf16(&tk, k, rows_kv, AS_TM) || !make_tmap_rows_bf16(&tv, v, rows_kv, AS_TM) ||
      !make_tmap_rows_bf16(&ta, anchors, rows_a, AS_TN / 2))
    return -1;
  anchor_prep_kernel<<<dim3((unsigned)((s.N + 7) / 8), (unsigned)bl), 256, 0, st>>>(
      (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, anchors, anorm, tnorm, s.G, s.N, stride, n_a, n_ap);
  const size_t smem = search_smem_bytes();
  cudaFuncSetAttribute(anchor_search_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  anchor_search_tc_kernel<<<dim3(2 * (unsigned)((s.N + 2 * AS_TM - 1) / (2 * AS_TM)), (unsigned)bl), AS_THREADS, smem, st>>>(
      tk, tv, ta, tnorm, anorm, idx_out, dist_out, dev_status, s.G, s.N, n_ap, c);
  return 2;
}

}  // namespace vr
