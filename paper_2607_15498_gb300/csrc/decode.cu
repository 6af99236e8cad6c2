// Step 4 — decode attention on the packed coefficients of one layer (attention of Sec. 3.1 on the
// cache of Eq. 5, never rebuilding K or V).
//
// For query head h of KV head g:  q~ = U_K q * log2(e)/sqrt(d);  score_t = q~[:r_t] . c^K_t[:r_t];
// o = U_V^T (sum_t 2^(score_t - m) c^V_t[:r_t]) / sum_t 2^(score_t - m)   (+ exact tail tokens).
//
// decode_rotate  q~ for every head (fp32 workspace).
// decode_split   grid (S x head quads, G, B), 8 warps. The coded elements of the (b, l, g) stream are split
//                into S contiguous cost ranges; a warp item is 32 slots of a rank bucket. Lane (phase,
//                sg) holds 8 slots (16-byte loads, addressed through the packed layout) of the rows
//                j = phase, phase + 8, ...: scores are its partial sums added over the phases by
//                shuffles; on the value side each lane keeps the partial outputs of its rows over its
//                slots, added over the four slot groups once at the end, so no item needs more
//                cross-lane work than its scores. Online softmax per warp; warps then merge in shared
//                memory and write one (max, sum, o~[128]) partial per head.
// decode_combine merges the S partials (and the exact tail), rotates back with U_V^T, writes out.
#include "common.cuh"
#include "kernels.h"

namespace vr {

namespace {

constexpr int kMaxR = kHeadDim;
constexpr int kWarps = 8;
constexpr int kItem = 32;         // slots per warp item: a quarter of a tile of the packed layout
constexpr int kPhases = 8;        // lanes that share the rows of a slot group
constexpr int kMaxTail = 4096;
constexpr int kMaxSplits = 128;

// Raw 8-element row fragment: bf16 -> one uint4, fp32 -> two float4.
template <typename T> struct Frag;
template <> struct Frag<__nv_bfloat16> {
  uint4 u;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { u = __ldcs(reinterpret_cast<const uint4*>(p)); }
  __device__ __forceinline__ void zero() { u = make_uint4(0, 0, 0, 0); }
  __device__ __forceinline__ float get(int i) const {
    const uint32_t w = (i < 2) ? u.x : (i < 4) ? u.y : (i < 6) ? u.z : u.w;
    return (i & 1) ? __uint_as_float(w & 0xffff0000u) : __uint_as_float(w << 16);
  }
};
template <> struct Frag<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p) {
    a = __ldcs(reinterpret_cast<const float4*>(p));
    b = __ldcs(reinterpret_cast<const float4*>(p) + 1);
  }
  __device__ __forceinline__ void zero() { a = b = make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ __forceinline__ float get(int i) const {
    switch (i) { case 0: return a.x; case 1: return a.y; case 2: return a.z; case 3: return a.w;
                 case 4: return b.x; case 5: return b.y; case 6: return b.z; default: return b.w; }
  }
};

// Quantized 8-slot row fragment (group-wise b-bit codes, varrate_qpacked layout): the raw codes of
// slots p0 .. p0 + 7 of one coefficient row (one 32-slot group) and the group's (offset, step);
// get(i) dequantizes slot p0 + i as fl32(lo + fl32(code * step)).
template <int BITS> struct QFrag {
  uint32_t w0, w1;
  float lo, st;
  __device__ __forceinline__ void zero() { w0 = w1 = 0u; lo = 0.f; st = 0.f; }
  __device__ __forceinline__ void load(const uint8_t* row, int p0, int tl) {
    if (BITS == 4) {
      w0 = __ldcs(reinterpret_cast<const unsigned int*>(row + (p0 >> 1)));
      w1 = 0u;
    } else {
      const uint2 u = __ldcs(reinterpret_cast<const uint2*>(row + p0));
      w0 = u.x; w1 = u.y;
    }
    const __half2 par = *reinterpret_cast<const __half2*>(row + tl * BITS / 8 + 4 * (p0 >> 5));
    lo = __low2float(par);
    st = __high2float(par);
  }
  __device__ __forceinline__ float get(int i) const {
    const uint32_t c = BITS == 4 ? (w0 >> (4 * i)) & 15u : ((i < 4 ? w0 : w1) >> (8 * (i & 3))) & 255u;
    return __fadd_rn(lo, __fmul_rn((float)c, st));
  }
};

// Where the split kernel reads coefficient rows from. DenseSrc: the packed cache of `T` elements
// (bucket offsets from its table). QuantSrc: the quantized cache (bucket element offsets rebuilt
// from the counts, byte offsets from qbase). bind() selects a stream pair, tile() the tile that holds
// bucket slot s0 (8 slots from there on), row() loads coefficient row j of those slots: `rot` is the
// position of their group in that row, (group + j) mod (tl / 8).
template <typename T> struct DenseSrc {
  using F = Frag<T>;
  static constexpr bool kTableBase = true;
  const T* coef;
  const int64_t* bucket_base;
  int64_t stride;   // elements per stream
  const T* cK;
  const T* tK;
  int tl;
  __device__ __forceinline__ void bind(int64_t stream0) { cK = coef + stream0 * stride; }
  __device__ __forceinline__ void tile(int r, long long b0, long long, int tl_, long long s0) {
    tK = cK + b0 + (s0 >> 7) * 128 * r;
    tl = tl_;
  }
  __device__ __forceinline__ void row(F& f, int kv, int j, int rot) const {
    f.load(tK + (kv ? stride : 0) + j * tl + rot * 8);
  }
};
template <int BITS> struct QuantSrc {
  using F = QFrag<BITS>;
  static constexpr bool kTableBase = false;
  const uint8_t* data;
  const int64_t* qbase;
  int64_t stride;   // bytes per stream
  const uint8_t* qK;
  const uint8_t* tK;
  int tl, p0;
  __device__ __forceinline__ void bind(int64_t stream0) { qK = data + stream0 * stride; }
  __device__ __forceinline__ void tile(int r, long long, long long qb0, int tl_, long long s0) {
    tK = qK + qb0 + (s0 >> 7) * r * qrow_bytes(128, BITS);
    tl = tl_;
    p0 = (int)(s0 & 127);
  }
  __device__ __forceinline__ void row(F& f, int kv, int j, int) const {
    f.load(tK + (kv ? stride : 0) + j * qrow_bytes(tl, BITS), p0, tl);
  }
};

constexpr int kRotSplit = 8;   // CTAs that share the rows of U_K of one head

// grid (G, B, kRotSplit), 256 threads: qt[b][h][j] = scale * sum_i U_K[j][i] q[b][h][i].
template <typename T>
__global__ void __launch_bounds__(256)
decode_rotate_kernel(const T* __restrict__ q, const T* __restrict__ basis_k, float* __restrict__ qt,
                     Shape s, int layer) {
  __shared__ float qs[8][kHeadDim];
  const int g = blockIdx.x, b = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < s.grp * kHeadDim; i += blockDim.x)
    qs[i / kHeadDim][i % kHeadDim] = to_f(q[((int64_t)b * s.H + g * s.grp) * kHeadDim + i]);
  __syncthreads();
  const T* U = basis_k + ((int64_t)layer * s.G + g) * kHeadDim * kHeadDim;
  const float scale = kLog2e * rsqrtf((float)kHeadDim);
  constexpr int kRows = kHeadDim / kRotSplit;
#pragma unroll
  for (int jj = warp; jj < kRows; jj += kWarps) {
    const int j = blockIdx.z * kRows + jj;
    const float4 u4 = load4(U + j * kHeadDim + lane * 4);
    const float u[4] = {u4.x, u4.y, u4.z, u4.w};
    for (int hh = 0; hh < s.grp; ++hh) {
      float acc = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) acc = fmaf(u[i], qs[hh][lane * 4 + i], acc);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) qt[((int64_t)b * s.H + g * s.grp + hh) * kHeadDim + j] = acc * scale;
    }
  }
}

// GH heads of the group per CTA (4, or the whole group when it is smaller); blockIdx.x = split * quads + quad.
// Bound by instructions and load latency. Whole 128-slot tiles per warp (8 slots on each of 16 lanes, value rows
// reduced over the warp eight at a time) left a 128-row tile to one warp for 80 us and more. Per layer
// call with rotation and combine, before / now: fp32, 8 heads x 8000 tokens x 2 sequences 280 / 92 us;
// bf16, 8 heads x 32768 with 400 tail tokens 347 / 114 us, 4 heads of group 7 with wide ranks 662 / 143
// us; 4-bit, 300 tail tokens 318 / 124 us.
template <class Src, int GP, int GH>
__global__ void __launch_bounds__(256, 1)
decode_split_kernel(Src src, const int32_t* __restrict__ bucket_count, const float* __restrict__ qt,
                    float* __restrict__ part, Shape s, int layer, int S, long long table_cap) {
  constexpr int kRowsPer = kHeadDim / kPhases;   // rows a lane owns
  constexpr int kBatch = 4;                      // rows whose loads are in flight together
  __shared__ __align__(16) float q_s[kHeadDim][GH];
  __shared__ int cnt[kMaxR + 1];
  __shared__ long long base[kMaxR + 2];
  __shared__ long long qb[kMaxR + 2];   // quantized source: byte offset of each bucket
  __shared__ int i_first[kMaxR + 1], i_last[kMaxR + 1];   // this split's items of each bucket
  __shared__ float wM[kWarps][GH], wL[kWarps][GH];
  __shared__ float wacc[kWarps][GH][kHeadDim];

  constexpr int kQuads = GP / GH;
  const int split = blockIdx.x / kQuads, h0 = blockIdx.x % kQuads * GH, g = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t bl = (int64_t)b * s.L + layer;
  for (int r = tid; r <= kMaxR + 1; r += blockDim.x) {
    if (r <= kMaxR) cnt[r] = bucket_count[bl * (kMaxR + 1) + r];
    if constexpr (Src::kTableBase) base[r] = src.bucket_base[bl * (kMaxR + 2) + r];
    else qb[r] = src.qbase[bl * (kMaxR + 2) + r];
  }
  if constexpr (!Src::kTableBase) {   // element offsets of the buckets, as the packed table has them
    __syncthreads();
    if (tid == 0) {
      long long acc = 0;
      for (int r = 0; r <= kMaxR; ++r) {
        base[r] = acc;
        if (r >= s.r_min && r <= s.r_max) acc += (long long)r * pad8(cnt[r]);
      }
      base[kMaxR + 1] = acc;
    }
  }
  for (int i = tid; i < kHeadDim * GH; i += blockDim.x) {
    const int j = i / GH, hh = h0 + i % GH;
    q_s[j][i % GH] = hh < s.grp ? qt[((int64_t)b * s.H + g * s.grp + hh) * kHeadDim + j] : 0.f;
  }
  __syncthreads();

  const long long W = base[kMaxR + 1];
  const bool table_ok = W <= s.cap && (Src::kTableBase || qb[kMaxR + 1] <= table_cap);
  const long long lo = table_ok ? W * split / S : 0, hi = table_ok ? W * (split + 1) / S : 0;
  src.bind((bl * s.G + g) * 2);
  // one bucket a thread: the 64-bit divisions of all buckets at once
  for (int r = tid; r <= kMaxR; r += blockDim.x) {
    int first = 0, last = 0;
    if (table_ok && r >= s.r_min && r <= s.r_max && cnt[r] > 0) {
      const long long b0 = base[r], unit = (long long)kItem * r;
      const long long nit = (pad8(cnt[r]) + kItem - 1) / kItem;
      first = (int)min(nit, lo > b0 ? (lo - b0 + unit - 1) / unit : 0);
      last = (int)min(nit, hi > b0 ? (hi - b0 + unit - 1) / unit : 0);
    }
    i_first[r] = first;
    i_last[r] = last;
  }
  __syncthreads();

  const int sg = lane & 3, phase = lane >> 2;
  float M[GH], Ls[GH], acc[kRowsPer][GH];
#pragma unroll
  for (int h = 0; h < GH; ++h) { M[h] = -INFINITY; Ls[h] = 0.f; }
#pragma unroll
  for (int a = 0; a < kRowsPer; ++a)
#pragma unroll
    for (int h = 0; h < GH; ++h) acc[a][h] = 0.f;

  int counter = 0;   // items of the split before the bucket: the warps take them in turn
  for (int r = s.r_min; r <= s.r_max && table_ok; ++r) {
    const int i0 = i_first[r], i_hi = i_last[r];
    if (i0 >= i_hi) continue;
    const int turn = (warp - counter) & (kWarps - 1);
    counter += i_hi - i0;
    for (int it = i0 + turn; it < i_hi; it += kWarps) {
      const int n = cnt[r];
      const long long s0 = (long long)it * kItem + sg * 8, n8 = pad8(n);
      const bool on = s0 < n8;                          // the last item of a bucket may hold fewer groups
      const int tl = (int)min(128ll, n8 - ((long long)it * kItem & ~127ll)), ng = tl >> 3;
      src.tile(r, base[r], Src::kTableBase ? 0 : qb[r], tl, s0);
      const int rot0 = ((int)(s0 & 127) / 8 + phase) % ng, rstep = kPhases % ng;

      // scores of 8 slots x GH heads over this lane's rows, then over the phases
      float sc[GH][8];
#pragma unroll
      for (int h = 0; h < GH; ++h)
#pragma unroll
        for (int i = 0; i < 8; ++i) sc[h][i] = 0.f;
      int rot = rot0;
      for (int j0 = phase; j0 < r; j0 += kPhases * kBatch) {
        typename Src::F f[kBatch];
#pragma unroll
        for (int jj = 0; jj < kBatch; ++jj) {
          f[jj].zero();
          if (on && j0 + jj * kPhases < r) src.row(f[jj], 0, j0 + jj * kPhases, rot);
          rot += rstep;
          if (rot >= ng) rot -= ng;
        }
#pragma unroll
        for (int jj = 0; jj < kBatch; ++jj) {
          const int j = min(j0 + jj * kPhases, kHeadDim - 1);   // a row past r was loaded as zeros
#pragma unroll
          for (int h = 0; h < GH; ++h) {
            const float qv = j0 + jj * kPhases < r ? q_s[j][h] : 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) sc[h][i] = fmaf(qv, f[jj].get(i), sc[h][i]);
          }
        }
      }
      __syncwarp();
      // online softmax over this item
#pragma unroll
      for (int h = 0; h < GH; ++h) {
        float mloc = -INFINITY;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) sc[h][i] += __shfl_xor_sync(0xffffffffu, sc[h][i], o);
          if (s0 + i >= n) sc[h][i] = -INFINITY;
          mloc = fmaxf(mloc, sc[h][i]);
        }
        mloc = fmaxf(mloc, __shfl_xor_sync(0xffffffffu, mloc, 1));
        mloc = fmaxf(mloc, __shfl_xor_sync(0xffffffffu, mloc, 2));
        const float nm = fmaxf(M[h], mloc);
        const float ref = nm == -INFINITY ? 0.f : nm;     // every score so far is -inf: weights 0, not NaN
        const float corr = exp2f(M[h] - ref);
        float sum = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) { sc[h][i] = exp2f(sc[h][i] - ref); sum += sc[h][i]; }
        Ls[h] = Ls[h] * corr + sum;
        M[h] = nm;
#pragma unroll
        for (int a = 0; a < kRowsPer; ++a) acc[a][h] *= corr;
      }

      // weighted value rows
      rot = rot0;
#pragma unroll
      for (int a0 = 0; a0 < kRowsPer; a0 += kBatch) {
        if (a0 * kPhases >= r) break;                   // warp-uniform
        typename Src::F f[kBatch];
#pragma unroll
        for (int jj = 0; jj < kBatch; ++jj) {
          const int j = phase + (a0 + jj) * kPhases;
          f[jj].zero();
          if (on && j < r) src.row(f[jj], 1, j, rot);
          rot += rstep;
          if (rot >= ng) rot -= ng;
        }
#pragma unroll
        for (int jj = 0; jj < kBatch; ++jj)
#pragma unroll
          for (int h = 0; h < GH; ++h) {
            float a2 = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) a2 = fmaf(sc[h][i], f[jj].get(i), a2);
            acc[a0 + jj][h] += a2;
          }
      }
    }
  }

  // merge the slot groups of each warp, then the warps of this CTA
#pragma unroll
  for (int h = 0; h < GH; ++h) {
    float l = Ls[h];
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    if (lane == 0) { wM[warp][h] = M[h]; wL[warp][h] = l; }
#pragma unroll
    for (int a = 0; a < kRowsPer; ++a) {
      float v = acc[a][h];
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      if (sg == 0) wacc[warp][h][phase + a * kPhases] = v;
    }
  }
  __syncthreads();
  float* out = part + ((((int64_t)b * s.G + g) * S + split) * GP + h0) * (kHeadDim + 2);
  for (int i = tid; i < GH * kHeadDim; i += blockDim.x) {
    const int h = i / kHeadDim, j = i % kHeadDim;
    float mx = -INFINITY;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) mx = fmaxf(mx, wM[w][h]);
    float o = 0.f, l = 0.f;
    if (mx != -INFINITY) {
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        const float f = exp2f(wM[w][h] - mx);
        o = fmaf(wacc[w][h][j], f, o);
        l = fmaf(wL[w][h], f, l);
      }
    }
    out[h * (kHeadDim + 2) + j] = o;
    if (j == 0) { out[h * (kHeadDim + 2) + kHeadDim] = mx; out[h * (kHeadDim + 2) + kHeadDim + 1] = l; }
  }
}

// grid (group, G, B), 512 threads, one query head each: merge partials and the exact tail, rotate back,
// normalise. Bound by latency: the weights are formed by one thread per split (S <= 128), then four
// quarters of the block sum the splits, the basis rows and the tail tokens for all 128 coordinates, with
// independent loads, and add up through shared memory in a fixed order. One CTA of 128 threads per KV head
// that walked its heads and splits one after another took 110 us for 128 splits of 4 heads, a CTA of 128
// threads per head 23 us, this 19 us (cold).
constexpr int kCombThreads = 512;
constexpr int kCombParts = kCombThreads / kHeadDim;

template <typename T, int GP>
__global__ void __launch_bounds__(kCombThreads)
decode_combine_kernel(const float* __restrict__ part, const T* __restrict__ q,
                      const T* __restrict__ basis_v, const T* __restrict__ tail_k,
                      const T* __restrict__ tail_v, int n_tail, T* __restrict__ out, Shape s,
                      int layer, int S) {
  __shared__ float ot[kCombParts][kHeadDim], yt[kCombParts][kHeadDim];
  __shared__ float lt[2][kCombParts];                 // softmax sums: of the splits, of the tail
  __shared__ float tsc[kMaxTail];
  __shared__ float wgt[kMaxSplits], lsum[kMaxSplits];
  __shared__ float red[kCombThreads / 32];
  const int hh = blockIdx.x, g = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int quart = tid / kHeadDim, col = tid % kHeadDim;
  const T* U = basis_v + ((int64_t)layer * s.G + g) * kHeadDim * kHeadDim;
  const float scale = kLog2e * rsqrtf((float)kHeadDim);
  const float* pb = part + (((int64_t)b * s.G + g) * S * GP + hh) * (kHeadDim + 2);
  constexpr int kStep = GP * (kHeadDim + 2);   // floats between the splits of a head
  const int h = g * s.grp + hh;
  // exact tail scores (log2 units)
  float mloc = -INFINITY;
  if (n_tail > 0) {
    const T* tk = tail_k + ((int64_t)b * s.G + g) * n_tail * kHeadDim;
    const float4 qv = load4(q + ((int64_t)b * s.H + h) * kHeadDim + lane * 4);
#pragma unroll 4
    for (int t = warp; t < n_tail; t += kCombThreads / 32) {
      const float4 kv = load4(tk + (int64_t)t * kHeadDim + lane * 4);
      float a = fmaf(qv.w, kv.w, fmaf(qv.z, kv.z, fmaf(qv.y, kv.y, qv.x * kv.x)));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      a *= scale;
      if (lane == 0) tsc[t] = a;
      mloc = fmaxf(mloc, a);
    }
  }
  // this thread's part of U_V, in flight while the partials are merged
  constexpr int kRows = kHeadDim / kCombParts;
  float u[kRows];
#pragma unroll
  for (int j = 0; j < kRows; ++j) u[j] = to_f(U[(quart * kRows + j) * kHeadDim + col]);
  const float m = tid < S ? pb[(int64_t)tid * kStep + kHeadDim] : -INFINITY;
  if (tid < S) lsum[tid] = pb[(int64_t)tid * kStep + kHeadDim + 1];
  mloc = fmaxf(mloc, m);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mloc = fmaxf(mloc, __shfl_xor_sync(0xffffffffu, mloc, o));
  if (lane == 0) red[warp] = mloc;
  __syncthreads();
  float mx = red[0];
#pragma unroll
  for (int w = 1; w < kCombThreads / 32; ++w) mx = fmaxf(mx, red[w]);
  if (tid < S) wgt[tid] = m == -INFINITY ? 0.f : exp2f(m - mx);   // an empty split holds zeros
  __syncthreads();
  {
    float l = 0.f, o = 0.f;
#pragma unroll 16
    for (int sp = quart; sp < S; sp += kCombParts) {
      l = fmaf(lsum[sp], wgt[sp], l);
      o = fmaf(pb[(int64_t)sp * kStep + col], wgt[sp], o);
    }
    ot[quart][col] = o;
    if (col == 0) lt[0][quart] = l;
  }
  float y = 0.f, l = 0.f;
  if (n_tail > 0) {
    const T* tv = tail_v + ((int64_t)b * s.G + g) * n_tail * kHeadDim;
#pragma unroll 8
    for (int t = quart; t < n_tail; t += kCombParts) {
      const float p = exp2f(tsc[t] - mx);
      l += p;
      y = fmaf(p, to_f(tv[(int64_t)t * kHeadDim + col]), y);
    }
  }
  if (col == 0) lt[1][quart] = l;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kRows; ++j) {
    float o = 0.f;
#pragma unroll
    for (int i = 0; i < kCombParts; ++i) o += ot[i][quart * kRows + j];
    y = fmaf(u[j], o, y);
  }
  yt[quart][col] = y;
  __syncthreads();
  if (quart == 0) {
    float sum = 0.f, l = 0.f;
#pragma unroll
    for (int i = 0; i < kCombParts; ++i) { sum += yt[i][col]; l += lt[0][i] + lt[1][i]; }
    out[((int64_t)b * s.H + h) * kHeadDim + col] = from_f<T>(sum / l);
  }
}

template <typename T, int GP>
void launch_decode_t(const Shape& s, const varrate_packed& c, const void* basis_k, const void* basis_v,
                     const void* q, int layer, const void* tail_k, const void* tail_v, int n_tail,
                     void* out, float* qt, float* part, int S, cudaStream_t st) {
  decode_rotate_kernel<T><<<dim3(s.G, s.B, kRotSplit), 256, 0, st>>>((const T*)q, (const T*)basis_k, qt, s, layer);
  constexpr int GH = GP < 4 ? GP : 4;
  DenseSrc<T> src{(const T*)c.coef, c.bucket_base, s.cap, nullptr, nullptr, 0};
  decode_split_kernel<DenseSrc<T>, GP, GH><<<dim3(S * (GP / GH), s.G, s.B), 256, 0, st>>>(
      src, c.bucket_count, qt, part, s, layer, S, 0);
  decode_combine_kernel<T, GP><<<dim3(s.grp, s.G, s.B), kCombThreads, 0, st>>>(part, (const T*)q, (const T*)basis_v,
                                                               (const T*)tail_k, (const T*)tail_v,
                                                               n_tail, (T*)out, s, layer, S);
}

template <typename T>
void dispatch_gp(int gp, const Shape& s, const varrate_packed& c, const void* bk, const void* bv,
                 const void* q, int layer, const void* tk, const void* tv, int nt, void* out,
                 float* qt, float* part, int S, cudaStream_t st) {
  switch (gp) {
    case 1: launch_decode_t<T, 1>(s, c, bk, bv, q, layer, tk, tv, nt, out, qt, part, S, st); break;
    case 2: launch_decode_t<T, 2>(s, c, bk, bv, q, layer, tk, tv, nt, out, qt, part, S, st); break;
    case 4: launch_decode_t<T, 4>(s, c, bk, bv, q, layer, tk, tv, nt, out, qt, part, S, st); break;
    default: launch_decode_t<T, 8>(s, c, bk, bv, q, layer, tk, tv, nt, out, qt, part, S, st); break;
  }
}

int group_pad(int grp) { return grp <= 1 ? 1 : grp <= 2 ? 2 : grp <= 4 ? 4 : 8; }

template <int GP>
void launch_decode_qt(const Shape& s, const varrate_qpacked& c, const void* basis_k, const void* basis_v,
                      const void* q, int layer, const void* tail_k, const void* tail_v, int n_tail,
                      void* out, float* qt, float* part, int S, cudaStream_t st) {
  using bf = __nv_bfloat16;
  constexpr int GH = GP < 4 ? GP : 4;
  decode_rotate_kernel<bf><<<dim3(s.G, s.B, kRotSplit), 256, 0, st>>>((const bf*)q, (const bf*)basis_k, qt, s, layer);
  if (c.bits == 4) {
    QuantSrc<4> src{c.data, c.qbase, c.qcap_bytes, nullptr, nullptr, 0, 0};
    decode_split_kernel<QuantSrc<4>, GP, GH><<<dim3(S * (GP / GH), s.G, s.B), 256, 0, st>>>(
        src, c.bucket_count, qt, part, s, layer, S, c.qcap_bytes);
  } else {
    QuantSrc<8> src{c.data, c.qbase, c.qcap_bytes, nullptr, nullptr, 0, 0};
    decode_split_kernel<QuantSrc<8>, GP, GH><<<dim3(S * (GP / GH), s.G, s.B), 256, 0, st>>>(
        src, c.bucket_count, qt, part, s, layer, S, c.qcap_bytes);
  }
  decode_combine_kernel<bf, GP><<<dim3(s.grp, s.G, s.B), kCombThreads, 0, st>>>(part, (const bf*)q, (const bf*)basis_v,
                                                               (const bf*)tail_k, (const bf*)tail_v,
                                                               n_tail, (bf*)out, s, layer, S);
}

}  // namespace

int decode_splits(const Shape& s, int num_sms) {
  const int64_t units = (int64_t)s.B * s.G;
  int64_t S = (4LL * num_sms + units - 1) / units;
  if (S < 1) S = 1;
  if (S > kMaxSplits) S = kMaxSplits;
  return (int)S;
}

size_t decode_ws_bytes(const Shape& s, int num_sms) {
  const int S = decode_splits(s, num_sms);
  size_t a = (size_t)s.B * s.H * kHeadDim * sizeof(float);
  a = (a + 255) & ~size_t(255);
  a += (size_t)s.B * s.G * S * group_pad(s.grp) * (kHeadDim + 2) * sizeof(float);
  const size_t m = decode_mma_part_bytes(s, num_sms);
  if (m > a) a = m;
  return kDecodeCounterBytes + ((a + 255) & ~size_t(255));
}

int launch_decode(const Shape& s, const varrate_packed& cache, const void* basis_k,
                  const void* basis_v, const void* q, int layer, const void* tail_k,
                  const void* tail_v, int n_tail, void* out, int32_t* dev_status, void* ws,
                  int num_sms, cudaStream_t st) {
  void* header = ws;   // completion counting: the first kDecodeCounterBytes of the workspace
  ws = static_cast<char*>(ws) + kDecodeCounterBytes;
  if (decode_mma_supported(s, n_tail, num_sms))
    return launch_decode_mma(s, cache, basis_k, basis_v, q, layer, tail_k, tail_v, n_tail, out,
                             dev_status, header, reinterpret_cast<float*>(ws), num_sms, st);
  const int S = decode_splits(s, num_sms);
  float* qt = reinterpret_cast<float*>(ws);
  size_t a = (size_t)s.B * s.H * kHeadDim * sizeof(float);
  a = (a + 255) & ~size_t(255);
  float* part = reinterpret_cast<float*>(static_cast<char*>(ws) + a);
  const int gp = group_pad(s.grp);
  if (s.dtype == VARRATE_BF16)
    dispatch_gp<__nv_bfloat16>(gp, s, cache, basis_k, basis_v, q, layer, tail_k, tail_v, n_tail, out, qt, part, S, st);
  else
    dispatch_gp<float>(gp, s, cache, basis_k, basis_v, q, layer, tail_k, tail_v, n_tail, out, qt, part, S, st);
  return 3;
}

int launch_decode_q(const Shape& s, const varrate_qpacked& cache, const void* basis_k,
                    const void* basis_v, const void* q, int layer, const void* tail_k,
                    const void* tail_v, int n_tail, void* out, void* ws, int num_sms, cudaStream_t st) {
  ws = static_cast<char*>(ws) + kDecodeCounterBytes;   // same scratch layout as the general path
  const int S = decode_splits(s, num_sms);
  float* qt = reinterpret_cast<float*>(ws);
  size_t a = (size_t)s.B * s.H * kHeadDim * sizeof(float);
  a = (a + 255) & ~size_t(255);
  float* part = reinterpret_cast<float*>(static_cast<char*>(ws) + a);
  switch (group_pad(s.grp)) {
    case 1: launch_decode_qt<1>(s, cache, basis_k, basis_v, q, layer, tail_k, tail_v, n_tail, out, qt, part, S, st); break;
    case 2: launch_decode_qt<2>(s, cache, basis_k, basis_v, q, layer, tail_k, tail_v, n_tail, out, qt, part, S, st); break;
    case 4: launch_decode_qt<4>(s, cache, basis_k, basis_v, q, layer, tail_k, tail_v, n_tail, out, qt, part, S, st); break;
    default: launch_decode_qt<8>(s, cache, basis_k, basis_v, q, layer, tail_k, tail_v, n_tail, out, qt, part, S, st); break;
  }
  return 3;
}

}  // namespace vr
