// Group-wise b-bit quantization of the packed coefficients (Sec. 3.3, "Composability": the stored
// coefficients can be quantized without changing the allocation).
//
// Groups: 32 consecutive slots (tokens of one rank, in bucket order) of one coefficient row j of a
// 128-slot tile. Asymmetric min-max with fp16 offset and step:
//   lo = fp16(min), step = fp16(fl32(max - lo) / (2^b - 1)),
//   code = clip(rint(fl32(fl32(x - lo) / step)), 0, 2^b - 1)   (step = 0: code 0),
// every operation an explicitly rounded IEEE fp32 operation, so the codes are a function of the
// stored bf16 coefficients. Quantized stream layout: bucket r at byte qbase[r], its tiles back to
// back, each r rows of qrow(tl) bytes: the tl codes (b = 4: two per byte, the even slot in the low
// nibble; b = 8: one per byte), then (fp16 lo, fp16 step) for each group of 32 slots, then zero
// padding to a multiple of 16 bytes.
#include "common.cuh"
#include "kernels.h"

namespace vr {

namespace {

constexpr int kMaxR = kHeadDim;

// grid (2 G, B L, splits), 256 threads: CTA (stream, bl, z) quantizes the z-th share of the tiles of stream
// (b, l, g, kv); the first CTA of a pair writes qbase. A warp takes one tile at a time and a lane one 32-slot
// group of a row: lane (lr, qp) reads the (up to) four 8-slot groups of group qp of row j = lr, lr + rps, ...
// (8-slot group gi is stored at position (gi + j) mod (tl / 8)), finds their min and max as bf16 pairs, and writes
// the codes (16 bytes at 4 bits, 32 at 8), (lo, step) and its share of the row's zero padding.
//
// Bound by instructions, and by loads in flight. The code is rint(fl((x - lo) / step)); an IEEE division per
// coefficient took most of them. With Q = 2^b - 1 and the exact product step Q, t = (x - lo) * fl(1 / (step Q)),
// saturated to [0, 1], times Q is within 2^-23 of the quotient relatively, and the rounded quotient within
// 2^-24, so for quotients below 2^b the two are less than 1.5 * 2^(b - 23) apart: when t Q is farther than
// 2^(b - 22) from the middle between two codes, both round to the same code (and outside [0, Q] both are the
// end of the range). The few lanes with a coefficient nearer than that divide.
// A call on 16 pairs of 32768 tokens at 8 bits (645 MB read and written): 804 us (of which 41 a serial kernel
// for the tables) with a division each, 244 us without, then 205 with a lane per 32-slot group in place of four
// (no shuffles, a quarter of the work on lo and step) and 169 with pairwise min and max, mixed-precision
// differences, saturation in place of two clamps and paired fp32 operations; at 4 bits 262 -> 167 us by the last
// two. More rows in flight per lane cost resident warps: three CTAs of 80 registers 181 us, with two rows 178.
constexpr uint32_t kBias4 = 0x3F400000u;   // sum over e of 0x4B400000 * 16^e, modulo 2^32

__device__ __forceinline__ int code_exact(float d, float s32, float qmax) {
  int cq = 0;
  if (s32 != 0.f) cq = __float2int_rn(__fdiv_rn(d, s32));
  return min(max(cq, 0), (int)qmax);
}

// Two fp32 operations as one instruction, each rounded to nearest.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 c;
  asm("{\n .reg .b64 x, y;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n add.rn.f32x2 x, x, y;\n mov.b64 {%0, %1}, x;\n}\n"
      : "=f"(c.x), "=f"(c.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return c;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mov.b64 z, {%6, %7};\n"
      " fma.rn.f32x2 x, x, y, z;\n mov.b64 {%0, %1}, x;\n}\n"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
// min(max(a b, 0), 1), NaN as 0
__device__ __forceinline__ float mul_sat(float a, float b) {
  float c;
  asm("mul.rn.sat.f32 %0, %1, %2;\n" : "=f"(c) : "f"(a), "f"(b));
  return c;
}
// Both bf16 of w (exact in fp32) + a, rounded to nearest.
__device__ __forceinline__ float2 add_bf2(uint32_t w, float a) {
  float2 c;
  asm("{\n .reg .b16 l, h;\n mov.b32 {l, h}, %2;\n add.rn.f32.bf16 %0, l, %3;\n add.rn.f32.bf16 %1, h, %3;\n}\n"
      : "=f"(c.x), "=f"(c.y) : "r"(w), "f"(a));
  return c;
}
__device__ __forceinline__ __nv_bfloat162 as_bf2(uint32_t w) { return *reinterpret_cast<const __nv_bfloat162*>(&w); }

// The codes of eight coefficients by division, packed as stored. Out of line: the few lanes that need it do not
// make the others' registers spill.
template <int BITS>
__device__ __noinline__ uint2 codes_exact(uint4 x, float lo32, float s32) {
  const uint32_t w4[4] = {x.x, x.y, x.z, x.w};
  constexpr float kQmax = (float)((1 << BITS) - 1);
  uint32_t c[2] = {0, 0};
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float2 d = add_bf2(w4[k >> 1], -lo32);
    c[k * BITS / 32] |= (uint32_t)code_exact(k & 1 ? d.y : d.x, s32, kQmax) << (k * BITS % 32);
  }
  return make_uint2(c[0], c[1]);
}

template <int BITS>
__global__ void __launch_bounds__(256, 4)
quantize_kernel(const __nv_bfloat16* __restrict__ coef, const int32_t* __restrict__ bucket_count,
                const int64_t* __restrict__ bucket_base, int64_t* __restrict__ qbase,
                uint8_t* __restrict__ qdata, int32_t* __restrict__ dev_status, Shape s, int64_t qcap) {
  __shared__ int cnt[kMaxR + 1];
  __shared__ long long base[kMaxR + 2];
  __shared__ long long qb[kMaxR + 2];
  __shared__ int tiles_pre[kMaxR + 2];   // tiles of the buckets before r
  const int kv = blockIdx.x & 1, g = blockIdx.x >> 1, z = blockIdx.z;
  const int64_t bl = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int r = tid; r <= kMaxR + 1; r += blockDim.x) {
    if (r <= kMaxR) cnt[r] = bucket_count[bl * (kMaxR + 1) + r];
    base[r] = bucket_base[bl * (kMaxR + 2) + r];
  }
  __syncthreads();
  if (warp == 0) {   // tiles and bytes before each bucket: five ranks a lane, a prefix over the lanes
    constexpr int kPer = 5;
    auto bytes_of = [&](int r) -> long long {
      const int n8 = (cnt[r] + 7) & ~7, last = n8 & 127;
      return (long long)r * ((long long)(n8 >> 7) * qrow_bytes(128, BITS) + (last ? qrow_bytes(last, BITS) : 0));
    };
    auto live = [&](int r) { return r >= s.r_min && r <= s.r_max; };
    int nt = 0;
    long long nb = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int r = lane * kPer + i;
      if (live(r)) { nt += (cnt[r] + 127) >> 7; nb += bytes_of(r); }
    }
    int it = nt;
    long long ib = nb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int ot = __shfl_up_sync(0xffffffffu, it, o);
      const long long ob = __shfl_up_sync(0xffffffffu, ib, o);
      if (lane >= o) { it += ot; ib += ob; }
    }
    it -= nt;
    ib -= nb;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int r = lane * kPer + i;
      if (r <= kMaxR + 1) { tiles_pre[r] = it; qb[r] = ib; }
      if (live(r)) { it += (cnt[r] + 127) >> 7; ib += bytes_of(r); }
    }
  }
  __syncthreads();
  // a table that does not fit the buffers (corrupt ranks upstream) is skipped, and marked so that decode skips it too
  const bool fits = base[kMaxR + 1] <= s.cap && qb[kMaxR + 1] <= qcap;
  if (blockIdx.x == 0 && z == 0)
    for (int r = tid; r <= kMaxR + 1; r += blockDim.x)
      qbase[bl * (kMaxR + 2) + r] = fits || r <= kMaxR ? qb[r] : INT64_MAX;
  if (!fits) {
    if (tid == 0 && blockIdx.x == 0 && z == 0) raise_status(dev_status, VARRATE_ERR_CORRUPT);
    return;
  }
  const int64_t stream = (bl * s.G + g) * 2 + kv;
  const __nv_bfloat16* src = coef + stream * s.cap;
  uint8_t* dst = qdata + stream * qcap;
  constexpr float kQmax = (float)((1 << BITS) - 1);
  constexpr float kMid = 0.5f - (float)(1 << BITS) / 4194304.f;   // 2^(b - 22) from the middle of two codes
  constexpr float kMagic = 12582912.f;                            // 1.5 * 2^23: adding it rounds to an integer
  const int total = tiles_pre[kMaxR + 1];
  const int T0 = (int)((long long)total * z / gridDim.z), T1 = (int)((long long)total * (z + 1) / gridDim.z);
  for (int T = T0 + warp; T < T1; T += blockDim.x / 32) {
    int lo_r = 0, hi_r = kMaxR + 1;   // tiles_pre[lo_r] <= T < tiles_pre[hi_r]
    while (hi_r - lo_r > 1) {
      const int mid = (lo_r + hi_r) >> 1;
      if (tiles_pre[mid] <= T) lo_r = mid; else hi_r = mid;
    }
    const int r = lo_r;
    const long long i = T - tiles_pre[r];
    const int tl = (int)min(128ll, pad8(cnt[r]) - 128 * i);
    const int ng = tl >> 3, nq = (ng + 3) >> 2;    // 8-slot groups and 32-slot groups of a row
    const int rps = 32 / nq;                       // rows per step
    const int lr = nq == 4 ? lane >> 2 : lane / nq, qp = lane - lr * nq;
    const int qrow = qrow_bytes(tl, BITS);
    const int raw = tl * BITS / 8 + 4 * nq;
    const __nv_bfloat16* stile = src + base[r] + 128 * i * r;
    uint8_t* qtile = dst + qb[r] + i * (long long)r * qrow_bytes(128, BITS);
    const int n8 = min(4, ng - 4 * qp);            // 8-slot groups of this lane's group
    for (int j0 = 0; j0 < r; j0 += rps) {
      uint4 x[4];
      const int j = j0 + lr;
      if (lr >= rps || j >= r) continue;
      const uint4* srow = reinterpret_cast<const uint4*>(stile + j * tl);
      if (ng == 16) {
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = __ldg(srow + ((4 * qp + e + j) & 15));
      } else {
        int pos = (4 * qp + j) % ng;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (e < n8) x[e] = __ldg(srow + pos);
          pos = pos + 1 == ng ? 0 : pos + 1;
        }
      }
      __nv_bfloat162 lo2 = as_bf2(x[0].x), hi2 = lo2;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (e < n8) {
          const uint32_t w4[4] = {x[e].x, x[e].y, x[e].z, x[e].w};
#pragma unroll
          for (int k = 0; k < 4; ++k) { lo2 = __hmin2(lo2, as_bf2(w4[k])); hi2 = __hmax2(hi2, as_bf2(w4[k])); }
        }
      }
      const float2 lf = __bfloat1622float2(lo2), hf = __bfloat1622float2(hi2);
      const float mn = fminf(fminf(INFINITY, lf.x), lf.y), mx = fmaxf(fmaxf(-INFINITY, hf.x), hf.y);   // NaN: left out
      const __half lo = __float2half_rn(mn);
      const float lo32 = __half2float(lo);
      // a range beyond the fp16 range saturates the step at the largest finite fp16
      const __half st = __float2half_rn(fminf(__fdiv_rn(__fsub_rn(mx, lo32), kQmax), 65504.f));
      const float s32 = __half2float(st);
      const float inv = s32 != 0.f ? __frcp_rn(__fmul_rn(s32, kQmax)) : 0.f;   // the product is exact
      uint8_t* row = qtile + (long long)j * qrow;
      uint32_t w[BITS];   // the group's 32 codes
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (e >= n8) break;
        const uint32_t w4[4] = {x[e].x, x[e].y, x[e].z, x[e].w};
        uint32_t q[8];
        float off = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 d = add_bf2(w4[k], -lo32);
          const float2 t = make_float2(mul_sat(d.x, inv), mul_sat(d.y, inv));   // NaN: 0
          const float2 m = fma2(t, make_float2(kQmax, kQmax), make_float2(kMagic, kMagic));
          const float2 f = fma2(t, make_float2(-kQmax, -kQmax), add2(m, make_float2(-kMagic, -kMagic)));
          off = fmaxf(off, fmaxf(fabsf(f.x), fabsf(f.y)));
          q[2 * k] = __float_as_uint(m.x);   // 0x4B400000 + code
          q[2 * k + 1] = __float_as_uint(m.y);
        }
        uint2 c8;
        if (BITS == 4) {
          c8.x = q[7];
#pragma unroll
          for (int k = 6; k >= 0; --k) c8.x = (c8.x << 4) + q[k];   // the biases add up to kBias4 modulo 2^32
          c8.x -= kBias4;
        } else {
          c8.x = __byte_perm(__byte_perm(q[0], q[1], 0x0040), __byte_perm(q[2], q[3], 0x0040), 0x5410);
          c8.y = __byte_perm(__byte_perm(q[4], q[5], 0x0040), __byte_perm(q[6], q[7], 0x0040), 0x5410);
        }
        if (off > kMid) c8 = codes_exact<BITS>(x[e], lo32, s32);
        w[BITS / 4 * e] = c8.x;
        if (BITS == 8) w[BITS / 4 * e + BITS / 8] = c8.y;
        if (n8 < 4) {
          if (BITS == 4) *reinterpret_cast<uint32_t*>(row + 16 * qp + 4 * e) = c8.x;
          else *reinterpret_cast<uint2*>(row + 32 * qp + 8 * e) = c8;
        }
      }
      if (n8 == 4) {
        uint4* d = reinterpret_cast<uint4*>(row + 4 * BITS * qp);
        d[0] = make_uint4(w[0], w[1], w[2], w[3]);
        if (BITS == 8) d[1] = make_uint4(w[BITS - 4], w[BITS - 3], w[BITS - 2], w[BITS - 1]);
      }
      *reinterpret_cast<__half2*>(row + tl * BITS / 8 + 4 * qp) = __halves2half2(lo, st);
      for (int z0 = raw + 4 * qp; z0 < qrow; z0 += 4 * nq) *reinterpret_cast<uint32_t*>(row + z0) = 0u;   // to a multiple of 16 bytes
    }
  }
}

}  // namespace

int launch_quantize(const Shape& s, const varrate_packed& in, const varrate_qpacked& out,
                    int32_t* dev_status, int num_sms, cudaStream_t st) {
  const int64_t pairs = (int64_t)s.B * s.L;
  // splits of a stream: sixteen CTAs of eight warps for each SM over all streams (four resident waves: 8 of them
  // 182 us against 176 for the 16 pairs above, 32 no gain), but at least four full tiles for the eight warps of a CTA
  const int64_t streams = 2 * s.G * pairs;
  int64_t z = (16LL * num_sms + streams - 1) / streams;
  const int64_t most = (s.N + 511) / 512;
  if (z > most) z = most;
  const dim3 grid(2 * s.G, (unsigned)pairs, (unsigned)(z < 1 ? 1 : z));
  if (out.bits == 4)
    quantize_kernel<4><<<grid, 256, 0, st>>>((const __nv_bfloat16*)in.coef, in.bucket_count,
                                             in.bucket_base, out.qbase, out.data, dev_status, s,
                                             out.qcap_bytes);
  else
    quantize_kernel<8><<<grid, 256, 0, st>>>((const __nv_bfloat16*)in.coef, in.bucket_count,
                                             in.bucket_base, out.qbase, out.data, dev_status, s,
                                             out.qcap_bytes);
  return 1;
}

}  // namespace vr
