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
constexpr int kGroup = 32;

// grid (2 G, B L, splits), 256 threads: CTA (stream, bl, z) quantizes the z-th share of the tiles of stream
// (b, l, g, kv); the first CTA of a pair writes qbase. A warp takes one tile at a time, its lanes as rows of
// ng4 = tl / 8 rounded up to 4: lane (lr, gp) reads the 8 bf16 coefficients of slot group gp of row
// j = lr, lr + rps, ... (stored at position (gp + j) mod (tl / 8)), the four lanes of a 32-slot group
// agree on its min and max by shuffles, and each lane writes its 8 codes (one 32-bit word at 4 bits, two
// at 8 bits); the group's first lane writes (lo, step) and the row's padding bytes are zeroed.
//
// Bound by instructions. The code is rint(fl((x - lo) / step)); an IEEE division per coefficient took
// most of them. t = (x - lo) * fl(1 / step) is within 2^-23 of the quotient relatively, and the rounded
// quotient within 2^-24, so for quotients below 2^b the two are less than 1.5 * 2^(b - 23) apart: when t is
// farther than 2^(b - 22) from the middle between two codes, both round to the same code. The few lanes
// with a coefficient nearer than that divide.
// 16 pairs of 32768 tokens at 8 bits (645 MB read and written): 787 us (of which 41 a serial kernel for the
// tables) -> 238 us; 32 pairs at 4 bits 1411 -> 484 us.
constexpr uint32_t kBias4 = 0x3F400000u;   // sum over e of 0x4B400000 * 16^e, modulo 2^32
constexpr int kStepRows = 4;   // row steps per lane whose loads are in flight together

__device__ __forceinline__ int code_exact(float d, float s32, float qmax) {
  int cq = 0;
  if (s32 != 0.f) cq = __float2int_rn(__fdiv_rn(d, s32));
  return min(max(cq, 0), (int)qmax);
}

template <int BITS>
__global__ void __launch_bounds__(256)
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
  if (blockIdx.x == 0 && z == 0)
    for (int r = tid; r <= kMaxR + 1; r += blockDim.x) qbase[bl * (kMaxR + 2) + r] = qb[r];
  // a table that does not fit the buffers (corrupt ranks upstream) is skipped
  if (base[kMaxR + 1] > s.cap || qb[kMaxR + 1] > qcap) {
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
    const int ng = tl >> 3, ng4 = (ng + 3) & ~3;
    const int rps = ng4 == 16 ? 2 : 32 / ng4;      // rows per step
    const int lr = ng4 == 16 ? lane >> 4 : lane / ng4, gp = lane - lr * ng4;
    const int qrow = qrow_bytes(tl, BITS);
    const int raw = tl * BITS / 8 + 4 * ((tl + kGroup - 1) / kGroup);
    const __nv_bfloat16* stile = src + base[r] + 128 * i * r;
    uint8_t* qtile = dst + qb[r] + i * (long long)r * qrow_bytes(128, BITS);
    const bool on = gp < ng && lr < rps;
    for (int j0 = 0; j0 < r; j0 += rps * kStepRows) {
      uint4 x[kStepRows];
#pragma unroll
      for (int u = 0; u < kStepRows; ++u) {   // every row's load in flight before the first use
        const int j = j0 + rps * u + lr;
        x[u] = make_uint4(0, 0, 0, 0);
        if (on && j < r)
          x[u] = __ldcs(reinterpret_cast<const uint4*>(stile + j * tl + 8 * (ng == 16 ? ((gp + j) & 15) : (gp + j) % ng)));
      }
#pragma unroll
      for (int u = 0; u < kStepRows; ++u) {
        if (j0 + rps * u >= r) break;   // warp-uniform: no row of this step
        const int j = j0 + rps * u + lr;
        const bool valid = on && j < r;   // other lanes may still have a row: no early exit
        float v[8];
        v[0] = __uint_as_float(x[u].x << 16); v[1] = __uint_as_float(x[u].x & 0xffff0000u);
        v[2] = __uint_as_float(x[u].y << 16); v[3] = __uint_as_float(x[u].y & 0xffff0000u);
        v[4] = __uint_as_float(x[u].z << 16); v[5] = __uint_as_float(x[u].z & 0xffff0000u);
        v[6] = __uint_as_float(x[u].w << 16); v[7] = __uint_as_float(x[u].w & 0xffff0000u);
        float mn = INFINITY, mx = -INFINITY;
        if (valid) {
          mn = fminf(fminf(fminf(v[0], v[1]), fminf(v[2], v[3])), fminf(fminf(v[4], v[5]), fminf(v[6], v[7])));
          mx = fmaxf(fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])), fmaxf(fmaxf(v[4], v[5]), fmaxf(v[6], v[7])));
        }
        // the four lanes of a 32-slot group (gp = 4 q .. 4 q + 3 of the same row)
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, 2));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const __half lo = __float2half_rn(mn);
        const float lo32 = __half2float(lo);
        // a range beyond the fp16 range saturates the step at the largest finite fp16
        const __half st = __float2half_rn(fminf(__fdiv_rn(__fsub_rn(mx, lo32), kQmax), 65504.f));
        const float s32 = __half2float(st);
        const float inv = s32 != 0.f ? __frcp_rn(s32) : 0.f;
        uint32_t q[8];
        float off = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float t = fminf(fmaxf(__fmul_rn(__fsub_rn(v[e], lo32), inv), 0.f), kQmax);   // NaN: code 0
          const float m = __fadd_rn(t, kMagic);
          off = fmaxf(off, fabsf(__fsub_rn(t, __fsub_rn(m, kMagic))));
          q[e] = __float_as_uint(m);   // 0x4B400000 + code
        }
        if (off > kMid) {
#pragma unroll
          for (int e = 0; e < 8; ++e) q[e] = 0x4B400000u + code_exact(__fsub_rn(v[e], lo32), s32, kQmax);
        }
        if (lr >= rps || j >= r) continue;
        uint8_t* row = qtile + (long long)j * qrow;
        if (on) {
          if (BITS == 4) {
            uint32_t w = q[7];
#pragma unroll
            for (int e = 6; e >= 0; --e) w = (w << 4) + q[e];   // the biases add up to kBias4 modulo 2^32
            *reinterpret_cast<uint32_t*>(row + 4 * gp) = w - kBias4;
          } else {
            *reinterpret_cast<uint2*>(row + 8 * gp) = make_uint2(
                __byte_perm(__byte_perm(q[0], q[1], 0x0040), __byte_perm(q[2], q[3], 0x0040), 0x5410),
                __byte_perm(__byte_perm(q[4], q[5], 0x0040), __byte_perm(q[6], q[7], 0x0040), 0x5410));
          }
          if ((gp & 3) == 0) *reinterpret_cast<__half2*>(row + tl * BITS / 8 + 4 * (gp >> 2)) = __halves2half2(lo, st);
        }
        for (int z0 = raw + gp; z0 < qrow; z0 += ng4) row[z0] = 0;   // zero padding of the row to its 16-byte size
      }
    }
  }
}

}  // namespace

int launch_quantize(const Shape& s, const varrate_packed& in, const varrate_qpacked& out,
                    int32_t* dev_status, int num_sms, cudaStream_t st) {
  const int64_t pairs = (int64_t)s.B * s.L;
  // splits of a stream: eight CTAs of eight warps for each SM over all streams (two resident waves), but at
  // least four full tiles for the eight warps of a CTA
  const int64_t streams = 2 * s.G * pairs;
  int64_t z = (8LL * num_sms + streams - 1) / streams;
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
