// Step 4 for a window of new tokens, bf16, more than 32 query rows per KV head: the coded part on the
// 5th-generation tensor cores (the same mathematics, cost line, q~ fragments and partials as
// decode_window.cu, whose first and last kernels run around this one).
//
// Per 128-slot item (one tile of the packed layout, rank r, R = r rounded up to 16) and 128 query rows:
//   scores  S[row][slot]  = Q~[row][j] C_K[j][slot]   M = 128, N = slots, K = R, once for the bf16 hi part of q~
//                                                     and once for the lo part
//   values  O[row][j]    += P[row][slot] C_V[j][slot]  M = 128, N = R, K = slots, P (bf16) read from TMEM
// A staged tile row is one coefficient of 64 consecutive slots (128 bytes, 128-byte swizzle, two panels), which
// is the MN-major image of C_K for the scores and the K-major image of C_V for the values.
//
// Two chains of seven warps take the items in turn (chain e: items of parity e) and share nothing but q~:
//   two producer warps   copy the 16-byte slot groups of a tile with cp.async from their rotated places to the
//                        swizzled ones, into the chain's ring (rows r .. R - 1 and a slot group that rounds the
//                        tile up to 16 slots are zero-filled);
//   one issuing warp     scores into the chain's score buffer, then, when the weights are there, values into its
//                        accumulator (TMEM: 2 x 128 + 2 x 128 columns);
//   four softmax warps   thread = query row: maximum, weights (bf16, over the scores they were made from), sum.
//                        The reference maximum of a row moves only when a score exceeds it by kSlack (log2
//                        units); then the row's accumulator is rescaled in TMEM.
// So the tensor work of one chain runs under the softmax of the other.
// At the end of a segment the chains merge into one partial (max, sum, o~[128]) per row.
// Bound by the two chains' latency: for a 128-slot item of rank 32 the issue of its 4 score and 8 value
// products takes 730 + 660 cycles and its softmax 2,500 of a period of 5,200 per chain. Launch times, 8 heads x
// 131072 tokens, 128 rows: 215 us with mma.sync (eight row groups in decode_window.cu), 97 us here; wide ranks, where
// most tiles are short, 590 / 124 us. Where the line between the two kernels lies stands at window_rg.
// Set aside: both groups' products from one issuing thread 125 us; weights kept in registers until the reference
// is known to stay (one pass over the scores) 175 us, with 536 bytes spilled; two threads per row 103 us.
// Every wait is bounded; one that gives up raises VARRATE_ERR_TIMEOUT, the CTA then streams nothing more and
// writes empty partials, after its copies and products in flight have ended.
#include <stddef.h>

#include <atomic>

#include "common.cuh"
#include "decode_common.cuh"
#include "kernels.h"

namespace vr {

namespace {

constexpr int kRows = 128;                                 // query rows (MMA M)
constexpr int kSoft = 8;                                   // softmax warps: four per chain
constexpr int kProd = 4;                                   // producer warps: two per chain
constexpr int kMma = 2;                                    // issuing warps: one per chain
constexpr int kThreads = (kSoft + kMma + kProd) * 32;
constexpr int kSlots = 4;                                  // ring slots of a chain: C_K and C_V of a tile of at most 32 rows each
constexpr int kQBytes = kRows * kHeadDim * 2;              // one part (hi or lo) of q~
constexpr int kSlotBytes = 32 * 512;
constexpr int kRing = 2 * kSlots * kSlotBytes;
constexpr int kPartStride = kHeadDim + 4;                  // o~[128], m, l, pad
constexpr int kQfWords = (kHeadDim / 16) * 2 * 32;         // q~ fragments of a row group, in uint4
constexpr int kRg = 8;                                     // row groups of the fragments

struct TcTables {
  uint64_t full[2][kSlots], empty[2][kSlots], sfull[2], pfull[2], ofull[2], drain[2];
  int4 info[2][kSlots];                                       // slot address, R and slots (rounded to 16) of an item
  long long base[kMaxR + 2];
  int cnt[kMaxR + 1];
  int it_lo[kMaxR + 1];
  int it_pref[kMaxR + 2];
  int err;
  uint32_t tmem;
  float M[2][kRows], L[2][kRows];
};

// K-major as sdesc_sw128; MN-major: 64-element blocks `lbo` bytes apart, 8-row groups along K 1024 bytes apart.
__device__ __forceinline__ uint64_t sdesc_sw128_mn(uint32_t saddr, uint32_t lbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
constexpr uint32_t kBMn = 1u << 16;   // instruction descriptor: B is MN-major
// The lane with `issue` set issues (the others pass by without a branch): D[tmem] (+)= A[smem] * B[smem]^T, and
// D[tmem] += A[tmem] * B[smem]^T (A: bf16 pairs, row = lane, 8 columns per K = 16).
__device__ __forceinline__ void tc_mma_bf16_if(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                               uint32_t accumulate, uint32_t issue) {
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(issue) : "memory");
}
__device__ __forceinline__ void tc_mma_bf16_ts_if(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc,
                                                  uint32_t issue) {
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, 1, 0;\n setp.ne.b32 q, %4, 0;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b), "r"(idesc), "r"(issue) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};\n"
      ::"r"(taddr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]),
      "f"(v[9]), "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]), "f"(v[16]), "f"(v[17]),
      "f"(v[18]), "f"(v[19]), "f"(v[20]), "f"(v[21]), "f"(v[22]), "f"(v[23]), "f"(v[24]), "f"(v[25]), "f"(v[26]),
      "f"(v[27]), "f"(v[28]), "f"(v[29]), "f"(v[30]), "f"(v[31]) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
      "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }

// Item i of the CTA's share, searched upward from bucket r (items are visited in increasing order).
__device__ __forceinline__ Item item_from(const TcTables& sm, int i, int r) {
  while (sm.it_pref[r + 1] <= i) ++r;
  Item x;
  x.r = r;
  x.it = sm.it_lo[r] + (i - sm.it_pref[r]);
  return x;
}
// First ring slot of a tile of R rows (a multiple of 16): 1, 2 or 4 slots, aligned to their number; `pos`
// advances past them.
__device__ __forceinline__ int slots_of(int R) { return R <= 32 ? 1 : R <= 64 ? 2 : 4; }
__device__ __forceinline__ int take_slots(int R, int& pos) {
  const int n = slots_of(R), a = (pos + n - 1) & ~(n - 1) & (kSlots - 1);
  pos = (a + n) & (kSlots - 1);
  return a;
}
__device__ __forceinline__ int item_slots(const TcTables& sm, Item x) {   // real slots, at most 128
  return (int)min((long long)ISL, sm.cnt[x.r] - (long long)x.it * ISL);
}

__global__ void __launch_bounds__(kThreads, 1)
decode_window_tc_kernel(const __nv_bfloat16* __restrict__ coef, const int32_t* __restrict__ bucket_count,
                        const int64_t* __restrict__ bucket_base, const uint4* __restrict__ qf,
                        float* __restrict__ part, int32_t* __restrict__ dev_status, Shape s, int layer, int ntt) {
  extern __shared__ __align__(1024) unsigned char raw_smem[];
  unsigned char* smem = raw_smem + ((1024 - (smem_addr(raw_smem) & 1023)) & 1023);
  unsigned char* qtile = smem;                             // hi part, lo part
  TcTables& sm = *reinterpret_cast<TcTables*>(smem + 2 * kQBytes + kRing);
  __shared__ long long segW[64];
  __shared__ long long segP[65];
  __shared__ long long cuts[kMaxCtas + 1];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int C = gridDim.x, cta = blockIdx.x;
  const int rows = 8 * ntt;                                // rows of a partial
  const uint32_t q_addr = smem_addr(qtile), ring = q_addr + 2 * kQBytes;

  pdl_trigger();
  if (tid == 0) {
    for (int e = 0; e < 2; ++e) {
      for (int i = 0; i < kSlots; ++i) { mbar_init(&sm.full[e][i], kProd / 2); mbar_init(&sm.empty[e][i], 1); }
      mbar_init(&sm.sfull[e], 1);
      mbar_init(&sm.pfull[e], 4);
      mbar_init(&sm.ofull[e], 1);
      mbar_init(&sm.drain[e], 1);
    }
    sm.err = 0;
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc(&sm.tmem, 512);
  pdl_wait();
  seg_lengths(bucket_base, s, layer, segW, segP, tid);
  const long long T = segP[64];
  for (int c2 = tid; c2 <= C; c2 += blockDim.x) cuts[c2] = cut_at(T, c2, C);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem;
  const long long lo_g = cuts[cta], hi_g = cuts[cta + 1];
  int b, g;
  segment_at(segP, segW, s.B, s.G, lo_g, b, g);
  auto seg_start = [&](int bb, int gg) { return segP[bb] + gg * (segW[bb] + kSegCost + kSegEnd) + kSegCost; };
  bool more = b < s.B && seg_start(b, g) < hi_g;

  // parities of the next completion to wait for, kept by each role for the barriers it waits on
  // every warp but for the shared parts works for one chain
  const int e = warp < kSoft ? warp >> 2 : warp < kSoft + kMma ? warp - kSoft : (warp - kSoft - kMma) >> 1;
  uint32_t n0 = 0;        // the chain's items of earlier segments: its item c uses barriers (n0 + c) mod kSlots
  int pos = 0;            // ring position (producers)
  uint32_t par_s = 0, par_p = 0, par_o = 0;
  bool dead = false;                                       // CTA-uniform

  while (more) {
    const long long W = segW[b];
    const long long P = seg_start(b, g);
    const long long lo = max(lo_g, P) - P, hi = min(hi_g, P + W) - P;
    const long long bl = (long long)b * s.L + layer;
    const long long seg = (long long)b * s.G + g;
    for (int r = tid; r <= kMaxR + 1; r += blockDim.x) {
      if (r <= kMaxR) sm.cnt[r] = bucket_count[bl * (kMaxR + 1) + r];
      sm.base[r] = bucket_base[bl * (kMaxR + 2) + r];
    }
    if (!dead) {
      // q~ of the segment from its fragments (window_qfrag_kernel) into the swizzled K-major tiles
      const uint4* src = qf + seg * kRg * kQfWords;
      for (int i = tid; i < kRg * kQfWords; i += kThreads) {
        const uint4 v = __ldg(src + i);
        const int rg = i / kQfWords, rest = i % kQfWords, jc = rest / 64, u = (rest / 32) & 1, l = rest & 31;
        const int rho = 8 * (rg + u * kRg) + (l >> 2), c = l & 3;
        unsigned char* d0 = qtile + sw128_offset(rho, 2 * jc, kRows) + 4 * c;
        unsigned char* d1 = qtile + sw128_offset(rho, 2 * jc + 1, kRows) + 4 * c;
        *reinterpret_cast<uint32_t*>(d0) = v.x;
        *reinterpret_cast<uint32_t*>(d1) = v.y;
        *reinterpret_cast<uint32_t*>(d0 + kQBytes) = v.z;
        *reinterpret_cast<uint32_t*>(d1 + kQBytes) = v.w;
      }
      fence_proxy_async_smem();
      if (warp < kSoft) {   // this group's accumulator starts at zero
        float z[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) z[k] = 0.f;
        const uint32_t o = tmem + 256 + 128 * (warp >> 2) + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll
        for (int cb = 0; cb < 4; ++cb) tmem_st32(o + 32 * cb, z);
        tmem_wait_st();
        tc_fence_before();
      }
    }
    __syncthreads();
    for (int r = tid; r <= kMaxR; r += blockDim.x) {
      long long i0 = 0, i1 = 0;
      if (r >= s.r_min && r <= s.r_max) bucket_range(sm, r, lo, hi, i0, i1);
      sm.it_lo[r] = (int)i0;
      sm.it_pref[r + 1] = (int)(i1 - i0);
    }
    __syncthreads();
    if (warp == 0) {   // inclusive scan of it_pref[1 .. 129], 5 entries per lane
      constexpr int kPer = (kMaxR + 1 + 31) / 32;
      int v[kPer], acc = 0;
#pragma unroll
      for (int e = 0; e < kPer; ++e) {
        const int r = lane * kPer + e;
        acc += r <= kMaxR ? sm.it_pref[r + 1] : 0;
        v[e] = acc;
      }
      int excl = acc;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, excl, o);
        if (lane >= o) excl += y;
      }
      excl -= acc;
#pragma unroll
      for (int e = 0; e < kPer; ++e) {
        const int r = lane * kPer + e;
        if (r <= kMaxR) sm.it_pref[r + 1] = excl + v[e];
      }
      if (lane == 0) sm.it_pref[0] = 0;
    }
    __syncthreads();
    tc_fence_after();
    const int total = dead ? 0 : (sm.it_pref[kMaxR + 1] + 1 - e) >> 1;   // the chain's items: item 2 c + e of the share
    float M = -INFINITY, L = 0.f;                                    // softmax threads: their row in their group

    if (warp >= kSoft + kMma) {
      // ------------------------------------------------------------------ producers
      const int t = tid & 63;
      const __nv_bfloat16* cK = coef + ((bl * s.G + g) * 2) * s.cap;
      // Tiles are handed on kAhead behind the copies; before a wait that needs tile q to have ended, every
      // earlier tile is handed on.
      constexpr int kAhead = 2;
      int owner[kSlots];                                             // last item in each slot, this segment
#pragma unroll
      for (int k = 0; k < kSlots; ++k) owner[k] = -1;
      int done = -1, handed = 0;            // items <= done have ended, items < handed are handed on
      auto hand_on = [&](int upto) {        // their copies have landed: visible to the tensor core, one arrival a warp
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0)
          for (int k = handed; k < upto; ++k) mbar_arrive(&sm.full[e][(n0 + k) & (kSlots - 1)]);
        handed = upto;
      };
      Item x;
      x.r = 0;
      int i = 0;
      for (; i < total; ++i) {
        x = item_from(sm, 2 * i + e, x.r);
        const int r = x.r, R = (r + 15) & ~15;
        const int n_real = item_slots(sm, x), tl = (n_real + 7) & ~7, ng = tl >> 3, ng2 = (ng + 1) & ~1;
        const __nv_bfloat16* tile = cK + sm.base[r] + (long long)x.it * ISL * r;
        const int a = take_slots(R, pos), na = slots_of(R);
        int q = i - kSlots;                                          // what has to have ended: the last user of
#pragma unroll
        for (int k = 0; k < kSlots; ++k)                             // the item's barriers and slots
          if (k >= a && k < a + na) { q = max(q, owner[k]); owner[k] = i; }
        if (q > done) {
          if (handed < i) {
            cp_async_wait<0>();
            hand_on(i);
          }
          const uint32_t n = n0 + q;
          const bool ok = mbar_wait_bounded(&sm.empty[e][n & (kSlots - 1)], (n / kSlots) & 1, kWaitTries);
          if (!__all_sync(0xffffffffu, ok)) { sm.err = 1; break; }
          done = q;
        }
        const uint32_t k0 = ring + (e * kSlots + a) * kSlotBytes, v0 = k0 + R * 256;
        if (t == 0) sm.info[e][(n0 + i) & (kSlots - 1)] = make_int4((int)k0, R, ng2 * 8, 0);
        if (ng == 16) {   // full tile: this thread's slot group of rows j0, j0 + 4, ...
          const int gd = t & 15, j0 = t >> 4;
          const uint32_t d0 = (gd >> 3) * (R * 128) + j0 * 128;
#pragma unroll 4
          for (int j = j0; j < R; j += 4) {
            const bool in = j < r;
            const __nv_bfloat16* p = in ? tile + j * ISL + ((gd + j) & 15) * 8 : tile;
            const uint32_t dst = d0 + (j - j0) * 128 + (((gd & 7) ^ (j & 7)) << 4);
            cp_async16(k0 + dst, p, in ? 16 : 0);
            cp_async16(v0 + dst, p + s.cap, in ? 16 : 0);
          }
        } else {
          const uint32_t inv = (65536u + ng2 - 1) / ng2;             // f / ng2 for f < 2048
          for (int f = t; f < R * ng2; f += 64) {
            const int j = (int)((f * inv) >> 16), gd = f - j * ng2;
            const bool in = j < r && gd < ng;
            const __nv_bfloat16* p = in ? tile + j * tl + (gd + j) % ng * 8 : tile;
            const uint32_t dst = (gd >> 3) * (R * 128) + j * 128 + (((gd & 7) ^ (j & 7)) << 4);
            cp_async16(k0 + dst, p, in ? 16 : 0);
            cp_async16(v0 + dst, p + s.cap, in ? 16 : 0);
          }
        }
        cp_async_commit();
        if (handed <= i - kAhead) {   // all but the newest kAhead tiles have landed
          cp_async_wait<kAhead>();
          hand_on(i - kAhead + 1);
        }
      }
      cp_async_wait<0>();
      hand_on(i);
    } else if (warp >= kSoft) {
      // ------------------------------------------------------------------ issuing warp: one lane issues
      // (the warp stays together, so that descriptors are formed in uniform registers)
      const uint32_t leader = lane == 0;
      const uint32_t ds = tmem + 128 * e, dout = tmem + 256 + 128 * e;
      const uint64_t qd = sdesc_sw128(q_addr);
      bool ok = true;
      for (int i = 0; i < total; ++i) {
        const uint32_t n = n0 + i, st = n & (kSlots - 1);
        // the item's tile; the chain's previous products have ended (its accumulator may be rescaled, and the
        // weights they read may be overwritten)
        ok = mbar_wait_bounded(&sm.full[e][st], (n / kSlots) & 1, kWaitTries) &&
             (i == 0 || mbar_wait_bounded(&sm.empty[e][(n - 1) & (kSlots - 1)], ((n - 1) / kSlots) & 1, kWaitTries));
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        const int4 inf = sm.info[e][st];
        const uint32_t k0 = __shfl_sync(0xffffffffu, inf.x, 0);
        const int R = __shfl_sync(0xffffffffu, inf.y, 0), n16 = __shfl_sync(0xffffffffu, inf.z, 0);
        const uint32_t idesc_s = idesc_bf16_f32(kRows, 0) | ((uint32_t)(n16 >> 3) << 17) | kBMn;
        const uint64_t kd = sdesc_sw128_mn(k0, (uint32_t)R * 128);
        for (int ks = 0; ks < (R >> 4); ++ks) {
          const uint64_t qk = qd + ((ks >> 2) * (kRows * 128) + (ks & 3) * 32) / 16;
          tc_mma_bf16_if(ds, qk, kd + ks * (2048 / 16), idesc_s, ks != 0, leader);
          tc_mma_bf16_if(ds, qk + kQBytes / 16, kd + ks * (2048 / 16), idesc_s, 1, leader);
        }
        if (leader) tc_commit(&sm.sfull[e]);
        __syncwarp();
        const uint32_t idesc_o = idesc_bf16_f32(kRows, 0) | ((uint32_t)(R >> 3) << 17);
        const uint64_t vd = sdesc_sw128(k0 + R * 256);
        const uint32_t panel = (uint32_t)R * (128 / 16);
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&sm.pfull[e], par_p, kWaitTries));
        if (!ok) break;
        par_p ^= 1;
        tc_fence_after();
        for (int ks = 0; ks < (n16 >> 4); ++ks)
          tc_mma_bf16_ts_if(dout, ds + 8 * ks, vd + (ks >> 2) * panel + (ks & 3) * 2, idesc_o, leader);
        if (leader) tc_commit(&sm.empty[e][st]);
        __syncwarp();
      }
      if (lane == 0) {
        if (ok) {
          if (total > 0) tc_commit(&sm.ofull[e]);
        } else {   // the products in flight end before TMEM is read or freed
          sm.err = 1;
          tc_commit(&sm.drain[e]);
          mbar_wait_bounded(&sm.drain[e], 0, kWaitTries);
        }
      }
      __syncwarp();
    } else {
      // ------------------------------------------------------------------ softmax: one query row per thread
      const int quarter = warp & 3;
      const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
      const uint32_t ts = tmem + 128 * e + lanes, to = tmem + 256 + 128 * e + lanes;
      const bool live = quarter * 32 < rows;               // warp-uniform: some row of the warp is a query row
      Item x;
      x.r = 0;
      bool ok = true;
      for (int i = 0; i < total && ok; ++i) {
        x = item_from(sm, 2 * i + e, x.r);
        const int n_real = item_slots(sm, x);
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&sm.sfull[e], par_s, kWaitTries));
        if (!ok) { sm.err = 1; break; }
        par_s ^= 1;
        tc_fence_after();
        if (live) {
          const int nb = (n_real + 31) / 32;
          float mx = -INFINITY;
          for (int cb = 0; cb < nb; ++cb) {
            float v[32];
            tmem_ld32(ts + 32 * cb, v);
            if (32 * cb + 32 > n_real) {
#pragma unroll
              for (int k = 0; k < 32; ++k) if (32 * cb + k >= n_real) v[k] = -INFINITY;
            }
            float m4[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
            for (int k = 4; k < 32; ++k) m4[k & 3] = fmaxf(m4[k & 3], v[k]);
            mx = fmaxf(mx, fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])));
          }
          if (__any_sync(0xffffffffu, mx > M + kSlack)) {
            const float nm = fmaxf(M, mx), corr = fast_exp2(M - nm);
            M = nm;
            L *= corr;
            // the accumulator holds every earlier item of the chain: those products have ended
#pragma unroll 1
            for (int cb = 0; cb < 4; ++cb) {
              float v[32];
              tmem_ld32(to + 32 * cb, v);
#pragma unroll
              for (int k = 0; k < 32; ++k) v[k] *= corr;
              tmem_st32(to + 32 * cb, v);
            }
          }
          for (int cb = 0; cb < nb; ++cb) {
            float v[32];
            tmem_ld32(ts + 32 * cb, v);
            float part4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 0; k < 32; ++k) v[k] = fast_exp2(v[k] - M);
            if (32 * cb + 32 > n_real) {
#pragma unroll
              for (int k = 0; k < 32; ++k) if (32 * cb + k >= n_real) v[k] = 0.f;
            }
            uint32_t p[16];
#pragma unroll
            for (int k = 0; k < 32; ++k) part4[k & 3] += v[k];
#pragma unroll
            for (int k = 0; k < 16; ++k) p[k] = pack_bf16(v[2 * k], v[2 * k + 1]);
            L += (part4[0] + part4[1]) + (part4[2] + part4[3]);
            tmem_st16(ts + 16 * cb, p);
          }
          tmem_wait_st();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.pfull[e]);
      }
      if (ok && total > 0) {   // every product of the segment has ended
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&sm.ofull[e], par_o, kWaitTries));
        if (!ok) sm.err = 1;
        par_o ^= 1;
        tc_fence_after();
      }
      sm.M[e][quarter * 32 + lane] = M;
      sm.L[e][quarter * 32 + lane] = L;
    }
    __syncthreads();
    dead = sm.err != 0;
    // one partial of (segment, CTA), in slot cta + seg (unique: a later CTA only meets later segments):
    // group e writes columns 64 e .. 64 e + 63 of both groups' merged rows
    if (warp < kSoft && (warp & 3) * 32 < rows) {
      const int rho = (warp & 3) * 32 + lane;
      const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
      const float m0 = sm.M[0][rho], m1 = sm.M[1][rho], mx = dead ? -INFINITY : fmaxf(m0, m1);
      const float w0 = mx == -INFINITY ? 0.f : fast_exp2(m0 - mx), w1 = mx == -INFINITY ? 0.f : fast_exp2(m1 - mx);
      float* pout = part + ((cta + seg) * (long long)rows + rho) * kPartStride;
      for (int cb = 2 * e; cb < 2 * e + 2; ++cb) {
        float a[32], c[32];
        if (!dead) {
          tmem_ld32(tmem + 256 + lanes + 32 * cb, a);
          tmem_ld32(tmem + 384 + lanes + 32 * cb, c);
        }
        if (rho < rows) {
#pragma unroll
          for (int k = 0; k < 32; k += 4) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (mx != -INFINITY)
              v = make_float4(fmaf(w0, a[k], w1 * c[k]), fmaf(w0, a[k + 1], w1 * c[k + 1]),
                              fmaf(w0, a[k + 2], w1 * c[k + 2]), fmaf(w0, a[k + 3], w1 * c[k + 3]));
            *reinterpret_cast<float4*>(pout + 32 * cb + k) = v;
          }
        }
        __syncwarp();
      }
      if (e == 0 && rho < rows) {
        pout[kHeadDim] = mx;
        pout[kHeadDim + 1] = mx == -INFINITY ? 0.f : fmaf(w0, sm.L[0][rho], w1 * sm.L[1][rho]);
      }
      tc_fence_before();
    }
    n0 += (uint32_t)total;
    if (++g == s.G) { ++b; g = 0; }
    while (b < s.B && segW[b] == 0) ++b;
    more = b < s.B && seg_start(b, g) < hi_g;
    __syncthreads();   // the tables, q~ and TMEM are free again
    tc_fence_after();
  }
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 512);
  if (tid == 0 && sm.err) raise_status(dev_status, VARRATE_ERR_TIMEOUT);
}

constexpr size_t window_tc_smem() { return 1024 + 2 * (size_t)kQBytes + kRing + sizeof(TcTables); }

}  // namespace

int launch_window_tc(const Shape& s, const varrate_packed& c, const uint4* qf, float* part, int32_t* dev_status,
                     int layer, int ntt, int num_sms, cudaStream_t st) {
  static std::atomic<int> smem_set[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 ||
      smem_set[dev].load(std::memory_order_acquire) == 0) {
    if (cudaFuncSetAttribute(decode_window_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)window_tc_smem()) != cudaSuccess)
      return -1;
    if (dev >= 0 && dev < 64) smem_set[dev].store(1, std::memory_order_release);
  }
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(num_sms);
  lc.blockDim = dim3(kThreads);
  lc.dynamicSmemBytes = window_tc_smem();
  lc.stream = st;
  lc.attrs = pdl;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, decode_window_tc_kernel, (const __nv_bfloat16*)c.coef, (const int32_t*)c.bucket_count,
                            (const int64_t*)c.bucket_base, qf, part, dev_status, s, layer, ntt) == cudaSuccess ? 1 : -1;
}

}  // namespace vr
