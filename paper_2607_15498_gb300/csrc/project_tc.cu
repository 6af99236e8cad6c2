// Step 3, bf16 — projection onto the per-head basis on the 5th-generation tensor cores
// (Algorithm 1's projection c_t = U x_t, Eq. 5 with the anchor mean at 0), written straight into
// the rank-bucketed layout.
//
// One CTA works for one (sequence, layer, head, K-or-V) stream, in one of two forms, chosen by the bucket table:
//
// By tile: the unit of work is a tile of the packed layout, 128 slots of one bucket (fewer at its end), whose r
// coefficient rows are one contiguous block of the stream. The CTA takes every n-th tile, with three warp roles
// over a 4-stage ring:
//   producer (4 warps)   read the tile's tokens from perm (one tile ahead) and copy their rows with 16-byte
//                        cp.async (two whole rows an instruction) into the 128-byte-swizzled K-major
//                        layout of the tensor core; the copies arrive on the stage's barrier themselves
//                        when they land, so up to four tiles are in flight;
//   mma (1 thread)       8 x tcgen05.mma (M = 128 slots, N = r rounded up to 16, K = 16) with U (128 x
//                        128, resident in shared memory) as B, into one of four TMEM accumulators;
//                        tcgen05.commit frees the stage and hands the accumulator on;
//   epilogue (12 warps)  three groups of four take the tiles round-robin (each group covers the 128 TMEM
//                        lanes); thread = slot: its TMEM row 32 columns at a time as bf16 into a staging
//                        block laid out as the packed tile (rotated 8-slot groups, padding slots zero),
//                        which one bulk copy then writes to the stream.
// By token: the CTA takes 128 consecutive tokens at a time, with
//   producer (1 thread)  two TMA loads a step (64 columns x 128 rows each) into a 5-stage ring;
//   mma (1 thread)       as above, N = 128;
//   epilogue (16 warps)  four groups; thread = token: its rank and its position in the bucket, then coefficient
//                        j < r to its slot, 2 bytes a store. The padding slots are zeroed up front.
//
// Bound by HBM: K and V are read once (by tile as 256-byte rows in bucket order) and the coefficients written once.
// By tile a step costs about the same whatever the number of its slots, so short tiles waste it; by token a
// step costs a store instruction's transactions for every row and every rank among a warp's 32 tokens,
//   S = sum over r of r (1 - (1 - n_r / N)^32)
// for tokens of independent ranks. A step on one SM, from launch times of 64 and 32 layers x 8 heads: by tile 0.95 us;
// by token 0.85 us for one rank (S = 24), 0.89 for three (75), 0.97 for four (102), 1.23 for six (159), 1.52 for
// eight (217), 2.10 and 2.83 for heavy-tailed ranks (357, 449): about max(0.9, 0.38 + 0.0055 S), and the rule compares
// the two sums. By token / by tile in us: 32 x 8 x 32768 tokens of one rank 734 / 818, of six 1061 / 840; heavy-tailed
// 64 x 8 x 16384 2440 / 1409, 64 x 8 x 600 184 / 347, 1 x 8 x 600 13.5 / 18.1.
// Set aside: TMA gathers of four rows as the producer by tile (about 85 cycles a gather on an SM: 2 to 3 times
// slower); producers that wait for a tile's copies and fence before they hand it on (the fence also waits for the
// copies of later tiles: 870 us where the arrival takes 819); tokens read four tiles ahead (no gain); the stores by
// token unrolled over all 128 rows (code that costs the form by tile 1.5 to 4 us a call).
// Every mbarrier wait is bounded; a timeout raises VARRATE_ERR_TIMEOUT.
#include <cudaTypedefs.h>

#include "common.cuh"
#include "kernels.h"

namespace vr {

namespace {

constexpr int kMaxR = kHeadDim;
constexpr int TM = 128;                    // slots per tile
constexpr int NST = 4;                     // operand stages
constexpr int TILE_BYTES = TM * kHeadDim * 2;
constexpr int NGRP = 3;                    // epilogue groups of four warps (tiles round-robin)
constexpr int kEpi = 4 * NGRP;             // epilogue warps
constexpr int NACC = 4;                    // TMEM accumulators of 128 columns (all 512 columns)
constexpr int kProd = 4;                   // producer warps (32 slots each)
constexpr int kMmaWarp = kEpi + kProd, kTmaWarp = kMmaWarp + 1;   // the TMA warp works by token only
constexpr int kThreads = (kTmaWarp + 1) * 32;
constexpr int STG_BYTES = 32 * TM * 2;     // staging block: 32 coefficient rows
constexpr int NST_TOK = NST + 1;           // operand stages by token: the staging blocks' memory is the fifth
constexpr int NGRP_TOK = 4;                // epilogue groups by token: the producers' warps too
static_assert(NGRP * 2 * STG_BYTES >= TILE_BYTES && 4 * NGRP_TOK == kMmaWarp, "roles by token");
constexpr uint32_t kWaitTries = 1u << 22;  // bounded mbarrier polls

struct ProjSmem {
  uint64_t full[NST_TOK], empty[NST_TOK], tfull[NACC], tempty[NACC], drain;
  uint32_t tmem_base;
  int err;
  int by_token;
  int count[kMaxR + 1];
  int tile_pre[kMaxR + 2];                 // tiles of the buckets before r
  int slot_start[kMaxR + 2];               // tokens of the buckets before r
  long long base[kMaxR + 2];
};

// 1-D bulk copy shared -> global (16-byte aligned, size a multiple of 16) in the thread's bulk group.
__device__ __forceinline__ void bulk_s2g(void* dst, uint32_t src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n cp.async.bulk.commit_group;\n"
               ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
// At most N of the thread's bulk groups still read shared memory.
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;\n" ::"n"(N) : "memory");
}

// This thread's copies issued so far arrive on `bar` (counted among its expected arrivals) when they have landed.
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive_n(uint64_t* bar, uint32_t n) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(n) : "memory");
}

// By token or by tile (the rule and its measurements stand at the head of the file).
__device__ __forceinline__ bool by_token_cheaper(float S, float steps, float tiles) {
  return steps * fmaxf(0.9f, fmaf(0.0055f, S, 0.38f)) < 0.95f * tiles;
}

// Bucket of tile T, searched upward from r (tiles are visited in increasing order).
__device__ __forceinline__ int bucket_of(const int* tile_pre, int T, int r) {
  while (tile_pre[r + 1] <= T) ++r;
  return r;
}

__device__ __forceinline__ void project_by_tile(ProjSmem& sm, const __nv_bfloat16* __restrict__ x,
                                                const int32_t* __restrict__ perm, unsigned char* staging,
                                                uint32_t stage0, uint32_t u_addr, uint32_t tmem, __nv_bfloat16* out) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int T_all = sm.tile_pre[kMaxR + 1], x0 = blockIdx.x, dx = gridDim.x;
  const int n_tiles = T_all > x0 ? (T_all - x0 + dx - 1) / dx : 0;   // tiles x0, x0 + dx, ...

  if (warp >= kEpi && warp < kMmaWarp) {
    // ------------------------------------------------------------------ producers: 32 slots a warp
    const unsigned char* src = reinterpret_cast<const unsigned char*>(x) + (lane & 15) * 16;
    const int row0 = (warp - kEpi) * 32;
    // tokens of tile i: this lane's slot (the last one repeated past the bucket's end), n slots in all
    int r = 0, n = 0, tok = 0;
    auto tokens = [&](int i) {
      if (i >= n_tiles) return;
      const int T = x0 + i * dx;
      r = bucket_of(sm.tile_pre, T, r);
      const int p0 = (T - sm.tile_pre[r]) * TM;
      n = min(TM, sm.count[r] - p0);
      tok = __ldg(perm + sm.slot_start[r] + p0 + min(row0 + lane, n - 1));
    };
    tokens(0);
    int i = 0;
    for (; i < n_tiles; ++i) {
      const int st = i % NST, ni = n, ti = tok;
      tokens(i + 1);
      const bool ok = mbar_wait_bounded(&sm.empty[st], ((i / NST) & 1) ^ 1, kWaitTries);
      if (!__all_sync(0xffffffffu, ok)) { sm.err = 1; break; }
      const uint32_t dst = stage0 + st * TILE_BYTES;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int sub = 2 * q + (lane >> 4);
        const int t = __shfl_sync(0xffffffffu, ti, sub);
        if (row0 + sub < ni)
          cp_async16(dst + sw128_offset(row0 + sub, lane & 15, TM), src + (int64_t)t * (kHeadDim * 2), 16);
      }
      cp_async_arrive(&sm.full[st]);
    }
    cp_async_wait_all();    // also after a wait that gave up: nothing is in flight when the block ends
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      int r = 0;
      for (int i = 0; i < n_tiles; ++i) {
        const int st = i % NST, b = i % NACC;
        if (!mbar_wait_bounded(&sm.full[st], (i / NST) & 1, kWaitTries) ||
            !mbar_wait_bounded(&sm.tempty[b], ((i / NACC) & 1) ^ 1, kWaitTries)) {
          sm.err = 1;
          tc_commit(&sm.drain);   // the products in flight end before TMEM is freed
          mbar_wait_bounded(&sm.drain, 0, kWaitTries);
          break;
        }
        fence_proxy_async_smem();   // the rows were copied by ordinary (generic) writes
        tc_fence_after();
        r = bucket_of(sm.tile_pre, x0 + i * dx, r);
        const uint32_t idesc = idesc_bf16_f32(TM, (r + 15) & ~15);   // rows of U past r are not needed
        const uint32_t a0 = stage0 + st * TILE_BYTES;
        const uint32_t d = tmem + (uint32_t)(b * kHeadDim);
#pragma unroll
        for (int ks = 0; ks < kHeadDim / 16; ++ks) {
          const uint32_t off = (ks >> 2) * (TM * 128) + (ks & 3) * 32;
          tc_mma_bf16(d, sdesc_sw128(a0 + off), sdesc_sw128(u_addr + off), idesc, ks > 0 ? 1u : 0u);
        }
        tc_commit(&sm.empty[st]);
        tc_commit(&sm.tfull[b]);
      }
    }
  } else if (warp < kEpi) {
    // ------------------------------------------------------------------ epilogue
    bool bad = false;
    const int eg = warp >> 2, row = tid & (TM - 1);   // epilogue group (tiles eg, eg + NGRP, ...), slot
    unsigned char* stg = staging + eg * 2 * STG_BYTES;
    int r = 0, blk = 0;
    for (int i = eg; i < n_tiles; i += NGRP) {
      const int b = i % NACC, T = x0 + i * dx;
      r = bucket_of(sm.tile_pre, T, r);
      const int p0 = (T - sm.tile_pre[r]) * TM;
      const int m = min(TM, sm.count[r] - p0);          // tokens of the tile
      const int tl = (m + 7) & ~7, ng = tl >> 3;        // its slots
      __nv_bfloat16* tile = out + sm.base[r] + (long long)p0 * r;
      if (!bad && !mbar_wait_bounded(&sm.tfull[b], (i / NACC) & 1, kWaitTries)) { sm.err = 1; bad = true; }
      tc_fence_after();
      const uint32_t taddr = tmem + (uint32_t)(b * kHeadDim) + ((uint32_t)((warp & 3) * 32) << 16);
      int grp = row < tl ? row >> 3 : 0;
      for (int c0 = 0; c0 < r; c0 += 32, ++blk) {
        const int nj = min(32, r - c0);
        float vals[32];
        tmem_ld32(taddr + c0, vals);   // columns past r hold older values: not used
        unsigned char* buf = stg + (blk & 1) * STG_BYTES;
        if (row == 0) bulk_wait_read<1>();   // the block written two rounds ago has left this buffer
        named_sync(1 + eg, 128);
        if (row < tl) {
          unsigned char* dst = buf + (row & 7) * 2;
#pragma unroll
          for (int jj = 0; jj < 32; ++jj) {
            if (jj < nj)
              *reinterpret_cast<__nv_bfloat16*>(dst + jj * tl * 2 + grp * 16) =
                  __float2bfloat16_rn(row < m ? vals[jj] : 0.f);
            grp = (grp + 1 == ng) ? 0 : grp + 1;
          }
        }
        fence_proxy_async_smem();
        named_sync(1 + eg, 128);
        if (row == 0 && !bad) bulk_s2g(tile + (long long)c0 * tl, smem_addr(buf), (uint32_t)(nj * tl * 2));
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.tempty[b]);
    }
    if (row == 0) asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
  }
}

// tmap: rows of the [B L G N][128] view; row0: the stream's first row.
__device__ __forceinline__ void project_by_token(ProjSmem& sm, const CUtensorMap* tmap, uint32_t stage0, uint32_t u_addr,
                                                 uint32_t tmem, const uint8_t* __restrict__ ranks,
                                                 const int32_t* __restrict__ pos, __nv_bfloat16* out, int64_t row0,
                                                 const Shape& s, int64_t chunk) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t t_begin = blockIdx.x * chunk, t_end = min(s.N, t_begin + chunk);
  const int n_tiles = t_end > t_begin ? (int)((t_end - t_begin + TM - 1) / TM) : 0;
  if (warp == kTmaWarp) {
    // ------------------------------------------------------------------ producer
    if (lane == 0) {
      int i = 0;
      for (; i < n_tiles; ++i) {
        const int st = i % NST_TOK;
        if (!mbar_wait_bounded(&sm.empty[st], ((i / NST_TOK) & 1) ^ 1, kWaitTries)) { sm.err = 1; break; }
        const uint32_t dst = stage0 + st * TILE_BYTES;
        mbar_arrive_n(&sm.full[st], kProd * 32 - 1);   // by tile every producer thread arrives
        mbar_arrive_expect_tx(&sm.full[st], TILE_BYTES);
        // rows past the stream's end belong to the next stream (or read as zero): their results
        // are never stored
        const int row = (int)(row0 + t_begin + (int64_t)i * TM);
        tma_load_2d(dst, tmap, 0, row, &sm.full[st]);
        tma_load_2d(dst + TM * 128, tmap, 64, row, &sm.full[st]);
      }
      // every copy has landed before the block ends, also after a wait that gave up
      for (int j = max(0, i - NST_TOK); j < i; ++j)
        mbar_wait_bounded(&sm.full[j % NST_TOK], (j / NST_TOK) & 1, kWaitTries);
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(TM, kHeadDim);
      for (int i = 0; i < n_tiles; ++i) {
        const int st = i % NST_TOK, b = i % NACC;
        if (!mbar_wait_bounded(&sm.full[st], (i / NST_TOK) & 1, kWaitTries) ||
            !mbar_wait_bounded(&sm.tempty[b], ((i / NACC) & 1) ^ 1, kWaitTries)) {
          sm.err = 1;
          tc_commit(&sm.drain);   // the products in flight end before TMEM is freed
          mbar_wait_bounded(&sm.drain, 0, kWaitTries);
          break;
        }
        tc_fence_after();
        const uint32_t a0 = stage0 + st * TILE_BYTES;
        const uint32_t d = tmem + (uint32_t)(b * kHeadDim);
#pragma unroll
        for (int ks = 0; ks < kHeadDim / 16; ++ks) {
          const uint32_t off = (ks >> 2) * (TM * 128) + (ks & 3) * 32;
          tc_mma_bf16(d, sdesc_sw128(a0 + off), sdesc_sw128(u_addr + off), idesc, ks > 0 ? 1u : 0u);
        }
        tc_commit(&sm.empty[st]);
        tc_commit(&sm.tfull[b]);
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue
    // padding slots [n, pad8(n)) of the buckets, a warp each: the end of the last 8-slot group of every row
    for (int r = warp + 4 * NGRP_TOK * blockIdx.x; r <= kMaxR; r += 4 * NGRP_TOK * gridDim.x) {
      const int n = sm.count[r], n8 = (n + 7) & ~7;
      if (n == n8) continue;
      const int p0 = (n8 - 1) & ~(TM - 1), tl = n8 - p0, ng = tl >> 3;
      __nv_bfloat16* tile = out + sm.base[r] + (long long)p0 * r;
      for (int j = lane; j < r; j += 32)
        for (int e = n & 7; e < 8; ++e) tile[j * tl + (ng - 1 + j) % ng * 8 + e] = __float2bfloat16_rn(0.f);
    }
    bool bad = false;
    const int eg = warp >> 2, row = tid & (TM - 1);   // epilogue group (steps eg, eg + NGRP_TOK, ...), token row
    // rank and bucket position of this thread's token, one step of its group ahead of its use
    auto meta = [&](int i, int& r, int& p) {
      const int64_t t = t_begin + (int64_t)i * TM + row;
      const bool ok = i < n_tiles && t < t_end;
      r = ok ? (int)ranks[t] : 0;
      p = ok ? pos[t] : 0;
    };
    int r_next, p_next;
    meta(eg, r_next, p_next);
    for (int i = eg; i < n_tiles; i += NGRP_TOK) {
      const int b = i % NACC;
      const int r = r_next, p = p_next;
      meta(i + NGRP_TOK, r_next, p_next);
      const bool valid = r >= s.r_min && r <= s.r_max;   // a token of this stream, rank in range
      if (!bad && !mbar_wait_bounded(&sm.tfull[b], (i / NACC) & 1, kWaitTries)) { sm.err = 1; bad = true; }
      tc_fence_after();
      const int rmax_w = __reduce_max_sync(0xffffffffu, valid ? r : 0);
      // this slot's position in its 128-slot tile (coef_offset): the row of coefficient j starts at
      // tile + j * tl, the slot's 8-group rotates by one position per row
      const int rr = valid ? r : s.r_min;
      const int p0 = p & ~(TM - 1), pl = p - p0;
      const int tl = min(TM, ((sm.count[rr] + 7) & ~7) - p0);
      const int ng = max(tl >> 3, 1);
      __nv_bfloat16* tile = out + sm.base[rr] + (long long)p0 * rr + (pl & 7);
      const uint32_t taddr = tmem + (uint32_t)(b * kHeadDim) + ((uint32_t)((warp & 3) * 32) << 16);
      int grp = (pl >> 3) % ng;
#pragma unroll 1
      for (int cb = 0; cb < kHeadDim / 32; ++cb) {
        if (cb * 32 >= rmax_w) break;          // warp-uniform
        float vals[32];
        tmem_ld32(taddr + cb * 32, vals);
#pragma unroll
        for (int jj = 0; jj < 32; ++jj) {
          const int j = cb * 32 + jj;
          if (!bad && valid && j < r) tile[j * tl + grp * 8] = __float2bfloat16_rn(vals[jj]);
          grp = (grp + 1 == ng) ? 0 : grp + 1;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.tempty[b]);
    }
  }
}

__global__ void __launch_bounds__(kThreads, 1)
project_tc_kernel(const __grid_constant__ CUtensorMap tk, const __grid_constant__ CUtensorMap tv,
                  const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                  const __nv_bfloat16* __restrict__ basis_k, const __nv_bfloat16* __restrict__ basis_v,
                  const int32_t* __restrict__ bucket_count, const int64_t* __restrict__ bucket_base,
                  const int32_t* __restrict__ perm, const uint8_t* __restrict__ ranks,
                  const int32_t* __restrict__ pos, __nv_bfloat16* __restrict__ coef,
                  int32_t* __restrict__ dev_status, Shape s, int64_t chunk) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // 1024-byte alignment for the swizzled operand tiles
  unsigned char* smem = smem_raw + ((1024 - (smem_addr(smem_raw) & 1023)) & 1023);
  unsigned char* u_tile = smem;                                   // U, 32 KB
  unsigned char* stages = smem + TILE_BYTES;                      // NST x 32 KB
  unsigned char* staging = stages + NST * TILE_BYTES;             // 2 x 8 KB per epilogue group
  ProjSmem& sm = *reinterpret_cast<ProjSmem*>(staging + NGRP * 2 * STG_BYTES);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t bl = blockIdx.z;
  const int g = blockIdx.y >> 1, kv = blockIdx.y & 1;
  const int64_t l = bl % s.L;

  for (int r = tid; r <= kMaxR + 1; r += blockDim.x) {
    if (r <= kMaxR) sm.count[r] = bucket_count[bl * (kMaxR + 1) + r];
    sm.base[r] = bucket_base[bl * (kMaxR + 2) + r];
  }
  if (tid == 0) sm.err = 0;
  __syncthreads();
  if (sm.base[kMaxR + 1] > s.cap || sm.base[kMaxR + 1] < 0) return;   // reported by pack_tables

  // U of this head into shared memory (row j = basis vector j), swizzled K-major
  const __nv_bfloat16* U = (kv ? basis_v : basis_k) + (l * s.G + g) * (int64_t)kHeadDim * kHeadDim;
  for (int idx = tid; idx < TM * 16; idx += blockDim.x) {
    const int row = idx >> 4, c = idx & 15;
    *reinterpret_cast<uint4*>(u_tile + sw128_offset(row, c, TM)) =
        __ldg(reinterpret_cast<const uint4*>(U + (int64_t)row * kHeadDim) + c);
  }
  if (warp == kEpi && lane == 0) {
    for (int i = 0; i < NST_TOK; ++i) { mbar_init(&sm.full[i], kProd * 32); mbar_init(&sm.empty[i], 1); }
    for (int i = 0; i < NACC; ++i) { mbar_init(&sm.tfull[i], 1); mbar_init(&sm.tempty[i], 4); }
    mbar_init(&sm.drain, 1);
    fence_mbar_init();
  }
  constexpr int kPer = 5;   // ranks a lane in the warps below
  if (warp == kMmaWarp) {   // tiles and tokens before each bucket, a prefix over the lanes
    int nt = 0, ns = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int r = lane * kPer + i;
      if (r <= kMaxR) { nt += (sm.count[r] + TM - 1) / TM; ns += sm.count[r]; }
    }
    int it = nt, is = ns;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int ot = __shfl_up_sync(0xffffffffu, it, o), os = __shfl_up_sync(0xffffffffu, is, o);
      if (lane >= o) { it += ot; is += os; }
    }
    it -= nt;
    is -= ns;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int r = lane * kPer + i;
      if (r <= kMaxR + 1) { sm.tile_pre[r] = it; sm.slot_start[r] = is; }
      if (r <= kMaxR) { it += (sm.count[r] + TM - 1) / TM; is += sm.count[r]; }
    }
  }
  if (warp == kTmaWarp) {   // the form; the same for every CTA of the (sequence, layer): all read the same table
    const float inv = __fdividef(1.f, (float)(int)s.N);
    float S = 0.f;
    int tiles = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int r = lane * kPer + i;
      if (r <= kMaxR) {
        float x = 1.f - (float)sm.count[r] * inv;
#pragma unroll
        for (int e = 0; e < 5; ++e) x *= x;
        S = fmaf((float)r, 1.f - x, S);
        tiles += (sm.count[r] + TM - 1) / TM;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
    tiles = __reduce_add_sync(0xffffffffu, tiles);
    if (lane == 0) sm.by_token = by_token_cheaper(S, (float)(((int)s.N + TM - 1) / TM), (float)tiles);
  }
  if (warp == 0) tmem_alloc(&sm.tmem_base, NACC * kHeadDim);
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;

  __nv_bfloat16* out = coef + ((bl * s.G + g) * 2 + kv) * s.cap;
  const uint32_t stage0 = smem_addr(stages), u_addr = smem_addr(u_tile);
  if (sm.by_token)
    project_by_token(sm, kv ? &tv : &tk, stage0, u_addr, tmem, ranks + bl * s.N, pos + bl * s.N, out, (bl * s.G + g) * s.N, s, chunk);
  else
    project_by_tile(sm, (kv ? v : k) + (bl * s.G + g) * s.N * kHeadDim, perm + bl * s.N, staging, stage0, u_addr, tmem, out);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, NACC * kHeadDim);
  if (tid == 0 && sm.err) raise_status(dev_status, VARRATE_ERR_TIMEOUT);
}

}  // namespace

bool make_tmap_rows_bf16(CUtensorMap* map, const void* base, uint64_t rows, uint32_t box_rows);

bool pack_ready(const Shape& s, const void* k, const void* v) {
  if (s.dtype != VARRATE_BF16) return true;
  const uint64_t rows = (uint64_t)s.B * s.L * s.G * s.N;
  CUtensorMap tk, tv;
  return rows <= (uint64_t)INT32_MAX && make_tmap_rows_bf16(&tk, k, rows, TM) &&
         make_tmap_rows_bf16(&tv, v, rows, TM);
}

size_t project_tc_smem_bytes() {
  return 1024 + (size_t)(1 + NST) * TILE_BYTES + NGRP * 2 * STG_BYTES + sizeof(ProjSmem);
}

int launch_project_tc(const Shape& s, const void* k, const void* v, const void* basis_k,
                      const void* basis_v, const varrate_packed& out, int32_t* dev_status,
                      int num_sms, cudaStream_t st) {
  const uint64_t rows = (uint64_t)s.B * s.L * s.G * s.N;
  if (rows > (uint64_t)INT32_MAX) return -1;   // TMA row coordinates are 32-bit
  CUtensorMap tk, tv;
  if (!make_tmap_rows_bf16(&tk, k, rows, TM) || !make_tmap_rows_bf16(&tv, v, rows, TM)) return -1;
  // CTAs per stream: the number that makes waves x (tiles of a CTA + its set-up, about four tiles) least
  const int64_t units = (int64_t)s.B * s.L * s.G * 2;
  const double tiles = (double)s.N / TM + 8;
  int n = 1;
  double best = 1e300;
  for (int c = 1; c <= num_sms && c <= tiles; ++c) {
    const double waves = (double)((units * c + num_sms - 1) / num_sms);
    const double cost = waves * (tiles / c + 4);
    if (cost < best * 0.999) { best = cost; n = c; }
  }
  const size_t smem = project_tc_smem_bytes();
  cudaFuncSetAttribute(project_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  project_tc_kernel<<<dim3(n, s.G * 2, s.B * s.L), kThreads, smem, st>>>(
      tk, tv, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, (const __nv_bfloat16*)basis_k, (const __nv_bfloat16*)basis_v, out.bucket_count,
      out.bucket_base, out.perm, out.ranks, out.pos, (__nv_bfloat16*)out.coef, dev_status, s,
      ((s.N + TM - 1) / TM + n - 1) / n * TM);
  return 1;
}

}  // namespace vr
