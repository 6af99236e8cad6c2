// Step 3, bf16 — projection onto the per-head basis on the 5th-generation tensor cores
// (Algorithm 1's projection c_t = U x_t, Eq. 5 with the anchor mean at 0), written straight into
// the rank-bucketed layout.
//
// The unit of work is a tile of the packed layout: 128 slots of one bucket (fewer at its end), whose r
// coefficient rows are one contiguous block of the stream. One CTA takes every n-th tile of one
// (sequence, layer, head, K-or-V) stream and runs three warp roles over a 4-stage ring:
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
// Bound by HBM: K and V are read once (256-byte rows in bucket order) and the coefficients written once,
// in whole blocks. Reading the tokens in sequence order instead makes the reads sequential but scatters
// every 2-byte coefficient to its own sector when the ranks of neighbours differ.
// Scattered stores from sequence order / this kernel: 4 layers x 4 heads x 32749 tokens, heavy-tailed ranks
// 376 / 95 us (floor 49 us at the copy bandwidth); 1 layer x 8 heads x 32768, 5 % outliers 76 / 48 us; 2 x
// 8 x 131072, wide 505 / 234 us; 32 x 8 x 32768, ranks within a few units of each other 832 / 894 us. TMA
// gathers of four rows as the producer: 190, 95, 612 and 2432 us (about 85 cycles a gather on an SM).
// With the producers waiting for a tile's copies and fencing before they handed it on (the fence also waits for
// the copies of later tiles) 32 x 8 x 32768 tokens of one rank took 870 us, now 819; ranks from r_min to d 64 x 8 x
// 16384 1487 / 1396, 16 x 8 x 600 118 / 105 (launch times).
// Every mbarrier wait is bounded; a timeout raises VARRATE_ERR_TIMEOUT.
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
constexpr int kThreads = (kEpi + kProd + 1) * 32;   // + MMA warp
constexpr int STG_BYTES = 32 * TM * 2;     // staging block: 32 coefficient rows
constexpr uint32_t kWaitTries = 1u << 22;  // bounded mbarrier polls

struct ProjSmem {
  uint64_t full[NST], empty[NST], tfull[NACC], tempty[NACC], drain;
  uint32_t tmem_base;
  int err;
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

// Bucket of tile T, searched upward from r (tiles are visited in increasing order).
__device__ __forceinline__ int bucket_of(const int* tile_pre, int T, int r) {
  while (tile_pre[r + 1] <= T) ++r;
  return r;
}

__global__ void __launch_bounds__(kThreads, 1)
project_tc_kernel(const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                  const __nv_bfloat16* __restrict__ basis_k, const __nv_bfloat16* __restrict__ basis_v,
                  const int32_t* __restrict__ bucket_count, const int64_t* __restrict__ bucket_base,
                  const int32_t* __restrict__ perm, __nv_bfloat16* __restrict__ coef,
                  int32_t* __restrict__ dev_status, Shape s) {
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
    for (int i = 0; i < NST; ++i) { mbar_init(&sm.full[i], kProd * 32); mbar_init(&sm.empty[i], 1); }
    for (int i = 0; i < NACC; ++i) { mbar_init(&sm.tfull[i], 1); mbar_init(&sm.tempty[i], 4); }
    mbar_init(&sm.drain, 1);
    fence_mbar_init();
  }
  if (warp == kEpi + kProd) {   // tiles and tokens before each bucket: five ranks a lane, a prefix over the lanes
    constexpr int kPer = 5;
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
  if (warp == 0) tmem_alloc(&sm.tmem_base, NACC * kHeadDim);
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;

  __nv_bfloat16* out = coef + ((bl * s.G + g) * 2 + kv) * s.cap;
  const int T_all = sm.tile_pre[kMaxR + 1], x0 = blockIdx.x, dx = gridDim.x;
  const int n_tiles = T_all > x0 ? (T_all - x0 + dx - 1) / dx : 0;   // tiles x0, x0 + dx, ...
  const uint32_t stage0 = smem_addr(stages), u_addr = smem_addr(u_tile);

  if (warp >= kEpi && warp < kEpi + kProd) {
    // ------------------------------------------------------------------ producers: 32 slots a warp
    const unsigned char* src = reinterpret_cast<const unsigned char*>((kv ? v : k) + (bl * s.G + g) * s.N * kHeadDim) +
                               (lane & 15) * 16;
    const int32_t* pm = perm + bl * s.N;
    const int row0 = (warp - kEpi) * 32;
    // tokens of tile i: this lane's slot (the last one repeated past the bucket's end), n slots in all
    int r = 0, n = 0, tok = 0;
    auto tokens = [&](int i) {
      if (i >= n_tiles) return;
      const int T = x0 + i * dx;
      r = bucket_of(sm.tile_pre, T, r);
      const int p0 = (T - sm.tile_pre[r]) * TM;
      n = min(TM, sm.count[r] - p0);
      tok = __ldg(pm + sm.slot_start[r] + p0 + min(row0 + lane, n - 1));
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
  } else if (warp == kEpi + kProd) {
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
  } else {
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
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, NACC * kHeadDim);
  if (tid == 0 && sm.err) raise_status(dev_status, VARRATE_ERR_TIMEOUT);
}

}  // namespace

size_t project_tc_smem_bytes() {
  return 1024 + (size_t)(1 + NST) * TILE_BYTES + NGRP * 2 * STG_BYTES + sizeof(ProjSmem);
}

int launch_project_tc(const Shape& s, const void* k, const void* v, const void* basis_k,
                      const void* basis_v, const varrate_packed& out, int32_t* dev_status,
                      int num_sms, cudaStream_t st) {
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
      (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, (const __nv_bfloat16*)basis_k, (const __nv_bfloat16*)basis_v, out.bucket_count,
      out.bucket_base, out.perm, (__nv_bfloat16*)out.coef, dev_status, s);
  return 1;
}

}  // namespace vr
