// Step 4 on a group-quantized cache (Sec. 3.3, "Composability": the stored coefficients are
// quantized without changing the allocation) — the fused tensor-core decode of decode_mma.cu with
// the coefficients expanded from each warp's ring, so a layer call reads the b-bit codes from
// HBM (31.5 % of the bf16 footprint at 4 bits, 56.5 % at 8) and nothing else of the cache.
//
// Same work split, cost line, online softmax, merge and combine as the bf16 kernel (the shared
// parts are in decode_parts.cuh). What differs:
//  - The cost line is measured in bytes of the quantized K stream (qbase), its allowances scaled
//    from the bf16 ones by the bytes of a 128-slot row (qrow(128) per 128 elements), and an item of
//    rank r spans r * qrow(128) bytes.
//  - A chunk is a run of quantized rows of one tile (qrow(tl) bytes each: the codes, then (fp16 lo,
//    fp16 step) per 32-slot group), one 1-D bulk copy into a ring stage. The codes become the
//    tensor-core fragments in registers, straight from the stage: nothing ties the order in which the
//    MMAs take a tile's slots to the order in memory, so each lane takes runs of slots. For the scores
//    (m = slots, k = rows) lane group g8 has slots 16 g8 .. 16 g8 + 15 of the lane's four rows, and a
//    byte permute pairs the codes of two rows; for the output (m = rows, k = slots) lane c has the 32
//    slots of group c of its two rows, and the pairs are 16 slots apart, which is where the scores'
//    fragments leave the weights of those slots.
//  - Expansion in fp16 half2 arithmetic: a code becomes the fp16 value 1024 + code (or 64 + code) by a
//    mask or a byte permute, the base is subtracted exactly, and code * step + lo is one fused
//    multiply-add rounded once to fp16 (the format's lo and step are fp16 already); x^ = lo + code *
//    step of the format is therefore held to within an fp16 rounding, finer than the bf16 rounding of
//    the bf16 path.
//  Bound by instructions and their latency at three warps a scheduler. With the rows first expanded into a
//  staging buffer in shared memory (16 stores and as many matrix loads for 32 rows, and the barrier between
//  them), 8 sequences of 32768 tokens at 4 bits took 84 us a layer, in fragments 63, and 58 with the rows
//  past the rank and the groups past the tile zeroed through (lo, step) instead of fragment by fragment;
//  4 sequences of spread ranks 67 -> 41 us, 1 sequence of wide ranks at 8 bits 39 -> 30.
//  - The tensor-core tiles are fp16 (mma m16n8k16 f16): q~ split hi + lo in fp16, the softmax
//    weights P in fp16 scaled by 2^kPShift (weights down to 2^-31 of the running max stay normal
//    numbers; the partials carry max - kPShift as their reference, so nothing downstream changes).
#include <atomic>

#include "common.cuh"
#include "decode_common.cuh"
#include "decode_parts.cuh"
#include "kernels.h"

namespace vr {

namespace {

constexpr int kPShift = 7;     // P in fp16 as 2^(score - max + kPShift) <= 2^(kSlack + kPShift)
static_assert(kSlack + kPShift <= 15, "scaled weights stay below the fp16 range");

// Bytes of a full 128-slot quantized row, and the cost-line allowances in bytes of the quantized
// K stream (the bf16 allowances, in elements, times the bytes per element of a full row).
template <int BITS> struct QLine {
  static constexpr long long row = ((128 * BITS / 8 + 4 * 4) + 15) & ~15;   // qrow(128)
  // ring stage: the largest chunk (4 bits: 32 rows x 80, 64 x 48 or 128 x 32 bytes; 8 bits:
  // 32 rows x 144, 64 x 80 or x 48)
  static constexpr int stage = BITS == 4 ? 4096 : 5120;
  static constexpr int stages = BITS == 4 ? 4 : 3;   // ring stages per warp (192 KB and 180 KB in all)
  static constexpr long long seg_cost = kSegCost * row / ISL;
  static constexpr long long seg_end = kSegEnd * row / ISL;
};
static_assert(QLine<4>::row == 80 && QLine<8>::row == 144, "quantized row sizes");

// Rows per chunk (log2): the bf16 kernel's chunking at 4 bits (32 rows of a full tile, 64 of one of
// at most 64 slots, 128 of one of at most 32); at 8 bits 32 rows of a tile over 64 slots and 64
// below, so that a chunk fits a stage.
__device__ __forceinline__ int chunk_lg_q(int tl, int bits) {
  return bits == 4 ? chunk_lg(tl) : (tl > 64 ? 5 : 6);
}

// Items of bucket r inside the byte range [lo, hi) of a quantized stream: [i0, i1). Item i starts
// at qbase[r] + i * r * qrow(128), so the items starting before x are ceil(x / (r * qrow(128))).
template <int BITS>
__device__ __forceinline__ void bucket_range_q(const SegSmem& sm, int r, long long lo, long long hi,
                                               long long& i0, long long& i1) {
  const int n = sm.cnt[r];
  if (n == 0) { i0 = i1 = 0; return; }
  const long long nit = (pad8(n) + ISL - 1) / ISL, b0 = sm.base[r];
  auto items_before = [&](long long x) -> long long {
    if (x <= 0) return 0;
    const unsigned long long a = ((unsigned long long)x + QLine<BITS>::row - 1) / QLine<BITS>::row;
    if (a < (1ull << 31)) return (long long)(((uint32_t)a + (uint32_t)r - 1u) / (uint32_t)r);
    return (long long)udiv_small(a + r - 1, (uint32_t)r);
  };
  i0 = items_before(lo - b0);
  i1 = items_before(hi - b0);
  if (i1 > nit) i1 = nit;
  if (i0 > i1) i0 = i1;
}

// D(16x8, fp32) += A(16x16, fp16, row) * B(16x8, fp16, col)
__device__ __forceinline__ void mma_f16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
  __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
// Two floats as fp16 hi parts and fp16 residuals: x ~ hi + lo to ~2^-22 relative.
__device__ __forceinline__ void split_f16(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  __half2 h = __floats2half2_rn(x0, x1);
  const float2 hf = __half22float2(h);
  __half2 l = __floats2half2_rn(x0 - hf.x, x1 - hf.y);
  hi = *reinterpret_cast<uint32_t*>(&h);
  lo = *reinterpret_cast<uint32_t*>(&l);
}

// Score-MMA B fragments of q~ in fp16 (hi + lo) for every 16-row chunk, one uint4 per lane.
__device__ __noinline__ void build_qfrag_f16(SegSmem& sm, int tid) {
  for (int i = tid; i < (kHeadDim / 16) * 32; i += NW * 32) {
    const int jc = i / 32, lane = i % 32, g8 = lane >> 2, c = lane & 3;
    const int j = jc * 16 + 2 * c;
    uint32_t h0, l0, h1, l1;
    split_f16(sm.qt[g8][j], sm.qt[g8][j + 1], h0, l0);
    split_f16(sm.qt[g8][j + 8], sm.qt[g8][j + 9], h1, l1);
    sm.qfrag[jc][lane][0] = h0;
    sm.qfrag[jc][lane][1] = h1;
    sm.qfrag[jc][lane][2] = l0;
    sm.qfrag[jc][lane][3] = l1;
  }
}

// Issue the next chunk of this warp's stream into `stage`: consecutive quantized rows of one tile
// are contiguous, so one bulk copy moves the chunk (qrow is a multiple of 16 bytes, and so is every
// tile and bucket start). Returns false (and issues nothing) when the stream is exhausted.
template <int BITS>
__device__ __forceinline__ bool issue_chunk_q(Prod& p, const SegSmem& sm, const uint8_t* cK, const uint8_t* cV,
                                              uint32_t stage_addr, uint64_t* bar, int total, int n_long,
                                              int lane, uint64_t policy) {
  if (p.k >= total) return false;
  const int r = p.item.r;
  const long long n8 = pad8(sm.cnt[r]);
  const long long t0 = (long long)p.item.it * ISL;            // first slot of the tile
  const int tl = (int)min((long long)ISL, n8 - t0);             // slots in the tile (multiple of 8)
  const int lgc = chunk_lg_q(tl, BITS);
  const int j0 = p.jc << lgc;
  const int rows = min(1 << lgc, r - j0);
  const int qrow = qrow_bytes(tl, BITS);
  if (lane == 0) {
    const uint32_t bytes = (uint32_t)(rows * qrow);
    mbar_arrive_expect_tx(bar, bytes);
    fence_proxy_async_smem();  // the generic reads above precede the async write
    bulk_g2s_hint(stage_addr, (p.phase ? cV : cK) + sm.base[r] + (long long)p.item.it * r * QLine<BITS>::row +
                                  (long long)j0 * qrow, bytes, bar, policy);
  }
  __syncwarp();   // lane 0 branched off: reconverge before the next warp-wide instruction
  const int nj = (r + (1 << lgc) - 1) >> lgc;
  if (++p.jc == nj) {
    p.jc = 0;
    if (++p.phase == 2) {
      p.phase = 0;
      p.k += NW;
      if (p.k < total) p.item = next_rr_split<NW>(sm, p.item, p.k, n_long);
    }
  }
  return true;
}

__device__ __forceinline__ uint4 ld_shared_v4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t ld_shared_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(v) : "r"(a));
  return v;
}
// Codes -> fp16 pairs. A code c becomes the fp16 number 1024 + c (0x6400 | c) or, four bits higher, 64 + c
// (0x5400 | c << 4), both exact; the base is subtracted exactly and lo + c * step is one fused multiply-add.
__device__ __forceinline__ uint32_t code_pair(uint32_t t, uint32_t base, uint32_t lo2, uint32_t st2) {
  const __half2 code = __hsub2(*reinterpret_cast<const __half2*>(&t), *reinterpret_cast<const __half2*>(&base));
  const __half2 x = __hfma2(code, *reinterpret_cast<const __half2*>(&st2), *reinterpret_cast<const __half2*>(&lo2));
  return *reinterpret_cast<const uint32_t*>(&x);
}
// u: four 4-bit codes in the low half, four in the high half. o[i] = (code i of the low, code i of the high half).
__device__ __forceinline__ void expand4(uint32_t u, uint32_t lo2, uint32_t st2, uint32_t* o) {
  const uint32_t v = u >> 8;
  o[0] = code_pair((u & 0x000F000Fu) | 0x64006400u, 0x64006400u, lo2, st2);
  o[1] = code_pair((u & 0x00F000F0u) | 0x54005400u, 0x54005400u, lo2, st2);
  o[2] = code_pair((v & 0x000F000Fu) | 0x64006400u, 0x64006400u, lo2, st2);
  o[3] = code_pair((v & 0x00F000F0u) | 0x54005400u, 0x54005400u, lo2, st2);
}
// a, b: four 8-bit codes each. o[i] = (code i of a, code i of b).
__device__ __forceinline__ void expand8(uint32_t a, uint32_t b, uint32_t lo2, uint32_t st2, uint32_t* o) {
  const uint32_t u = __byte_perm(a, b, 0x5140), v = __byte_perm(a, b, 0x7362);
  o[0] = code_pair(__byte_perm(u, 0x64646464u, 0x4140), 0x64006400u, lo2, st2);
  o[1] = code_pair(__byte_perm(u, 0x64646464u, 0x4342), 0x64006400u, lo2, st2);
  o[2] = code_pair(__byte_perm(v, 0x64646464u, 0x4140), 0x64006400u, lo2, st2);
  o[3] = code_pair(__byte_perm(v, 0x64646464u, 0x4342), 0x64006400u, lo2, st2);
}
// 16 slots of two streams of codes -> o[x] = (slot x of a, slot x of b); a, b: 16 codes each (BITS / 2 words).
template <int BITS>
__device__ __forceinline__ void expand16(const uint32_t* a, const uint32_t* b, uint32_t lo2, uint32_t st2, uint32_t* o) {
#pragma unroll
  for (int h = 0; h < BITS / 2; ++h) {
    if (BITS == 4) {
      expand4(__byte_perm(a[h], b[h], 0x5410), lo2, st2, o + 8 * h);
      expand4(__byte_perm(a[h], b[h], 0x7632), lo2, st2, o + 8 * h + 4);
    } else {
      expand8(a[h], b[h], lo2, st2, o + 4 * h);
    }
  }
}
// 16 codes of one row at shared address x
template <int BITS>
__device__ __forceinline__ void ld_codes16(uint32_t x, uint32_t* w) {
  if (BITS == 4) {
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];\n" : "=r"(w[0]), "=r"(w[1]) : "r"(x));
  } else {
    const uint4 v = ld_shared_v4(x);
    w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
  }
}
// The row of a 16-row tile of V that lane group g8 takes (and 8 rows on): at 4 bits the even groups rows 0 .. 3
// and the odd ones rows 4 .. 7, so that the two rows of a quarter warp's 16-byte loads are 4 x 80 bytes apart.
template <int BITS>
__device__ __forceinline__ int v_row(int g8) { return BITS == 4 ? (g8 >> 1) + 4 * (g8 & 1) : g8; }

// The A fragments of one 16-row step of K against a tile's 128 slots: m16 x k16, m = slots, k = rows. Row g8 of
// tile mt is slot 16 g8 + 2 mt, row g8 + 8 the slot after it, so a lane's 16 slots are one run of codes in each
// of its four rows. `row`: the lane's first row (2 c of the step), pq: its group's (lo, step) in that row;
// left: rows of the item from that row on. The others are whatever the stage held: with (0, 0) for their (lo, step)
// they are zeros, since a code is a finite number whatever its bits are.
template <int BITS>
__device__ __forceinline__ void k_frags(uint32_t row, uint32_t qrow, uint32_t codes, uint32_t pq, int left,
                                        uint32_t (&a)[ISL / 16][4]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {   // rows 2c, 2c + 1; then 8 rows on
    const uint32_t r0 = row + 8 * h * qrow, r1 = r0 + qrow;
    uint32_t w0[BITS / 2], w1[BITS / 2], o[16];
    ld_codes16<BITS>(r0 + codes, w0);
    ld_codes16<BITS>(r1 + codes, w1);
    uint32_t p0 = ld_shared_u32(r0 + pq), p1 = ld_shared_u32(r1 + pq);
    if (8 * h >= left) p0 = 0u;
    if (8 * h + 1 >= left) p1 = 0u;
    expand16<BITS>(w0, w1, __byte_perm(p0, p1, 0x5410), __byte_perm(p0, p1, 0x7632), o);
#pragma unroll
    for (int mt = 0; mt < ISL / 16; ++mt) { a[mt][2 * h] = o[2 * mt]; a[mt][2 * h + 1] = o[2 * mt + 1]; }
  }
}

// One row's 32 slots of group c: o[x] = (slot 32 c + x, slot 32 c + 16 + x), as the weights' fragments pair them.
// !on (a row past the rank, a group past the tile): zeros. The weights of slots past the tile are 0 and their codes,
// of whatever the row holds there, stay within the range of the group's (lo, step).
template <int BITS>
__device__ __forceinline__ void v_row32(uint32_t row, uint32_t pbase, int c, bool on, uint32_t (&o)[16]) {
  uint32_t w0[BITS / 2], w1[BITS / 2];
  const uint4 x = ld_shared_v4(row + 4 * BITS * c);
  if (BITS == 4) {
    w0[0] = x.x; w0[1] = x.y; w1[0] = x.z; w1[1] = x.w;
  } else {
    const uint4 y = ld_shared_v4(row + 4 * BITS * c + 16);
    w0[0] = x.x; w0[1] = x.y; w0[BITS / 2 - 2] = x.z; w0[BITS / 2 - 1] = x.w;
    w1[0] = y.x; w1[1] = y.y; w1[BITS / 2 - 2] = y.z; w1[BITS / 2 - 1] = y.w;
  }
  uint32_t p = ld_shared_u32(row + pbase + 4 * c);
  if (!on) p = 0u;
  expand16<BITS>(w0, w1, __byte_perm(p, p, 0x1010), __byte_perm(p, p, 0x3232), o);
}

// Short tiles (at most 32 slots, one group): row g8 of tile mt of two is slot 4 g8 + 2 mt, row g8 + 8 the one
// after it; k pairs of the weights are slots 8 c + x and 8 c + 4 + x.
template <int BITS>
__device__ __forceinline__ uint32_t ld_codes4(uint32_t x) {
  if (BITS == 8) return ld_shared_u32(x);
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];\n" : "=h"(v) : "r"(x));
  return v;
}
template <int BITS>
__device__ __forceinline__ void k_frags_short(uint32_t row, uint32_t qrow, uint32_t codes, uint32_t pbase, int left,
                                              uint32_t (&a)[2][4]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t r0 = row + 8 * h * qrow, r1 = r0 + qrow;
    const uint32_t w0 = ld_codes4<BITS>(r0 + codes), w1 = ld_codes4<BITS>(r1 + codes);
    uint32_t p0 = ld_shared_u32(r0 + pbase), p1 = ld_shared_u32(r1 + pbase);
    if (8 * h >= left) p0 = 0u;
    if (8 * h + 1 >= left) p1 = 0u;
    const uint32_t lo2 = __byte_perm(p0, p1, 0x5410), st2 = __byte_perm(p0, p1, 0x7632);
    uint32_t o[4];
    if (BITS == 4) expand4(__byte_perm(w0, w1, 0x5410), lo2, st2, o);
    else expand8(w0, w1, lo2, st2, o);
    a[0][2 * h] = o[0]; a[0][2 * h + 1] = o[1];
    a[1][2 * h] = o[2]; a[1][2 * h + 1] = o[3];
  }
}
template <int BITS>
__device__ __forceinline__ void v_row_short(uint32_t row, uint32_t pbase, int c, bool on, uint32_t (&o)[4]) {
  uint32_t p = ld_shared_u32(row + pbase);
  if (!on) p = 0u;
  const uint32_t lo2 = __byte_perm(p, p, 0x1010), st2 = __byte_perm(p, p, 0x3232);
  if (BITS == 4) {
    expand4(ld_shared_u32(row + 4 * c), lo2, st2, o);
  } else {
    uint32_t w[4];
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];\n" : "=r"(w[0]), "=r"(w[1]) : "r"(row + 8 * c));
    expand8(w[0], w[1], lo2, st2, o);
  }
}

template <int BITS>
__global__ void __launch_bounds__(NW * 32, 1)
decode_q_kernel(const uint8_t* __restrict__ qdata, const int32_t* __restrict__ bucket_count,
                  const int64_t* __restrict__ bucket_base, const __nv_bfloat16* __restrict__ basis_k,
                  const __nv_bfloat16* __restrict__ basis_v, const __nv_bfloat16* __restrict__ qin,
                  const __nv_bfloat16* __restrict__ tail_k, const __nv_bfloat16* __restrict__ tail_v,
                  int n_tail, __nv_bfloat16* __restrict__ out, float* __restrict__ part,
                  DecodeHeader* __restrict__ hdr, int32_t* __restrict__ dev_status, Shape s,
                  int layer, int64_t qcap) {
  constexpr long long kSegCostQ = QLine<BITS>::seg_cost, kSegEndQ = QLine<BITS>::seg_end;
  extern __shared__ __align__(256) unsigned char smem[];
  constexpr int STQ = QLine<BITS>::stage;
  constexpr int SQ = QLine<BITS>::stages;
  unsigned char* ring = smem;   // NW * SQ * STQ of quantized chunks
  constexpr int kRing = NW * SQ * STQ;
  SegSmem& sm = *reinterpret_cast<SegSmem*>(smem + kRing);
  // the merge and combine buffers alias the ring (idle while a segment is merged)
  static_assert(kRing % 256 == 0 && sizeof(Merge) <= kRing && sizeof(CombSmem) <= kRing, "they fit in the ring");
  Merge& mg = *reinterpret_cast<Merge*>(smem);
  __shared__ long long segW[64];                                  // per-sequence stream length
  __shared__ long long segP[65];                                  // start of sequence b on the cost line
  __shared__ long long cuts[kMaxCtas + 1];                        // start of CTA c's range
  __shared__ int n_empty;                                         // sequences with no coded tokens
  __shared__ int last_cta;                                        // this CTA closes the segment
  __shared__ uint32_t parity;                                     // counter set of this call
  __shared__ uint64_t bar_all[NW * SQ];                           // one full-barrier per ring stage
  __shared__ uint64_t bar_comb;                                   // U_V copy of a combine

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g8 = lane >> 2, c = lane & 3;
  const int C = gridDim.x, cta = blockIdx.x;
  const uint64_t policy = l2_evict_first_policy();   // coefficient chunks are read once

  // the next grid in the stream may be scheduled now: it only starts on SMs this grid has left,
  // and waits (griddepcontrol.wait) for this grid to finish before it reads anything
  pdl_trigger();
  // self-contained setup first (it may overlap the tail of the preceding grid)
  if (tid < NW * SQ) mbar_init(&bar_all[tid], 1);
  if (tid == NW * SQ) mbar_init(&bar_comb, 1);
  fence_mbar_init();
  fence_proxy_async_smem();
  pdl_wait();   // everything below reads data written by earlier grids
  if (tid == 0) parity = (uint32_t)(*reinterpret_cast<volatile unsigned long long*>(&hdr->calls) & 1ull);
  // stream length of every sequence of this layer (same for every head); poisoned tables -> 0
  for (int b = tid; b < s.B; b += blockDim.x) {
    const long long w = bucket_base[((long long)b * s.L + layer) * (kMaxR + 2) + kMaxR + 1];
    segW[b] = (w >= 0 && w <= qcap) ? w : 0;
  }
  __syncthreads();
  {   // the other set: used by the previous call (finished), counted on by the next one
    uint32_t* other = hdr->arrived[parity ^ 1u];
    for (int i = cta * (int)blockDim.x + tid; i < kDecodeMaxSegs; i += C * (int)blockDim.x) other[i] = 0u;
    if (cta == 0 && tid == 0) hdr->exits[parity ^ 1u] = 0u;
  }
  uint32_t* arrived = hdr->arrived[parity];
  uint32_t n_issued = 0;   // chunks this warp has consumed (== index of its next chunk)
  int n_pending = 0;       // chunks issued but not yet consumed
  bool timed_out = false;  // this thread saw a bounded wait give up
  // CTA-uniform: some wait of this CTA gave up, so bulk copies may still be landing in the ring.
  // From then on nothing writes the ring (merge and combine buffers alias it) and nothing streams;
  // the CTA still writes an empty partial and arrives on every segment it covers, so the counts of
  // the other CTAs stay consistent.
  bool dead = false;
  uint32_t n_comb = 0;     // combines done by this CTA (phase of bar_comb)
  // Cost line: sequence b holds G segments of kSegCost + W_b + kSegEnd elements each (W_b > 0): the
  // set-up allowance, the coefficients, the end allowance. segP = exclusive prefix over sequences (B <= 64: two per lane).
  if (warp == 0) {
    __syncwarp();   // lanes left the loads above apart: reconverge before the shuffles
    const int e0 = 2 * lane, e1 = 2 * lane + 1;
    const long long v0 = (e0 < s.B && segW[e0]) ? (segW[e0] + kSegCostQ + kSegEndQ) * s.G : 0;
    const long long v1 = (e1 < s.B && segW[e1]) ? (segW[e1] + kSegCostQ + kSegEndQ) * s.G : 0;
    long long inc = v0 + v1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    segP[e0] = inc - v0 - v1;
    segP[e1] = inc - v1;
    if (lane == 31) segP[64] = inc;
    const unsigned m0 = __ballot_sync(0xffffffffu, e0 < s.B && segW[e0] == 0);
    const unsigned m1 = __ballot_sync(0xffffffffu, e1 < s.B && segW[e1] == 0);
    if (lane == 0) n_empty = __popc(m0) + __popc(m1);
  }
  __syncthreads();
  const long long T = segP[64];
  for (int c2 = tid; c2 <= C; c2 += blockDim.x) cuts[c2] = cut_at(T, c2, C);
  __syncthreads();
  const long long lo_g = cuts[cta], hi_g = cuts[cta + 1];

  // first segment of this CTA: the sequence whose span holds lo_g, then the head within it
  int b = 0, g = 0;
  {
    int lo_b = 0, hi_b = s.B;
    while (lo_b < hi_b) {
      const int mid = (lo_b + hi_b) >> 1;
      if (segP[mid + 1] > lo_g) hi_b = mid; else lo_b = mid + 1;
    }
    b = lo_b;
    if (b < s.B) {   // g = floor(x / w), estimated in fp32 and corrected
      const long long x = lo_g - segP[b], w = segW[b] + kSegCostQ + kSegEndQ;
      g = (int)((float)x / (float)w);
      while (g > 0 && (long long)g * w > x) --g;
      while ((long long)(g + 1) * w <= x) ++g;
    }
  }
  auto seg_start = [&](int bb, int gg) { return segP[bb] + gg * (segW[bb] + kSegCostQ + kSegEndQ) + kSegCostQ; };
  if (b < s.B && seg_start(b, g) + segW[b] <= lo_g) {   // the range starts in a segment's end allowance
    if (++g == s.G) { ++b; g = 0; }
    while (b < s.B && segW[b] == 0) ++b;
  }
  bool more = b < s.B && seg_start(b, g) < hi_g;
  while (more) {
    {
      const long long W = segW[b];
      const long long P = seg_start(b, g);   // first coefficient of segment (b, g) on the cost line
      const long long lo = max(lo_g, P) - P, hi = min(hi_g, P + W) - P;
      const long long bl = (long long)b * s.L + layer;
      RotRegs rr;   // this segment's U_K tile and queries, in flight with the table loads below
      rot_load(rr, basis_k + ((long long)layer * s.G + g) * kHeadDim * kHeadDim,
               qin + ((long long)b * s.H + (long long)g * s.grp) * kHeadDim, s.grp, warp, lane);
      // U_V of this head, for whichever CTA merges the segment: into L2 while it streams
      if (tid == 0) bulk_prefetch_l2(basis_v + ((long long)layer * s.G + g) * kHeadDim * kHeadDim, kHeadDim * kHeadDim * 2);
      __syncthreads();
      for (int r = tid; r <= kMaxR + 1; r += blockDim.x) {
        if (r <= kMaxR) sm.cnt[r] = bucket_count[bl * (kMaxR + 1) + r];
        sm.base[r] = bucket_base[bl * (kMaxR + 2) + r];
      }
      __syncthreads();
      for (int r = tid; r <= kMaxR; r += blockDim.x) {
        long long i0 = 0, i1 = 0;
        if (r >= s.r_min && r <= s.r_max) bucket_range_q<BITS>(sm, r, lo, hi, i0, i1);
        sm.it_lo[r] = (int)i0;
        sm.it_pref[r + 1] = split_count(i0, i1, sm.cnt[r]);   // counts first, prefixed below
      }
      __syncthreads();
      if (warp == 0) {   // inclusive scan of it_pref[1 .. 129], 5 entries per lane
        __syncwarp();
        constexpr int kPer = (kMaxR + 1 + 31) / 32;
        uint32_t v[kPer], acc = 0;
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
          const int r = lane * kPer + e;
          acc += r <= kMaxR ? sm.it_pref[r + 1] : 0u;
          v[e] = acc;
        }
        uint32_t excl = acc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, excl, o);
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
      // start this warp's loads first: they do not depend on the rotated queries
      const uint8_t* cK = qdata + ((bl * s.G + g) * 2) * qcap;
      const uint8_t* cV = cK + qcap;
      const uint32_t ring_w = smem_addr(ring) + warp * SQ * STQ;
      uint64_t* bars = &bar_all[warp * SQ];

      float Mx[2] = {-INFINITY, -INFINITY}, Ls[2] = {0.f, 0.f};
      float oacc[kHeadDim / 16][4];
#pragma unroll
      for (int t = 0; t < kHeadDim / 16; ++t) oacc[t][0] = oacc[t][1] = oacc[t][2] = oacc[t][3] = 0.f;

      // long items first, then the short ones: every warp takes both in turn
      const int n_long = dead ? 0 : (int)(sm.it_pref[kMaxR + 1] & kLongMask);
      const int total = dead ? 0 : n_long + (int)(sm.it_pref[kMaxR + 1] >> 24);
      Prod pr;
      pr.k = warp; pr.phase = 0; pr.jc = 0;
      if (pr.k < total) pr.item = item_at_split(sm, pr.k, n_long);
      int cons_k = pr.k;
      Item cons = pr.item;
#pragma unroll
      for (int i = 0; i < SQ; ++i)   // every stage of the ring in flight
        if (issue_chunk_q<BITS>(pr, sm, cK, cV, ring_w + ((n_issued + i) % SQ) * STQ,
                        &bars[(n_issued + i) % SQ], total, n_long, lane, policy)) ++n_pending;
      int c0, c1;   // the CTAs that share this segment (their partials are merged by the last one)
      seg_cta_range([&](int i) { return cuts[i]; }, T, C, P, W, c0, c1);
      __syncwarp();
      if (warp < kHeadDim / 16) rot_compute(sm, rr, s.grp, warp, lane);
      __syncthreads();
      build_qfrag_f16(sm, tid);
      __syncthreads();

      // chunk k of this warp (counted over the whole kernel) lives in stage k % SQ, phase (k / SQ) & 1

      auto wait_chunk = [&]() -> bool {
        const uint32_t k = n_issued;
        if (!mbar_wait_bounded(&bars[k % SQ], (k / SQ) & 1u, kWaitTries)) { timed_out = true; return false; }
        return true;
      };
      auto next_chunk = [&]() {
        // the consumed stage is free again: refill it with the chunk SQ ahead, so that all the
        // other stages stay in flight while the warp computes
        ++n_issued;
        --n_pending;
        if (issue_chunk_q<BITS>(pr, sm, cK, cV, ring_w + ((n_issued + SQ - 1) % SQ) * STQ,
                        &bars[(n_issued + SQ - 1) % SQ], total, n_long, lane, policy)) ++n_pending;
      };

      while (cons_k < n_long && !timed_out) {
        const int r = cons.r;
        const long long n_real = sm.cnt[r] - (long long)cons.it * ISL;   // real slots of this item
        const int tl = (int)min((long long)ISL, pad8(sm.cnt[r]) - (long long)cons.it * ISL);
        const uint32_t qrow = qrow_bytes(tl, BITS), pbase = tl * BITS / 8;
        const int lgc = chunk_lg_q(tl, BITS);           // same chunking as the producer
        const int nj = (r + (1 << lgc) - 1) >> lgc;
        float sc[ISL / 16][4];
#pragma unroll
        for (int t = 0; t < ISL / 16; ++t) sc[t][0] = sc[t][1] = sc[t][2] = sc[t][3] = 0.f;

        // ---- K chunks: scores (rows >= r as zeros)
        for (int jc = 0; jc < nj; ++jc) {
          if (!wait_chunk()) break;
          const int j0 = jc << lgc, j1 = min(r, j0 + (1 << lgc));
          const uint32_t row0 = ring_w + (n_issued % SQ) * STQ + 2 * c * qrow;
          for (int j16 = j0; j16 < j1; j16 += 16) {
            const uint4 qf = *reinterpret_cast<const uint4*>(&sm.qfrag[j16 >> 4][lane][0]);
            uint32_t a[ISL / 16][4];
            k_frags<BITS>(row0 + (j16 - j0) * qrow, qrow, 2 * BITS * g8, pbase + 4 * (g8 >> 1), r - j16 - 2 * c, a);
#pragma unroll
            for (int mt = 0; mt < ISL / 16; ++mt) mma_f16_16816(sc[mt], a[mt], qf.x, qf.y);
#pragma unroll
            for (int mt = 0; mt < ISL / 16; ++mt) mma_f16_16816(sc[mt], a[mt], qf.z, qf.w);
          }
          __syncwarp();   // every lane has read the stage before it is refilled
          next_chunk();
        }
        if (timed_out) break;

        // ---- online softmax over the item's slots (heads 2c, 2c+1 per lane)
        float mloc[2] = {-INFINITY, -INFINITY};
        const bool full_item = n_real >= ISL;           // warp-uniform: no slot to mask
#pragma unroll
        for (int mt = 0; mt < ISL / 16; ++mt) {
          if (!full_item) {
            const int s0 = 16 * g8 + 2 * mt;
            if (s0 >= n_real) { sc[mt][0] = sc[mt][1] = -INFINITY; }
            if (s0 + 1 >= n_real) { sc[mt][2] = sc[mt][3] = -INFINITY; }
          }
          mloc[0] = fmaxf(mloc[0], fmaxf(sc[mt][0], sc[mt][2]));
          mloc[1] = fmaxf(mloc[1], fmaxf(sc[mt][1], sc[mt][3]));
        }
        // The reference max only moves when some score exceeds it by more than kSlack (log2
        // units): weights stay <= 2^kSlack, exact after the final normalisation, and the common
        // case costs one warp vote instead of a shuffle reduction and a rescale.
        float corr[2] = {1.f, 1.f};
        if (!__all_sync(0xffffffffu, mloc[0] <= Mx[0] + kSlack && mloc[1] <= Mx[1] + kSlack)) {
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) {
            mloc[0] = fmaxf(mloc[0], __shfl_xor_sync(0xffffffffu, mloc[0], o));
            mloc[1] = fmaxf(mloc[1], __shfl_xor_sync(0xffffffffu, mloc[1], o));
          }
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float nm = fmaxf(Mx[e], mloc[e]);
            corr[e] = fast_exp2(Mx[e] - nm);
            Mx[e] = nm;
          }
#pragma unroll
          for (int t = 0; t < kHeadDim / 16; ++t) {
            oacc[t][0] *= corr[0]; oacc[t][1] *= corr[1];
            oacc[t][2] *= corr[0]; oacc[t][3] *= corr[1];
          }
        }
        float lsum[2] = {0.f, 0.f};
        const float Mr[2] = {Mx[0] - kPShift, Mx[1] - kPShift};   // weights scaled by 2^kPShift
        uint32_t pb[ISL / 16][2];   // per slot tile: b0, b1 of P^T
#pragma unroll
        for (int mt = 0; mt < ISL / 16; ++mt) {
          const float p0 = fast_exp2(sc[mt][0] - Mr[0]), p1 = fast_exp2(sc[mt][1] - Mr[1]);
          const float p2 = fast_exp2(sc[mt][2] - Mr[0]), p3 = fast_exp2(sc[mt][3] - Mr[1]);
          lsum[0] += p0 + p2;
          lsum[1] += p1 + p3;
          pb[mt][0] = movmatrix_trans(pack_f16(p0, p1));
          pb[mt][1] = movmatrix_trans(pack_f16(p2, p3));
        }
        Ls[0] = Ls[0] * corr[0] + lsum[0];
        Ls[1] = Ls[1] * corr[1] + lsum[1];

        // ---- V chunks: weighted coefficient rows (rows >= r as zeros)
        {
          int left = 0;             // rows of the current chunk not used yet
          uint32_t row = 0;         // this lane's row of the next 16-row tile
#pragma unroll
          for (int jp = 0; jp < kHeadDim / 32; ++jp) {   // two 16-row tiles of o~ (chunks are 32 rows or more)
            if (jp * 32 >= r) break;                     // warp-uniform
            if (left == 0) {                             // the tiles start a chunk
              if (!wait_chunk()) break;
              row = ring_w + (n_issued % SQ) * STQ + v_row<BITS>(g8) * qrow;
              left = 1 << lgc;
            }
#pragma unroll
            for (int jt = 2 * jp; jt < 2 * jp + 2; ++jt) {
              if (jt * 16 >= r) break;
              uint32_t o0[16], o1[16];
              const int left_r = r - jt * 16 - v_row<BITS>(g8);
              v_row32<BITS>(row, pbase, c, left_r > 0 && 32 * c < tl, o0);
              v_row32<BITS>(row + 8 * qrow, pbase, c, left_r > 8 && 32 * c < tl, o1);
              row += 16 * qrow;
#pragma unroll
              for (int kt = 0; kt < ISL / 16; ++kt) {
                const uint32_t a[4] = {o0[2 * kt], o1[2 * kt], o0[2 * kt + 1], o1[2 * kt + 1]};
                mma_f16_16816(oacc[jt], a, pb[kt][0], pb[kt][1]);
              }
            }
            left -= 32;
            if (left == 0 || jp * 32 + 32 >= r) {        // the chunk's last rows
              __syncwarp();   // every lane has read the stage before it is refilled
              next_chunk();
              left = 0;
            }
          }
        }
        cons_k += NW;
        if (cons_k < total) cons = next_rr_split<NW>(sm, cons, cons_k, n_long);
      }
      // Short items (at most kShort slots): the same steps on two 16-slot tiles instead of eight, in a loop of
      // their own as in decode_mma.cu (one chunk each of K and V rows, at 8 bits two past 64 rows). Before / with
      // it, us per call: 1 sequence, 8 bits, wide ranks 57 / 39; 4 sequences, 4 bits, spread ranks 79 / 67.
      while (cons_k < total && !timed_out) {
        const int r = cons.r;
        const int n_real = sm.cnt[r] - cons.it * ISL, tl = (n_real + 7) & ~7;
        const uint32_t qrow = qrow_bytes(tl, BITS), pbase = tl * BITS / 8;
        const int lgc = chunk_lg_q(tl, BITS);
        float sh[2][4] = {}, sl[2][4] = {};
        for (int j0 = 0; j0 < r; j0 += 1 << lgc) {
          if (!wait_chunk()) break;
          const int j1 = min(r, j0 + (1 << lgc));
          const uint32_t row0 = ring_w + (n_issued % SQ) * STQ + 2 * c * qrow;
          for (int j16 = j0; j16 < j1; j16 += 16) {
            const uint4 qf = *reinterpret_cast<const uint4*>(&sm.qfrag[j16 >> 4][lane][0]);
            uint32_t a[2][4];
            k_frags_short<BITS>(row0 + (j16 - j0) * qrow, qrow, BITS / 2 * g8, pbase, r - j16 - 2 * c, a);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
              mma_f16_16816(sh[mt], a[mt], qf.x, qf.y);
              mma_f16_16816(sl[mt], a[mt], qf.z, qf.w);
            }
          }
          __syncwarp();   // every lane has read the stage before it is refilled
          next_chunk();
        }
        if (timed_out) break;
        float mloc[2] = {-INFINITY, -INFINITY};
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
          const int s0 = 4 * g8 + 2 * mt;
#pragma unroll
          for (int e = 0; e < 4; ++e) sh[mt][e] = s0 + (e >> 1) < n_real ? sh[mt][e] + sl[mt][e] : -INFINITY;
          mloc[0] = fmaxf(mloc[0], fmaxf(sh[mt][0], sh[mt][2]));
          mloc[1] = fmaxf(mloc[1], fmaxf(sh[mt][1], sh[mt][3]));
        }
        if (!__all_sync(0xffffffffu, mloc[0] <= Mx[0] + kSlack && mloc[1] <= Mx[1] + kSlack)) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) mloc[e] = fmaxf(mloc[e], __shfl_xor_sync(0xffffffffu, mloc[e], o));
            const float nm = fmaxf(Mx[e], mloc[e]);
            const float corr = fast_exp2(Mx[e] - nm);
            Mx[e] = nm;
            Ls[e] *= corr;
#pragma unroll
            for (int t = 0; t < kHeadDim / 16; ++t) { oacc[t][e] *= corr; oacc[t][e + 2] *= corr; }
          }
        }
        const float Mr[2] = {Mx[0] - kPShift, Mx[1] - kPShift};   // weights scaled by 2^kPShift
        uint32_t pb[2][2];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
          const float p0 = fast_exp2(sh[mt][0] - Mr[0]), p1 = fast_exp2(sh[mt][1] - Mr[1]);
          const float p2 = fast_exp2(sh[mt][2] - Mr[0]), p3 = fast_exp2(sh[mt][3] - Mr[1]);
          Ls[0] += p0 + p2;
          Ls[1] += p1 + p3;
          pb[mt][0] = movmatrix_trans(pack_f16(p0, p1));
          pb[mt][1] = movmatrix_trans(pack_f16(p2, p3));
        }
        uint32_t row = 0;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {                 // 64 rows: one chunk of 8-bit rows, half a chunk of 4-bit rows
          if (hf * 64 >= r) break;                       // warp-uniform
          if (hf == 0 || lgc == 6) {
            if (!wait_chunk()) break;
            row = ring_w + (n_issued % SQ) * STQ + v_row<BITS>(g8) * qrow;
          }
#pragma unroll
          for (int jt = 4 * hf; jt < 4 * hf + 4; ++jt) {
            if (jt * 16 >= r) break;
            uint32_t o0[4], o1[4];
            const int left_r = r - jt * 16 - v_row<BITS>(g8);
            v_row_short<BITS>(row, pbase, c, left_r > 0, o0);
            v_row_short<BITS>(row + 8 * qrow, pbase, c, left_r > 8, o1);
            row += 16 * qrow;
#pragma unroll
            for (int kt = 0; kt < 2; ++kt) {
              const uint32_t a[4] = {o0[2 * kt], o1[2 * kt], o0[2 * kt + 1], o1[2 * kt + 1]};
              mma_f16_16816(oacc[jt], a, pb[kt][0], pb[kt][1]);
            }
          }
          if (lgc == 6 || hf == 1 || r <= 64) {          // the chunk's last rows
            __syncwarp();   // every lane has read the stage before it is refilled
            next_chunk();
          }
        }
        cons_k += NW;
        if (cons_k < total) cons = next_rr_split<NW>(sm, cons, cons_k, n_long);
      }
      // drain: never leave bulk copies in flight into this ring (a copy whose wait gave up stays
      // counted in n_pending and is waited for once more before the CTA exits)
      while (n_pending > 0 && !timed_out) {
        if (!mbar_wait_bounded(&bars[n_issued % SQ], (n_issued / SQ) & 1u, kWaitTries)) {
          timed_out = true;
          break;
        }
        ++n_issued;
        --n_pending;
      }

      // ---- merge the warps of this CTA for this segment
      __syncwarp();
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) Ls[e] += __shfl_xor_sync(0xffffffffu, Ls[e], o);
      dead = __syncthreads_or(dead || timed_out);   // every warp has finished this segment
      if (!dead && g8 == 0) {
        mg.M[warp][2 * c] = Mx[0] - kPShift; mg.M[warp][2 * c + 1] = Mx[1] - kPShift;
        mg.L[warp][2 * c] = Ls[0]; mg.L[warp][2 * c + 1] = Ls[1];
      }
      if (!dead) {
#pragma unroll
        for (int t = 0; t < kHeadDim / 16; ++t) {
          mg.acc[warp][2 * c][t * 16 + v_row<BITS>(g8)] = oacc[t][0];
          mg.acc[warp][2 * c + 1][t * 16 + v_row<BITS>(g8)] = oacc[t][1];
          mg.acc[warp][2 * c][t * 16 + v_row<BITS>(g8) + 8] = oacc[t][2];
          mg.acc[warp][2 * c + 1][t * 16 + v_row<BITS>(g8) + 8] = oacc[t][3];
        }
      }
      if (!dead && tid < kHeadsPad) {
        const int h = tid;
        float mx = -INFINITY, l = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) mx = fmaxf(mx, mg.M[w][h]);
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          const float f = mx == -INFINITY ? 0.f : fast_exp2(mg.M[w][h] - mx);
          mg.F[w][h] = f;
          l = fmaf(mg.L[w][h], f, l);
        }
        mg.mx[h] = mx;
        mg.l[h] = l;
      }
      __syncthreads();
      // partial slot of this (segment, CTA): index cta + segment number (unique: a CTA after this
      // one only meets segments after this one)
      const long long seg = (long long)b * s.G + g;
      float* pout = part + (cta + seg) * (long long)kHeadsPad * kPartStride;
      for (int i = tid; i < kHeadsPad * kHeadDim; i += blockDim.x) {
        const int h = i / kHeadDim, j = i % kHeadDim;
        float o = 0.f;
        if (!dead) {
#pragma unroll
          for (int w = 0; w < NW; ++w) o = fmaf(mg.acc[w][h][j], mg.F[w][h], o);
        }
        pout[h * kPartStride + j] = o;
        if (j == 0) {   // an abandoned CTA contributes an empty partial
          pout[h * kPartStride + kHeadDim] = dead ? -INFINITY : mg.mx[h];
          pout[h * kPartStride + kHeadDim + 1] = dead ? 0.f : mg.l[h];
        }
      }
      // the last CTA to finish this segment merges every partial of it
      __syncthreads();
      if (tid == 0) {
        // release: this CTA's partial (ordered before by the barrier) is visible to whoever sees
        // the count; acquire: the last arrival then sees every other CTA's partial
        const uint32_t n = (uint32_t)(c1 - c0 + 1);   // CTAs that share this segment
        const uint32_t done = atom_add_acq_rel_gpu(&arrived[seg], 1u);
        last_cta = done == n - 1u;
        if (done >= n) raise_status(dev_status, VARRATE_ERR_CORRUPT);   // counts left by an earlier call
      }
      __syncthreads();
      if (last_cta && !dead) {
        if (!combine_segment(*reinterpret_cast<CombSmem*>(ring), &bar_comb, n_comb & 1u, part, c0, c1, seg,
                             qin + ((long long)b * s.H + (long long)g * s.grp) * kHeadDim,
                             basis_v + ((long long)layer * s.G + g) * kHeadDim * kHeadDim,
                             n_tail ? tail_k + ((long long)b * s.G + g) * n_tail * kHeadDim : nullptr,
                             n_tail ? tail_v + ((long long)b * s.G + g) * n_tail * kHeadDim : nullptr, n_tail,
                             out + ((long long)b * s.H + (long long)g * s.grp) * kHeadDim, s.grp, tid)) {
          timed_out = true;
          dead = true;   // CTA-uniform: the U_V copy of the combine may still be landing
        }
        ++n_comb;
      }
      __syncthreads();
    }
    if (++g == s.G) { ++b; g = 0; }
    while (b < s.B && segW[b] == 0) ++b;
    more = b < s.B && seg_start(b, g) < hi_g;
    if (more && !dead) {
      fence_proxy_async_smem();   // the merge and combine wrote the ring: before the next copies
      __syncthreads();
    }
  }
  // segments with an empty coded stream (tail only): one CTA each, no partials
  if (n_empty && !dead)
  for (int b = 0; b < s.B; ++b)
    for (int g = 0; g < s.G; ++g) {
      const long long seg = (long long)b * s.G + g;
      if (segW[b] != 0 || seg % C != cta || dead) continue;   // CTA-uniform
      __syncthreads();
      if (!combine_segment(*reinterpret_cast<CombSmem*>(ring), &bar_comb, n_comb & 1u, part, 0, -1, seg,
                           qin + ((long long)b * s.H + (long long)g * s.grp) * kHeadDim,
                           basis_v + ((long long)layer * s.G + g) * kHeadDim * kHeadDim,
                           n_tail ? tail_k + ((long long)b * s.G + g) * n_tail * kHeadDim : nullptr,
                           n_tail ? tail_v + ((long long)b * s.G + g) * n_tail * kHeadDim : nullptr, n_tail,
                           out + ((long long)b * s.H + (long long)g * s.grp) * kHeadDim, s.grp, tid)) {
        timed_out = true;
        dead = true;
      }
      ++n_comb;
    }
  if (dead) {
    // last bounded waits for copies that may still be landing in this CTA's shared memory
    for (; n_pending > 0; --n_pending, ++n_issued)
      if (!mbar_wait_bounded(&bar_all[warp * SQ + n_issued % SQ], (n_issued / SQ) & 1u, kWaitTries)) break;
    if (n_comb > 0 && tid == 0) mbar_wait_bounded(&bar_comb, (n_comb - 1) & 1u, kWaitTries);
  }
  if (timed_out && lane == 0) raise_status(dev_status, VARRATE_ERR_TIMEOUT);
  // the CTA that completes a multiple of the grid size of exits advances the call count (a
  // multiple rather than exactly C - 1: the count then stays consistent whatever the set held)
  __syncthreads();
  if (tid == 0 && (atomicAdd(&hdr->exits[parity], 1u) + 1u) % (uint32_t)C == 0u)
    atomicAdd(&hdr->calls, 1ull);
}

}  // namespace

size_t decode_q_smem_bytes(int bits) {
  const int stq = bits == 4 ? QLine<4>::stage : QLine<8>::stage;
  return (size_t)NW * stq * (bits == 4 ? QLine<4>::stages : QLine<8>::stages) + sizeof(SegSmem);
}

bool decode_q_supported(const Shape& s, int bits, int64_t qcap, int n_tail, int num_sms) {
  const long long cost = bits == 4 ? QLine<4>::seg_cost + QLine<4>::seg_end : QLine<8>::seg_cost + QLine<8>::seg_end;
  const unsigned long long line = (unsigned long long)s.B * s.G * ((unsigned long long)qcap + (unsigned long long)cost);
  return s.dtype == VARRATE_BF16 && (bits == 4 || bits == 8) && qcap > 0 && qcap % 16 == 0 && s.B <= 64 &&
         (long long)s.B * s.G <= kDecodeMaxSegs && n_tail <= kMaxTailFused && num_sms >= 1 &&
         num_sms <= kMaxCtas && line <= (1ull << 62) / (unsigned long long)num_sms;
}

int launch_decode_q_fused(const Shape& s, const varrate_qpacked& c, const void* basis_k, const void* basis_v,
                          const void* q, int layer, const void* tail_k, const void* tail_v, int n_tail, void* out,
                          int32_t* dev_status, void* header, float* part, int num_sms, cudaStream_t st) {
  const size_t smem = decode_q_smem_bytes(c.bits);
  auto kern = c.bits == 4 ? decode_q_kernel<4> : decode_q_kernel<8>;
  static std::atomic<int> smem_set[2][64];   // the opt-in is per device and per instantiation
  const int bi = c.bits == 4 ? 0 : 1;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 ||
      smem_set[bi][dev].load(std::memory_order_acquire) == 0) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
      return -1;
    if (dev >= 0 && dev < 64) smem_set[bi][dev].store(1, std::memory_order_release);
  }
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(num_sms);
  lc.blockDim = dim3(NW * 32);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  lc.attrs = pdl;
  lc.numAttrs = 1;
  cudaLaunchKernelEx(&lc, kern, (const uint8_t*)c.data, (const int32_t*)c.bucket_count, (const int64_t*)c.qbase,
                     (const __nv_bfloat16*)basis_k, (const __nv_bfloat16*)basis_v, (const __nv_bfloat16*)q,
                     (const __nv_bfloat16*)tail_k, (const __nv_bfloat16*)tail_v, n_tail, (__nv_bfloat16*)out, part,
                     reinterpret_cast<DecodeHeader*>(header), dev_status, s, layer, (int64_t)c.qcap_bytes);
  return 1;
}

}  // namespace vr
