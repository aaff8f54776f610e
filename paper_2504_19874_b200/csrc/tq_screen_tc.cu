// Screening scan of many-query top-k: cheap bounds of the estimates decide which rows the exact engine has to score.
//
// The exact many-query engine (tq_scan_tc.cu) spends six to eight K-bytes and three accumulator columns per (coordinate, query)
// on fixed-point sums whose last bits matter only for the rows that end up in a top-k list.  Here one fp16 pass
//     acc[vector, query] = sum_j c16[idx_j] q16_j + sum_j (+-gamma16) q16''_j        (one fp32 accumulator, kind::f16)
// gives every estimate within a bound that is known per query and row:
//     |estimate - nu acc| <= nu (1 + gamma) E_q.
// E_q adds up, entry by entry, what rounding the query, the codebook and gamma to fp16 can do (exact differences times the largest
// factor they meet), the truncating additions of the tensor core, and the fixed-point rounding of the exact engine itself: it is
// a worst case, not a likely one.  A row whose upper bound misses a lower bound of the k-th best estimate cannot be among the
// k best; the few that are left (about k + k / 3 of 10^6 rows) are scored again by the exact integers (tscan::rescore), so the
// results are the bits that the exact engine returns for every row.
//
// CTA pair (cta_group::2, M = 256 rows, 128 per CTA; N = 256 queries, or 128), persistent over row tiles, 896 threads per CTA:
//   warp 0        TMA producer of the query operand: per k-block (64 coordinates) the CTA's half of its rows
//   warp 1        MMA issuer (of the leader)
//   warp 2        TMA producer of the packed rows
//   warps 4..11   expansion (thread = row): packed codes -> fp16 by byte permutes over the codebook's bytes -> the stage's A tile; two
//                 sets of four warps take the k-blocks in turn
//   warps 12..27  epilogue (thread = row, a quarter of the queries): one FMA chain per pair of estimates, the hits one by one
// Five stages of 32 KB (A and half of B), two accumulators of 256 columns (all of TMEM), so that a tile is read while the next one's
// MMAs run.  The single-lane roles are chains of dependent instructions at six cycles each, of which the tensor pipe's queue hides only
// a part: with 128 columns the issuer's chain is longer than a k-block's 256 cycles of MMAs.  Hence one barrier for both operands and
// counters instead of divisions in its loop.  One thread issues all MMAs of an accumulator: those of two threads are in order only
// where the threads order them, and handing every k-block's turn over a barrier costs more than the second issuer gains (65 queries,
// 10^6 rows of d = 768 prod b = 4: 659 us, 635 with one issuer; 256 queries 849 and 807; 10^4 queries of d = 200 prod b = 3 alike, 16.5 ms).
// All waits are bounded.
#include <algorithm>
#include <atomic>
#include <cfloat>
#include <cmath>

#include <cuda_fp16.h>

#include "tq_nib_common.cuh"
#include "tq_quantize_tc.h"
#include "tq_screen_tc.h"
#include "tq_tc.cuh"

namespace tq {
namespace screen {

namespace {

using namespace tq::tc;

constexpr int TILE = 128;                   // rows per CTA = TMEM lanes
constexpr int STAGES = 5;                   // ring of k-blocks
// A parity wait also passes when its barrier is two completions behind, so whoever waits for a k-block must have waited for the one
// before on the same barrier.  The two expansion sets take every second k-block, so operands are announced and MMAs complete on rings
// of twice the stages: the set of k-block k has waited for k - RING there.
constexpr int RING = 2 * STAGES;
constexpr int ATILE = TILE * 128, BTILE = kQueries / 2 * 128;   // bytes of a k-block in one CTA: 128 rows, 128 queries x 64 fp16
constexpr int STAGE = ATILE + BTILE;
constexpr int PSTAGES = 3, PTILE = TILE * 64;
constexpr int TMEM_COLS = 512;
constexpr int NEXP0 = 4, NEPI0 = 12;        // first expansion and epilogue warp
constexpr int NEPI = 16;                    // epilogue warps
constexpr int NTHREADS = 32 * (NEPI0 + NEPI);
constexpr int LBUF = 16;                    // candidates per query a CTA collects before it appends them
constexpr size_t kSmemBytes = 1024 + (size_t)STAGES * STAGE + PSTAGES * PTILE + 512 +
                              kQueries * (sizeof(float4) / 2 + sizeof(float) + sizeof(int) + LBUF * sizeof(uint2));
static_assert(kSmemBytes <= 227 * 1024, "shared memory");

// k-blocks of 64 coordinates: those of the centroid term, then those of the sign term; nibble layout: per 64-byte block of the
// combined row [idx row | qjl row] centroids and signs of its first 64 coordinates, then of the others.
struct Geo {
  int bm, d, kba, kbs, nib, nbi, nblk, idx_rb, qjl_rb;
  __host__ __device__ int kblocks() const { return nib ? 4 * nblk : kba + kbs; }
};
__host__ __device__ constexpr int a_group_kb(int bm) { return bm >= 3 ? 2 : 4; }                    // k-blocks per row group
__host__ __device__ constexpr int a_group_bytes(int bm) { return bm == 1 ? 32 : bm == 3 ? 48 : 64; }
constexpr int S_GROUP_KB = 4, S_GROUP_BYTES = 32;

Geo make_geo(const tq_plan* plan) {
  Geo g;
  g.bm = plan->mse_bits;
  g.d = plan->d;
  g.kba = g.bm > 0 ? (plan->d + 63) / 64 : 0;
  g.kbs = plan->mode == TQ_PROD ? (plan->d + 63) / 64 : 0;
  g.nib = plan->layout == TQ_LAYOUT_NIBBLE ? 1 : 0;
  g.nbi = plan->nb.nbi;
  g.nblk = plan->nb.nbi + plan->nb.nbq;
  g.idx_rb = (int)plan->idx_row_bytes;
  g.qjl_rb = (int)plan->qjl_row_bytes;
  return g;
}

// Coordinate and part of K element e (0, 1) of 32-bit column c of k-block f; coord < 0: zero.  The columns lie as the expansion
// threads form them.
struct Element {
  int coord;
  bool sign;
};
__device__ __forceinline__ Element element_of(const Geo& g, int f, int c, int e) {
  const int nat = 2 * c + e;                                        // centroids of 3 and 4 bits, and of the nibble layout
  const int nsg = 8 * (c >> 2) + (c & 3) + 4 * e;                    // sign bits of the nibble layout
  const int bit = 32 * (c >> 4) + (c & 15) + 16 * e;                 // bit streams of one bit per coordinate
  const int two = 16 * (c >> 3) + 8 * (c & 1) + ((c >> 1) & 3) + 4 * e;   // two-bit codes
  Element r;
  if (g.nib) {
    r.sign = (f & 1) != 0;
    r.coord = nib::coord_of_block(g.nbi, g.idx_rb, g.qjl_rb, g.d, f >> 2, 64 * ((f >> 1) & 1) + (r.sign ? nsg : nat));
    return r;
  }
  r.sign = f >= g.kba;
  const int within = r.sign || g.bm == 1 ? bit : g.bm == 2 ? two : nat;
  r.coord = 64 * (r.sign ? f - g.kba : f) + within;
  if (r.coord >= g.d) r.coord = -1;
  return r;
}

// ------------------------------------------------------------------ query operand and error constants
template <typename T>
__device__ __forceinline__ T block_sum(T v, T* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  T s = 0;
  for (int w = 0; w < 8; ++w) s += red[w];
  return s;
}
__device__ __forceinline__ float block_max(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float s = 0.f;
  for (int w = 0; w < 8; ++w) s = fmaxf(s, red[w]);
  return s;
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}
// Eight 3-bit codes (low 24 bits) as eight nibbles.
__device__ __forceinline__ uint32_t spread3(uint32_t x) {
  x = (x & 0x00000fffu) | ((x & 0x00fff000u) << 4);
  x = (x & 0x003f003fu) | ((x & 0x0fc00fc0u) << 2);
  return (x & 0x07070707u) | ((x & 0x38383838u) << 1);
}

// The exact engine's weights are whole numbers: what rounding them can do to the centroid term of an estimate and to its sign term
// (per unit of gamma), for a query with maxima mx1, mx2 and sum |q'| = l1.
struct EngineRounding {
  int nib, d, planes;   // planes: weights per coordinate of the bit streams
  float amax2;          // 2 max |Walsh coefficient|
  float delta;          // step of the nibble layout's 16-bit centroid table
  float coef;
};
__device__ __forceinline__ float2 engine_error(const EngineRounding& r, float mx1, float mx2, float l1) {
  if (r.nib) {
    const nib::QScale s = nib::make_scale(mx1, mx2);
    // half a unit of the weights of h (at most 128) and of l (at most 255) per coordinate, half a unit of the 16-bit centroid
    return make_float2((float)r.d * 192.f * r.delta * (float)ldexp(1.0, 8 - s.fh) + l1 * r.delta, (float)r.d * (float)(1.0 / s.sq) * r.coef);
  }
  // a weight of bit k of a byte is rounded to 2^(k - f): 255 / 8 half units per weight and byte on average
  auto unit = [](float wmax) {
    if (!(wmax > 0.f)) return 0.f;
    int e;
    frexpf(wmax, &e);
    return ldexpf(1.f, e - 22);
  };
  return make_float2((float)(r.d * r.planes + 64) * 16.f * unit(r.amax2 * mx1 * 1.0001f), (float)(r.d + 64) * 16.f * unit(2.f * mx2 * 1.0001f) * r.coef);
}
EngineRounding engine_rounding(const tq_plan* plan) {
  EngineRounding r;
  r.nib = plan->layout == TQ_LAYOUT_NIBBLE ? 1 : 0;
  r.d = plan->d;
  r.planes = plan->mse_bits == 3 ? 4 : plan->mse_bits == 4 ? 8 : plan->mse_bits;
  r.amax2 = (float)(2.0 * plan->ms.amax);
  r.delta = (float)plan->nb.delta;
  r.coef = plan->coef;
  return r;
}

struct PrepArgs {
  const float* Qcat;
  int64_t ldq;
  int dpad, nq, prod;
  Geo g;
  float cscale;        // 2^ec: the codebook's largest entry times this is in [1, 2)
  int ec;
  float cmax, dcmax;   // largest |c16|, largest |c16 - c 2^ec|
  float coef;
  EngineRounding engine;
  __half* B;           // [kQueries][64 kblocks]
  QueryTerms* terms;
};

// One CTA per query: the fp16 operand row in the order of the k-blocks, the error constant.
__global__ void __launch_bounds__(256) screen_prep_kernel(PrepArgs a) {
  __shared__ float red[8];
  allow_successor();
  wait_for_predecessor();   // the rotated queries are its output; the operand may still be read by it
  const int q = blockIdx.x, tid = threadIdx.x, d = a.g.d;
  const int words = 32 * a.g.kblocks();
  uint32_t* out = reinterpret_cast<uint32_t*>(a.B) + (size_t)q * words;
  const float* qa = a.Qcat + (int64_t)q * a.ldq;
  const float* qs = qa + a.dpad;
  float mx1 = 0.f, mx2 = 0.f;
  bool odd = false, nan = false;
  if (q < a.nq) {
    for (int j = tid; j < d; j += 256) {
      const float u = qa[j], v = a.prod ? qs[j] : 0.f;
      odd |= !(fabsf(u) <= FLT_MAX) || !(fabsf(v) <= FLT_MAX);
      nan |= isnan(a.prod ? v : u);   // the estimate's constant term is the sum of these
      mx1 = fmaxf(mx1, fabsf(u));
      mx2 = fmaxf(mx2, fabsf(v));
    }
  }
  odd = __syncthreads_or(odd) != 0;
  nan = __syncthreads_or(nan) != 0;
  mx1 = block_max(mx1, red);
  mx2 = block_max(mx2, red);
  // the largest operand entry goes to [2^9, 2^10)
  const float sgn = a.coef * a.cscale;
  const float mx = fmaxf(a.g.bm > 0 ? mx1 : 0.f, mx2 * sgn);
  int x = 0;
  if (mx > 0.f && mx <= FLT_MAX) x = 9 - ilogbf(mx);
  odd = odd || !(mx <= FLT_MAX) || x > 60 || x < -60;
  const bool zero = !odd && (a.g.bm == 0 || mx1 == 0.f) && mx2 == 0.f;
  if (q >= a.nq || odd || zero) {   // an absent query, or one whose estimates the bounds do not cover: every row passes
    for (int i = tid; i < words; i += 256) out[i] = 0u;
    if (tid == 0) a.terms[q] = {q >= a.nq ? 0.f : nan ? kNanQuery : zero ? kZeroQuery : 1e30f, 1.f};
    return;
  }
  const float sa = ldexpf(1.f, x), ss = sgn * sa;
  for (int i = tid; i < words; i += 256) {
    uint32_t w = 0u;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const Element el = element_of(a.g, i >> 5, i & 31, e);
      if (el.coord < 0) continue;
      const float v = el.sign ? qs[el.coord] * ss : qa[el.coord] * sa;
      w |= (uint32_t)__half_as_ushort(__float2half_rn(v)) << (16 * e);
    }
    out[i] = w;
  }
  float e1 = 0.f, e2 = 0.f, l1 = 0.f, l2 = 0.f;
  for (int j = tid; j < d; j += 256) {
    if (a.g.bm > 0) {
      const float v = qa[j] * sa, h = __half2float(__float2half_rn(v));
      e1 += fabsf(v - h) * a.cmax + fabsf(v) * a.dcmax;
      l1 += fabsf(v);
    }
    if (a.prod) {
      const float v = qs[j] * ss, h = __half2float(__float2half_rn(v));
      e2 += fabsf(v - h);
      l2 += fabsf(v);
    }
  }
  e1 = block_sum(e1, red);
  e2 = block_sum(e2, red);
  l1 = block_sum(l1, red);
  l2 = block_sum(l2, red);
  if (tid != 0) return;
  const float scale = a.cscale * sa;   // screened values are the estimates times this
  // The tensor core truncates as it adds: 2^-21 of the largest possible sum per instruction is eight times the last place of fp32.
  const float adds = (float)(4 * a.g.kblocks() + 8) * 4.76837158e-7f;
  e1 += adds * l1 * a.cmax + l2 * 2.98023224e-8f;          // gamma below fp16's normal range: 2^-25 absolute
  e2 = e2 * 1.001f + l2 * 4.8828125e-4f + adds * l2;       // gamma to 11 bits
  const float2 engine = engine_error(a.engine, mx1, mx2, l1 / sa);
  e1 += engine.x * scale;
  e2 += engine.y * scale;
  // one constant for both terms, one per cent for the roundings of these sums and of the few fp32 operations behind the accumulator
  a.terms[q] = {fmaxf(e1, e2) * 1.01f + 1e-30f, 1.f / scale};
}

// ------------------------------------------------------------------ scan
struct ScanArgs {
  int64_t n;
  Geo g;
  int ngroups;
  uint32_t tab[4];         // bytes of the codebook in fp16: low bytes of entries 0..3, 4..7, high bytes alike; two bits: entries 0, 1 and 2, 3;
                           // four bits: of the eight positive entries; one bit: tab[0] = the pair of positive entries
  int nqp, ncols;          // queries, MMA columns (128 or 256)
  const QueryTerms* terms;
  const float* gamma;
  const float* norms;
  int64_t step;
  float* dense;
  int64_t lds;
  const float* tau;
  int* count;
  float* cand_s;
  int* cand_i;
  int cap;
  int* status;
};

struct RowGroup {
  int f0, cnt;
  bool sign, from_qjl;
  int x, bytes;
};
template <int BM, bool NIB>
__device__ __forceinline__ RowGroup row_group(const Geo& g, int gi) {
  RowGroup rg;
  if (NIB) {
    rg.f0 = 4 * gi;
    rg.cnt = 4;
    rg.sign = false;
    rg.from_qjl = gi >= g.nbi;
    rg.x = 64 * (rg.from_qjl ? gi - g.nbi : gi);
    rg.bytes = 64;
    return rg;
  }
  constexpr int GA = a_group_kb(BM);
  const int ga = (g.kba + GA - 1) / GA;
  rg.sign = rg.from_qjl = gi >= ga;
  if (!rg.sign) {
    rg.f0 = GA * gi;
    rg.cnt = min(GA, g.kba - GA * gi);
    rg.bytes = a_group_bytes(BM);
    rg.x = gi * rg.bytes;
  } else {
    rg.f0 = g.kba + S_GROUP_KB * (gi - ga);
    rg.cnt = min(S_GROUP_KB, g.kbs - S_GROUP_KB * (gi - ga));
    rg.bytes = S_GROUP_BYTES;
    rg.x = (gi - ga) * S_GROUP_BYTES;
  }
  return rg;
}
// K steps of 16 elements that k-block f needs.  A step holds 16 neighbouring codes of two bits or more; of one-bit streams, half of the
// pairs (b, b + 16) of a word: with 9 to 15 coordinates of a word both of its steps.
template <int BM, bool NIB>
__device__ __forceinline__ int k_steps(const Geo& g, int f) {
  if (NIB) return 4;
  const int left = g.d - 64 * (f < g.kba ? f : f - g.kba);
  if (left >= 64) return 4;
  if (f < g.kba && BM >= 2) return (left + 15) >> 4;
  return 2 * (left >> 5) + ((left & 31) == 0 ? 0 : (left & 31) <= 8 ? 1 : 2);
}

// Eight selectors (nibbles 0..7) -> eight fp16 centroids in natural order.
__device__ __forceinline__ void centroids8(const uint32_t (&tab)[4], uint32_t sel, uint32_t* v) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t s = h == 0 ? sel : sel >> 16;
    const uint32_t lo = prmt(tab[0], tab[1], s), hi = prmt(tab[2], tab[3], s);
    v[2 * h] = prmt(lo, hi, 0x5140u);
    v[2 * h + 1] = prmt(lo, hi, 0x7362u);
  }
}
// The same for 4-bit codes of an antisymmetric codebook: magnitudes from the table, signs from the top bits.
__device__ __forceinline__ void centroids8_wide(const uint32_t (&tab)[4], uint32_t x, uint32_t* v) {
  const uint32_t top = x & 0x88888888u, m = top - (top >> 3);   // 7 where the code is 8 or more
  const uint32_t sel = ~(x ^ m) & 0x77777777u, sg = (x >> 1) & 0x77777777u;   // 8 + i and 7 - i -> magnitude i
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t s = h == 0 ? sel : sel >> 16, t = h == 0 ? sg : sg >> 16;
    const uint32_t lo = prmt(tab[0], tab[1], s), hi = prmt(tab[2], tab[3], s) | prmt(0x80808080u, 0u, t);
    v[2 * h] = prmt(lo, hi, 0x5140u);
    v[2 * h + 1] = prmt(lo, hi, 0x7362u);
  }
}
// Sixteen 2-bit codes: a selector byte 0x10 + 0x22 v names the two bytes of entry v.
__device__ __forceinline__ void centroids16_two(const uint32_t (&tab)[4], uint32_t w, uint32_t* v) {
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const uint32_t sel = ((w >> (2 * s)) & 0x03030303u) * 0x22u + 0x10101010u;
    v[2 * s] = prmt(tab[0], tab[1], sel);
    v[2 * s + 1] = prmt(tab[0], tab[1], sel >> 16);
  }
}
// Two columns at a time: v = acc nu + (rho E - tau), e = (E, E', -tau, -tau').
__device__ __forceinline__ void test_pair(float& v0, float& v1, float nu, float rho, const float4& e) {
  asm("{\n\t.reg .b64 a, b, c, d;\n\t"
      "mov.b64 a, {%3, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
      "fma.rn.f32x2 c, a, b, c;\n\t"
      "mov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %2};\n\t"
      "fma.rn.f32x2 d, a, b, c;\n\t"
      "mov.b64 {%0, %1}, d;\n\t}"
      : "+f"(v0), "+f"(v1)
      : "f"(nu), "f"(rho), "f"(e.x), "f"(e.y), "f"(e.z), "f"(e.w));
}

template <int BM, bool NIB, int MODE>
__global__ void __launch_bounds__(NTHREADS, 1)
screen_kernel(const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmPa, const __grid_constant__ CUtensorMap tmPs,
              const __grid_constant__ ScanArgs a) {
  allow_successor();
  const int rank = (int)cluster_ctarank();
  const int64_t unit = blockIdx.x / 2, nunits = gridDim.x / 2;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* pring = smem + STAGES * STAGE;
  uint64_t* bars = reinterpret_cast<uint64_t*>(pring + PSTAGES * PTILE);
  uint64_t* full = bars;                  // [RING]  TMA, and A stored by its set's four warps of both CTAs -> MMA (the leader's)
  uint64_t* empty = full + RING;          // [RING]  the k-block's MMAs complete
  uint64_t* pfull = empty + RING;         // [PSTAGES]  TMA (packed rows) -> expansion
  uint64_t* pempty = pfull + PSTAGES;     // [PSTAGES]  expansion -> TMA
  uint64_t* dfull = pempty + PSTAGES;     // [2]  accumulator complete -> epilogue
  uint64_t* dfree = dfull + 2;            // [2]  accumulator read -> issuer (the leader's)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(dfree + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  // [128] of two queries each: error constants, then thresholds, negative; scaled like the accumulators
  float4* et = reinterpret_cast<float4*>(reinterpret_cast<unsigned char*>(bars) + 512);
  float* unscale = reinterpret_cast<float*>(et + kQueries / 2);
  int* lcnt = reinterpret_cast<int*>(unscale + kQueries);
  uint2* lbuf = reinterpret_cast<uint2*>(lcnt + kQueries);          // [256][LBUF] (lower bound, row)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkb = a.g.kblocks(), ngroups = a.ngroups;
  const int64_t nrounds = (a.n + 2 * TILE - 1) / (2 * TILE);

  if (threadIdx.x == 0) {
    for (int s = 0; s < RING; ++s) {
      mbar_init(&full[s], 8 + 1);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < PSTAGES; ++s) {
      mbar_init(&pfull[s], 1);
      mbar_init(&pempty[s], 8);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&dfull[i], 1);
      mbar_init(&dfree[i], 2 * NEPI);
    }
    *abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmB);
    tma_prefetch_desc(&tmPa);
    tma_prefetch_desc(&tmPs);
  }
  wait_for_predecessor();   // every input may be its output
  if (threadIdx.x < kQueries) {
    const int q = threadIdx.x;
    float2 v = make_float2(0.f, -INFINITY);
    float un = 0.f;
    if (q < a.nqp) {
      const QueryTerms t = a.terms[q];
      if (t.err >= 0.f) v = make_float2(t.err, MODE == 1 ? -a.tau[q] / t.unscale : 0.f);   // the scale is a power of two
      un = t.unscale;
    }
    float* pair = reinterpret_cast<float*>(et + (q >> 1)) + (q & 1);
    pair[0] = v.x;
    pair[2] = v.y;
    unscale[q] = un;
    lcnt[q] = 0;
  }
  if (warp == 3) tmem_alloc_pair(tmem_slot, TMEM_COLS);
  tc_fence_before();
  cluster_sync();   // the partner's barriers exist before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // The stage of k-block kt was last read by the MMAs of k-block kt - STAGES.
  auto stage_free = [&](uint32_t kt) -> bool {
    const uint32_t kp = kt - STAGES;
    return kt < STAGES || mbar_wait_suspended(&empty[kp % RING], (kp / RING) & 1u, abort_flag, a.status);
  };

  if (warp < NEXP0) {
    if (warp == 0) {
      // ---------------------------------------------------------------- query operand
      if (lane == 0) {
        uint32_t kt = 0;
        bool ok = true;
        for (int64_t rnd = unit; rnd < nrounds && ok; rnd += nunits) {
          for (int f = 0; f < nkb; ++f, ++kt) {
            if (!(ok = stage_free(kt))) break;
            uint64_t* bar = &full[kt % RING];
            if (rank == 0) mbar_arrive_expect_tx(bar, 128u * (uint32_t)a.ncols);
            tma_load_2d_pair(smem + kt % STAGES * STAGE + ATILE, &tmB, bar, f * 64, rank * (a.ncols / 2));   // this CTA's half of the queries
          }
        }
        if (!ok) {
          for (int i = 0; i < 2000; ++i) __nanosleep(1000);   // let copies in flight land
        }
      }
      __syncwarp();
    } else if (warp == 1) {
      // ---------------------------------------------------------------- MMA issuer
      if (lane == 0 && rank == 0) {
        // fp16 x fp16 -> fp32, both K-major
        const uint32_t idesc = (1u << 4) | ((uint32_t)(a.ncols >> 3) << 17) | ((uint32_t)((2 * TILE) >> 4) << 24);
        const uint64_t adesc0 = smem_desc_sw128(smem_u32(smem)), bdesc0 = smem_desc_sw128(smem_u32(smem + ATILE));
        // K steps of the parts' last k-blocks
        const int end0 = a.g.kba - 1, end1 = nkb - 1;
        const int last0 = k_steps<BM, NIB>(a.g, max(end0, 0)), last1 = k_steps<BM, NIB>(a.g, end1);
        bool ok = true;
        uint32_t it = 0, st = 0, at = 0, ph = 0;   // stage and barrier of the next k-block
        for (int64_t rnd = unit; rnd < nrounds && ok; rnd += nunits, ++it) {
          const uint32_t d = it & 1u, d_tmem = tmem_base + d * 256u;
          if (!(ok = mbar_wait_suspended(&dfree[d], ((it >> 1) & 1u) ^ 1u, abort_flag, a.status))) break;
          for (int f = 0; f < nkb; ++f) {
            const uint64_t off = (uint64_t)(st * (STAGE >> 4));
            const uint64_t adesc = adesc0 + off, bdesc = bdesc0 + off;
            const int steps = NIB ? 4 : f == end0 ? last0 : f == end1 ? last1 : 4;
            if (!(ok = mbar_wait_suspended(&full[at], ph, abort_flag, a.status))) break;
            tc_fence_after();
#pragma unroll
            for (int s = 0; s < 4; ++s)
              if (s < steps) umma_bf16_pair(d_tmem, adesc + 2 * s, bdesc + 2 * s, idesc, s != 0 || f != 0 ? 1u : 0u);
            umma_commit_pair(&empty[at]);
            if (++st == STAGES) st = 0;
            if (++at == RING) {
              at = 0;
              ph ^= 1u;
            }
          }
          if (ok) umma_commit_pair(&dfull[d]);
        }
      }
      __syncwarp();
    } else if (warp == 2) {
      // ---------------------------------------------------------------- packed rows
      if (lane == 0) {
        uint32_t pst = 0, ph = 1;
        bool ok = true;
        for (int64_t rnd = unit; rnd < nrounds && ok; rnd += nunits) {   // rows past the last one read zeros
          for (int gi = 0; gi < ngroups; ++gi) {
            const RowGroup rg = row_group<BM, NIB>(a.g, gi);
            if (!(ok = mbar_wait_suspended(&pempty[pst], ph, abort_flag, a.status))) break;
            mbar_arrive_expect_tx(&pfull[pst], (uint32_t)(TILE * rg.bytes));
            tma_load_2d(pring + pst * PTILE, rg.from_qjl ? &tmPs : &tmPa, &pfull[pst], rg.x, (int)((rnd * 2 + rank) * TILE));
            if (++pst == PSTAGES) {
              pst = 0;
              ph ^= 1u;
            }
          }
        }
        if (!ok) {
          for (int i = 0; i < 2000; ++i) __nanosleep(1000);
        }
      }
      __syncwarp();
    }
  } else if (warp >= NEXP0 && warp < NEPI0) {
    // ---------------------------------------------------------------- expansion: thread = row; the sets take the k-blocks in turn
    const int set = (warp - NEXP0) >> 2, quad = warp & 3;
    const int r = quad * 32 + lane;
    bool ok = true;
    uint32_t it = 0;
    auto load_gamma = [&](int64_t tl) -> float {
      const int64_t rw = tl * TILE + r;
      return ((NIB || a.g.kbs > 0) && rw < a.n) ? __ldg(a.gamma + rw * a.step) : 0.f;
    };
    float g_next = load_gamma(unit * 2 + rank);
    for (int64_t rnd = unit; rnd < nrounds && ok; rnd += nunits, ++it) {
      const int64_t tile = rnd * 2 + rank;
      const float gm = g_next;
      g_next = load_gamma(tile + 2 * nunits);
      const uint32_t g16 = (uint32_t)__half_as_ushort(__float2half_rn(row_terms(1.f, gm).gamma));
      const uint32_t neg = (g16 | (g16 << 16)) ^ 0x80008000u;
      const uint32_t kt0 = it * (uint32_t)nkb;
      // The tensor core of this SM reads what these threads write, in a pair too: the proxy fence orders the writes, the arrival only
      // tells the leader's issuer.
      auto fill = [&](uint32_t kt, auto&& pieces) {
        const uint32_t st = kt % STAGES;
        if (!(ok = stage_free(kt))) return;
        unsigned char* dst = smem + st * STAGE + r * 128;
        // 16-byte piece p of the row, 128-byte swizzle
        pieces([&](int p, const uint32_t* v) { *reinterpret_cast<uint4*>(dst + ((p ^ (r & 7)) << 4)) = make_uint4(v[0], v[1], v[2], v[3]); });
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive_leader(&full[kt % RING]);
      };
      auto mine = [&](uint32_t kt) { return (int)(kt & 1u) == set; };
      for (int gi = 0; gi < ngroups && ok; ++gi) {
        const RowGroup rg = row_group<BM, NIB>(a.g, gi);
        const uint32_t gc = it * (uint32_t)ngroups + (uint32_t)gi, pst = gc % PSTAGES;
        if (!(ok = mbar_wait_suspended(&pfull[pst], (gc / PSTAGES) & 1u, abort_flag, a.status))) break;
        const unsigned char* ps = pring + pst * PTILE;
        uint32_t w[16];
        if (rg.bytes == 64) {          // 64-byte swizzle: piece c at c ^ ((row >> 1) & 3)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint4 v4 = *reinterpret_cast<const uint4*>(ps + r * 64 + ((j ^ ((r >> 1) & 3)) << 4));
            w[4 * j] = v4.x; w[4 * j + 1] = v4.y; w[4 * j + 2] = v4.z; w[4 * j + 3] = v4.w;
          }
        } else if (rg.bytes == 48) {   // plain
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const uint4 v4 = *reinterpret_cast<const uint4*>(ps + r * 48 + j * 16);
            w[4 * j] = v4.x; w[4 * j + 1] = v4.y; w[4 * j + 2] = v4.z; w[4 * j + 3] = v4.w;
          }
          w[12] = w[13] = w[14] = w[15] = 0u;
        } else {                       // 32-byte swizzle: piece c at c ^ ((row >> 2) & 1)
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const uint4 v4 = *reinterpret_cast<const uint4*>(ps + r * 32 + ((j ^ ((r >> 2) & 1)) << 4));
            w[4 * j] = v4.x; w[4 * j + 1] = v4.y; w[4 * j + 2] = v4.z; w[4 * j + 3] = v4.w;
          }
#pragma unroll
          for (int j = 8; j < 16; ++j) w[j] = 0u;
        }
        release_stage(&pempty[pst], lane);
        const uint32_t kt = kt0 + (uint32_t)rg.f0;
        if (NIB) {
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            if (ok && mine(kt + 2 * half))
              fill(kt + 2 * half, [&](auto&& put) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  uint32_t v[4];
                  centroids8(a.tab, w[8 * half + j] & 0x77777777u, v);
                  put(j, v);
                }
              });
            if (ok && mine(kt + 2 * half + 1))
              fill(kt + 2 * half + 1, [&](auto&& put) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  uint32_t v[4];
#pragma unroll
                  for (int p = 0; p < 4; ++p) v[p] = neg ^ ((w[8 * half + j] << (12 - 4 * p)) & 0x80008000u);
                  put(j, v);
                }
              });
          }
        } else if (BM <= 1 || rg.sign) {
          const uint32_t pair = BM == 1 && !rg.sign ? a.tab[0] ^ 0x80008000u : neg;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (ok && j < rg.cnt && mine(kt + j))
              fill(kt + j, [&](auto&& put) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {   // bits b and b + 16 of a word are a pair
                  uint32_t v[4];
#pragma unroll
                  for (int p = 0; p < 4; ++p) v[p] = pair ^ ((w[2 * j + (i >> 2)] << (15 - 4 * (i & 3) - p)) & 0x80008000u);
                  put(i, v);
                }
              });
          }
        } else {
#pragma unroll
          for (int j = 0; j < a_group_kb(BM); ++j) {
            if (ok && j < rg.cnt && mine(kt + j))
              fill(kt + j, [&](auto&& put) {
                if (BM == 2) {
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    uint32_t v[8];
                    centroids16_two(a.tab, w[4 * j + i], v);
                    put(2 * i, v);
                    put(2 * i + 1, v + 4);
                  }
                } else if (BM == 3) {
#pragma unroll
                  for (int i = 0; i < 2; ++i) {   // 32 codes in three words
                    const uint32_t* x = w + 6 * j + 3 * i;
                    const uint32_t sel[4] = {x[0], __funnelshift_r(x[0], x[1], 24), __funnelshift_r(x[1], x[2], 16), x[2] >> 8};
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                      uint32_t v[4];
                      centroids8(a.tab, spread3(sel[p] & 0xffffffu), v);
                      put(4 * i + p, v);
                    }
                  }
                } else {
#pragma unroll
                  for (int i = 0; i < 8; ++i) {
                    uint32_t v[4];
                    centroids8_wide(a.tab, w[8 * j + i], v);
                    put(i, v);
                  }
                }
              });
          }
        }
      }
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- epilogue: thread = row, a quarter of the columns
    const int h = (warp - NEPI0) >> 2, quad = warp & 3;
    const int r = quad * 32 + lane, chunks = a.ncols / 128;   // chunks of 32 columns
    bool ok = true;
    uint32_t it = 0;
    auto load = [&](const float* src, int64_t tl, float otherwise) -> float {
      const int64_t rw = tl * TILE + r;
      return (src != nullptr && rw < a.n) ? __ldg(src + rw * a.step) : otherwise;
    };
    const float* gsrc = (NIB || a.g.kbs > 0) ? a.gamma : nullptr;
    float nu_next = load(a.norms, unit * 2 + rank, 1.f), g_next = load(gsrc, unit * 2 + rank, 0.f);
    for (int64_t rnd = unit; rnd < nrounds && ok; rnd += nunits, ++it) {
      const int64_t tile = rnd * 2 + rank, row = tile * TILE + r;
      // (a NaN scalar makes every estimate NaN, which no list holds)
      const bool row_ok = row < a.n && (MODE == 0 || !(isnan(nu_next) || isnan(g_next)));
      const RowTerms t = row_terms(nu_next, g_next);
      nu_next = load(a.norms, tile + 2 * nunits, 1.f);
      g_next = load(gsrc, tile + 2 * nunits, 0.f);
      const uint32_t d = it & 1u;
      if (!(ok = mbar_wait_suspended(&dfull[d], (it >> 1) & 1u, abort_flag, a.status))) break;
      tc_fence_after();
      const uint32_t addr = tmem_base + ((uint32_t)(quad * 32) << 16) + d * 256u;
#pragma unroll 1
      for (int c = 0; c < chunks; ++c) {
        const int q0 = (h * chunks + c) * 32;
        uint32_t acc[32];
        __syncwarp();
        tmem_ld32(addr + q0, acc);
        tmem_ld_wait();
        if (c == chunks - 1) {   // the last columns are in registers
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_leader(&dfree[d]);
        }
        if (q0 >= a.nqp) continue;
        auto err_of = [&](int q) -> float { return reinterpret_cast<const float*>(et + (q >> 1))[q & 1]; };
        if (MODE == 0) {
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float low = fmaxf(fmaf(__uint_as_float(acc[i]), t.nu, -t.rho * err_of(q0 + i)) * unscale[q0 + i], -FLT_MAX);
            if (row_ok && q0 + i < a.nqp && TQ_DEVICE_CHECK(row >= 0 && row < a.lds, a.status)) a.dense[(int64_t)(q0 + i) * a.lds + row] = low;
          }
          continue;
        }
        // Sign bit clear: the row's upper bound reaches the threshold.  The signs of eight columns are ANDed, one three-input
        // operation per pair, and looked at together.
        float v[32];
        uint32_t none[4] = {~0u, ~0u, ~0u, ~0u};
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          v[i] = __uint_as_float(acc[i]);
          v[i + 1] = __uint_as_float(acc[i + 1]);
          test_pair(v[i], v[i + 1], t.nu, t.rho, et[(q0 + i) >> 1]);
          none[i >> 3] &= __float_as_uint(v[i]) & __float_as_uint(v[i + 1]);
        }
        if (!row_ok || (int)(none[0] & none[1] & none[2] & none[3]) < 0) continue;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          if ((int)none[g] < 0) continue;
          uint32_t hits = 0u;
#pragma unroll
          for (int i = 0; i < 8; ++i) hits |= (~__float_as_uint(v[8 * g + i]) >> 31) << i;
          while (hits != 0u) {   // a lane takes its own hits one after the other
            const int i = __ffs((int)hits) - 1, q = q0 + 8 * g + i;
            hits &= hits - 1u;
            if (q >= a.nqp) break;   // absent queries have no list: rho E is NaN for them where a row's bound is infinite
            const float x0 = (i & 1) ? v[8 * g + 1] : v[8 * g], x1 = (i & 1) ? v[8 * g + 3] : v[8 * g + 2];
            const float x2 = (i & 1) ? v[8 * g + 5] : v[8 * g + 4], x3 = (i & 1) ? v[8 * g + 7] : v[8 * g + 6];
            const float y0 = (i & 2) ? x1 : x0, y1 = (i & 2) ? x3 : x2, val = (i & 4) ? y1 : y0;
            const float* pair = reinterpret_cast<const float*>(et + (q >> 1)) + (q & 1);
            // the lower bound: val + tau - 2 rho E.  val is rounded on the grid of tau, which a row of small norm may lie far below.
            const float low = fmaf(fabsf(pair[2]), -kThresholdSlack, fmaf(-2.f * t.rho, pair[0], val) - pair[2]);
            const int ls = atomicAdd(&lcnt[q], 1);
            if (ls < LBUF) {
              lbuf[q * LBUF + ls] = make_uint2(__float_as_uint(low), (uint32_t)row);
            } else {   // the CTA's buffer is full: straight to the list
              const int slot = atomicAdd(a.count + q, 1);
              if (slot < a.cap && TQ_DEVICE_CHECK(slot >= 0 && row < a.n, a.status)) {
                a.cand_s[(int64_t)q * a.cap + slot] = fmaxf(low * unscale[q], -FLT_MAX);
                a.cand_i[(int64_t)q * a.cap + slot] = (int)row;
              }
            }
          }
        }
      }
    }
    __syncwarp();
  }

  tc_fence_before();
  cluster_sync();   // neither CTA leaves while the partner may still arrive on its barriers
  if (warp == 3) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, TMEM_COLS);
  }
  if (MODE == 1) {
    for (int q = warp; q < a.nqp; q += NTHREADS / 32) {
      const int m = min(lcnt[q], LBUF);
      if (m == 0) continue;
      int base = 0;
      if (lane == 0) base = atomicAdd(a.count + q, m);
      base = __shfl_sync(0xffffffffu, base, 0);
      for (int i = lane; i < m; i += 32) {
        const int slot = base + i;
        if (slot < a.cap && TQ_DEVICE_CHECK(slot >= 0, a.status)) {
          const uint2 e = lbuf[q * LBUF + i];
          a.cand_s[(int64_t)q * a.cap + slot] = fmaxf(__uint_as_float(e.x) * unscale[q], -FLT_MAX);   // (not finite: no lower bound)
          a.cand_i[(int64_t)q * a.cap + slot] = (int)e.y;
        }
      }
    }
  }
}

template <int BM, bool NIB, int MODE>
cudaError_t launch(const CUtensorMap& mb, const CUtensorMap& pa, const CUtensorMap& ps, const ScanArgs& args, cudaStream_t st) {
  auto kern = screen_kernel<BM, NIB, MODE>;
  static std::atomic<unsigned long long> smem_devices{0};
  cudaError_t e = allow_largest_smem(reinterpret_cast<const void*>(kern), smem_devices);
  if (e != cudaSuccess) return e;
  const int64_t rounds = (args.n + 2 * TILE - 1) / (2 * TILE);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * std::min<int64_t>(rounds, sm_count() / 2)));
  cfg.blockDim = dim3(NTHREADS);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  count_launches(1);
  e = cudaLaunchKernelEx(&cfg, kern, mb, pa, ps, args);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int MODE>
cudaError_t launch_bm(const CUtensorMap& mb, const CUtensorMap& pa, const CUtensorMap& ps, const ScanArgs& a, cudaStream_t st) {
  if (a.g.nib) return launch<3, true, MODE>(mb, pa, ps, a, st);
  switch (a.g.bm) {
    case 0: return launch<0, false, MODE>(mb, pa, ps, a, st);
    case 1: return launch<1, false, MODE>(mb, pa, ps, a, st);
    case 2: return launch<2, false, MODE>(mb, pa, ps, a, st);
    case 3: return launch<3, false, MODE>(mb, pa, ps, a, st);
    default: return launch<4, false, MODE>(mb, pa, ps, a, st);
  }
}

// The codebook in fp16, scaled by a power of two so that its largest entry lies in [1, 2).
struct Table {
  int ec;
  float c16[16];
  uint16_t bits[16];
  float cmax, dcmax;
};
Table make_table(const tq_plan* plan) {
  Table t = {};
  const int levels = plan->mse_bits > 0 ? 1 << plan->mse_bits : 0;
  double mx = 0.0;
  for (int i = 0; i < levels; ++i) mx = std::max(mx, std::fabs((double)plan->cb.c[i]));
  t.ec = mx > 0.0 ? -std::ilogb(mx) : 0;
  for (int i = 0; i < levels; ++i) {
    const float v = (float)std::ldexp((double)plan->cb.c[i], t.ec);
    const __half_raw h = __half(__float2half_rn(v));
    t.bits[i] = h.x;
    t.c16[i] = __half2float(__half(h));
  }
  if (plan->mse_bits == 1 || plan->mse_bits == 4) {   // expanded from the positive half: the codebook is antisymmetric
    for (int i = 0; i < levels / 2; ++i) {
      t.bits[i] = t.bits[levels - 1 - i] ^ 0x8000u;
      t.c16[i] = -t.c16[levels - 1 - i];
    }
  }
  for (int i = 0; i < levels; ++i) {
    t.cmax = std::max(t.cmax, std::fabs(t.c16[i]));
    t.dcmax = std::max(t.dcmax, (float)std::fabs((double)t.c16[i] - std::ldexp((double)plan->cb.c[i], t.ec)));
  }
  t.dcmax *= 1.001f;
  return t;
}

int columns(int nqp) { return nqp > kQueries / 2 ? kQueries : kQueries / 2; }
size_t operand_bytes(const Geo& g) { return (size_t)kQueries * g.kblocks() * 128; }

}  // namespace

int k_blocks(const tq_plan* plan) { return make_geo(plan).kblocks(); }

size_t workspace_bytes(const tq_plan* plan) { return (operand_bytes(make_geo(plan)) + kQueries * sizeof(QueryTerms) + 255) / 256 * 256; }

const QueryTerms* query_terms(const tq_plan* plan, const void* workspace) {
  return reinterpret_cast<const QueryTerms*>(static_cast<const char*>(workspace) + operand_bytes(make_geo(plan)));
}

int prepare(const tq_plan* plan, const float* Qcat, int nqp, void* workspace, cudaStream_t st, const char* who) {
  const Table t = make_table(plan);
  PrepArgs a;
  a.Qcat = Qcat;
  a.ldq = (int64_t)plan->ncat * plan->dpad;
  a.dpad = plan->dpad;
  a.nq = nqp;
  a.prod = plan->mode == TQ_PROD ? 1 : 0;
  a.g = make_geo(plan);
  a.ec = t.ec;
  a.cscale = (float)std::ldexp(1.0, t.ec);
  a.cmax = t.cmax;
  a.dcmax = t.dcmax;
  a.coef = plan->coef;
  a.engine = engine_rounding(plan);
  a.B = static_cast<__half*>(workspace);
  a.terms = const_cast<QueryTerms*>(query_terms(plan, workspace));
  count_launches(1);
  TQ_CHECK_CUDA(launch_dependent(screen_prep_kernel, dim3((unsigned)columns(nqp)), dim3(256), 0, st, a), who);
  return TQ_OK;
}

int run(const tq_plan* plan, int nqp, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma, const float* norms,
        float* dense, int64_t lds, const float* tau, int* count, float* cand_s, int* cand_i, int cap, const void* workspace,
        cudaStream_t st, const char* who, int64_t step) {
  const Table t = make_table(plan);
  ScanArgs a;
  a.g = make_geo(plan);
  const Geo& g = a.g;
  const int ga = g.bm > 0 ? (g.kba + a_group_kb(g.bm) - 1) / a_group_kb(g.bm) : 0;
  a.ngroups = g.nib ? g.nblk : ga + (g.kbs + S_GROUP_KB - 1) / S_GROUP_KB;
  a.n = n;
  a.nqp = nqp;
  a.ncols = columns(nqp);
  a.terms = query_terms(plan, workspace);
  a.gamma = gamma;
  a.norms = norms;
  a.step = step;
  a.dense = dense;
  a.lds = lds;
  a.tau = tau;
  a.count = count;
  a.cand_s = cand_s;
  a.cand_i = cand_i;
  a.cap = cap;
  a.status = plan->d_status;
  for (int p = 0; p < 4; ++p) a.tab[p] = 0u;
  if (g.bm == 1) {
    a.tab[0] = (uint32_t)t.bits[1] * 0x10001u;
  } else if (g.bm == 2) {
    for (int i = 0; i < 4; ++i) a.tab[i >> 1] |= (uint32_t)t.bits[i] << (16 * (i & 1));
  } else if (g.bm >= 3) {
    for (int i = 0; i < 8; ++i) {
      const uint16_t h = g.bm == 4 ? t.bits[8 + i] : t.bits[i];
      a.tab[i >> 2] |= (uint32_t)(h & 255u) << (8 * (i & 3));
      a.tab[2 + (i >> 2)] |= (uint32_t)(h >> 8) << (8 * (i & 3));
    }
  }
  CUtensorMap mb, pa, ps;
  TQ_REQUIRE(make_half_map(&mb, static_cast<const __half*>(workspace), kQueries, 64 * g.kblocks(), 64 * g.kblocks(), a.ncols / 2), TQ_ERR_CUDA,
             "%s: cuTensorMapEncodeTiled failed (query operand)", who);
  const int ab = g.nib ? 64 : a_group_bytes(g.bm), sb = g.nib ? 64 : S_GROUP_BYTES;
  if (g.bm > 0)
    TQ_REQUIRE(make_byte_map(&pa, idx, (uint64_t)n, plan->idx_row_bytes, plan->idx_row_bytes * step, ab, TILE, ab == 48 ? 0 : ab), TQ_ERR_CUDA,
               "%s: cuTensorMapEncodeTiled failed (idx rows)", who);
  if (plan->mode == TQ_PROD)
    TQ_REQUIRE(make_byte_map(&ps, qjl, (uint64_t)n, plan->qjl_row_bytes, plan->qjl_row_bytes * step, sb, TILE, sb), TQ_ERR_CUDA,
               "%s: cuTensorMapEncodeTiled failed (qjl rows)", who);
  if (g.bm == 0) pa = ps;
  if (plan->mode != TQ_PROD) ps = pa;
  TQ_CHECK_CUDA(dense != nullptr ? launch_bm<0>(mb, pa, ps, a, st) : launch_bm<1>(mb, pa, ps, a, st), who);
  return TQ_OK;
}

}  // namespace screen
}  // namespace tq
