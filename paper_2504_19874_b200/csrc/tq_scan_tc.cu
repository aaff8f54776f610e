// Many-query packed-code scan on tcgen05: the same bit-plane form of the estimator as in
// tq_scan_mma.cu (codebook expanded over the index bits, raw bits and parity words as a 0/1 matrix,
// query weights as fixed-point radix-256 digits, identical integers), but with the multiply-accumulate
// on the 5th-generation tensor cores:
//     D[128 vectors, 96 columns] += A[128, 32] * B[96, 32]^T,   kind::i8, s32 accumulators in TMEM.
// 96 columns hold 32 queries x 3 digits, so one pass over the codes serves 32 queries and the decode
// (one AND per four bits, once per vector) is amortised over all of them.  A tcgen05 MMA of this shape
// costs about the same 55-64 cycles for any N <= 128, which is why this path is for many queries and
// the register-fed mma.sync path for few.
//
// The A operand never touches shared memory: byte-expanded bit planes are 8x the packed codes, and
// writing + reading them there would cost more shared-memory cycles than the MMAs take.  Each
// transform thread owns one vector row = one TMEM lane; it expands the row's four packed words of a
// k-block into 32 registers and stores them with tcgen05.st into the 32 TMEM columns of that k-block,
// from where the MMA takes A directly.
//
// CTA (one per SM, persistent over pairs of 128-vector tiles):
//   warp 0       TMA producer: per k-block (128 K-bytes) one [96 rows x 128 B] box of B (128-byte swizzle); per
//                four k-blocks the packed rows of the pair ([256 rows x 32..64 B], swizzled for row-per-thread reads)
//   warps 1..2   MMA issuers (warp 1 owns TMEM): k-blocks alternate between them, 8 MMAs (K = 32, 4 per tile)
//                + one commit each.  A tcgen05.commit keeps its thread for ~350 cycles while the 8 MMAs take
//                ~420, so a single issuer leaves the tensor pipe idle half of the time (measured: 95 cycles
//                per MMA with one issuing thread, 70 with two).
//   warps 3..10  transform + epilogue (thread = vector row): zero the row's accumulators (tcgen05.st), then per
//                k-block the row's packed bytes from shared memory, 3 index words + their parity word (b_m = 3)
//                -> 32 x (w & (0x01010101 << k)) -> tcgen05.st; after the last k-block the row's accumulators
//                are read back (tcgen05.ld), the digits recombined, estimates emitted.
// Every MMA accumulates onto the zeroed accumulators; the sums are integers, so the order in which the
// k-blocks of the two issuers reach the pipe does not matter.
// TMEM (512 columns): tile t: MSE-part accumulator at 192 t + [0, 96), QJL-part at 192 t + [96, 192);
// A: two k-block slots of 32 columns per tile at 384 + 64 t.  The two tiles share every B box (halves
// the L2 traffic of B).  Rings: 2 A slots (TMEM), 8 B stages and 4 packed-row stages (shared memory) with
// full mbarriers; one tcgen05.commit per k-block releases both the A slot and the B stage; accumulator-full
// barrier (one commit per issuer).  Ring positions and phases are masks and shifts of 32-bit counters: the
// single-lane roles run dependent instruction chains, where 64-bit division costs real time.  All waits
// are bounded.
//
// Calls of more than 32 queries run the wide form of this kernel (tq_scan_tcw.cuh: 64 queries per pass, one tile
// per iteration, four A slots, N = 192); this one serves 7..32 queries and the last, short pass of a longer call.
#include <atomic>
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "tq_nib_common.cuh"
#include "tq_quantize_tc.h"
#include "tq_scan_tc.h"
#include "tq_screen_tc.h"
#include "tq_tc.cuh"

namespace tq {
namespace tscan {

namespace {

constexpr int TILE = 128;              // vectors per M tile = TMEM lanes
constexpr int LIMBS = 3;               // signed radix-256 digits per weight (|J| < 2^23)
constexpr int NCOL = 96;               // MMA N: 3 digits x 32 queries, digit-major (column = 32 digit + query)
constexpr int KB_BYTES = 128;          // K extent of one k-block (one swizzled row)
constexpr int A_SLOTS = 2;             // k-blocks of A per tile resident in TMEM
constexpr int B_STAGES = 8;            // ring of B tiles in shared memory (TMA from L2); a power of two, so that ring
                                       // positions and phases of 32-bit counters are masks and shifts
constexpr int BTILE_BYTES = NCOL * KB_BYTES;         // 12 KB
constexpr int P_STAGES = 4;            // ring of packed-row groups (4 k-blocks of the pair's 256 rows each)
constexpr int PTILE_BYTES = 2 * TILE * 64;           // 16 KB: 256 rows x at most 64 bytes
constexpr int D_COLS = 2 * NCOL;                     // accumulator columns per tile (MSE part, QJL part)
constexpr int A_COL0 = 2 * D_COLS;                   // first TMEM column of the A slots
constexpr int N_ISSUERS = 2;             // MMA-issuing warps (a tcgen05.commit stalls its thread; a second issuer hides it)
// The barrier rings count on this number: a parity wait also passes when its barrier is two completions behind, so the
// thread that waits for k-block k must itself have waited for the completion before it on the same barrier -- A_SLOTS
// and B_STAGES are multiples of N_ISSUERS.  (Three issuers with rings of 6 / 9 / 16 barriers, as in the 64-query
// kernel, were measured here: 464 against 471 us per pass; this kernel is bound by its transform warps.)
static_assert(A_SLOTS % N_ISSUERS == 0 && B_STAGES % N_ISSUERS == 0, "a waiter has seen the completion before the one it waits for");
constexpr int NTHREADS = 32 * (1 + N_ISSUERS + 8);
constexpr int TMEM_COLS = 512;
constexpr int LBUF = 128;              // candidates per query a CTA collects in shared memory before it appends them
constexpr size_t kConstBytes = 256 * 48;             // per-query constants of one group

struct QConst {
  float sa, ca;    // a = T_a * sa + ca   (MSE term)
  float ss, cs;    // s = T_s * ss + cs   (QJL term)
  int fa, fs;
  int pad[2];
};

struct Geo {
  int bm, d, dpad;
  int widx, wq;    // 32-bit words per idx / qjl row
  int kba, kbs;    // k-blocks of the MSE part and of the QJL part
  // TQ_LAYOUT_NIBBLE: every 64-byte block of the combined row [idx row | qjl row] gives three k-blocks in turn --
  // the h bytes (signed A), the l bytes, the sign bits -- of its 128 coordinates; kba holds their total, kbs = 0
  int nib, nbi, nblk, idx_rb, qjl_rb;
};

__host__ __device__ inline int div_up(int a, int b) { return (a + b - 1) / b; }
// packed idx bytes of one row consumed by a group of four k-blocks
__host__ __device__ constexpr int group_bytes(int bm) { return bm == 3 ? 48 : bm == 4 ? 32 : 64; }

Geo make_geo(const tq_plan* plan) {
  Geo g;
  g.bm = plan->mse_bits;
  g.d = plan->d;
  g.dpad = plan->dpad;
  g.widx = (int)(plan->idx_row_bytes / 4);
  g.wq = (plan->mode == TQ_PROD) ? (int)(plan->qjl_row_bytes / 4) : 0;
  g.kba = g.bm == 0 ? 0 : g.bm == 3 ? div_up(g.widx, 3) : g.bm == 4 ? div_up(g.widx, 2) : div_up(g.widx, 4);
  g.kbs = div_up(g.wq, 4);
  g.nib = plan->layout == TQ_LAYOUT_NIBBLE ? 1 : 0;
  g.nbi = plan->nb.nbi;
  g.nblk = plan->nb.nbi + plan->nb.nbq;
  g.idx_rb = (int)plan->idx_row_bytes;
  g.qjl_rb = (int)plan->qjl_row_bytes;
  if (g.nib) {
    g.kba = 3 * g.nblk;
    g.kbs = 0;
  }
  return g;
}

// K slot (part, k-block, word wl of the block, bit of the word) -> (coordinate, Walsh term).
// MSE part, b_m = 1, 2: four index words per block.  b_m = 3: the three words of one 96-bit group of 32
// coordinates and their parity word.  b_m = 4: two index words and their two words of 3-subset parities.
struct Slot {
  int coord, term;
};
__device__ inline Slot slot_a(const Geo& g, int kb, int wl, int bit) {
  if (g.bm <= 2) {
    const int P = 32 * (4 * kb + wl) + bit;
    return {P / g.bm, P % g.bm};
  }
  if (g.bm == 3) {
    if (wl < 3) {
      const int P = 32 * (3 * kb + wl) + bit;
      return {P / 3, P % 3};
    }
    const int m = bit % 3;
    const int c = (m == 0) ? bit / 3 : (m == 1) ? (32 + bit) / 3 : (64 + bit) / 3;
    return {32 * kb + c, 4};
  }
  if (wl < 2) {
    const int P = 32 * (2 * kb + wl) + bit;
    return {P / 4, P % 4};
  }
  return {8 * (2 * kb + wl - 2) + bit / 4, 4 + (bit & 3)};
}

// The parity word of 32 three-bit codes, and the 3-subset parities of eight four-bit codes.
__device__ __forceinline__ uint32_t parity3(uint32_t w0, uint32_t w1, uint32_t w2) {
  const uint32_t p0 = w0 ^ __funnelshift_r(w0, w1, 1) ^ __funnelshift_r(w0, w1, 2);
  const uint32_t p1 = w1 ^ __funnelshift_r(w1, w2, 1) ^ __funnelshift_r(w1, w2, 2);
  const uint32_t p2 = w2 ^ (w2 >> 1) ^ (w2 >> 2);
  return (p0 & 0x49249249u) | (p1 & 0x92492492u) | (p2 & 0x24924924u);
}
__device__ __forceinline__ uint32_t parities4(uint32_t x) {
  const uint32_t M = 0x11111111u, s1 = x >> 1, s2 = x >> 2, s3 = x >> 3;
  return ((x ^ s1 ^ s2) & M) | (((x ^ s1 ^ s3) & M) << 1) | (((x ^ s2 ^ s3) & M) << 2) | (((s1 ^ s2 ^ s3) & M) << 3);
}

// ------------------------------------------------------------------ per-query constants and B matrices
// Ba[pass*96 + n][kba*128], Bs[pass*96 + n][kbs*128], n = 32 * digit + (query in pass); K-major int8.
// Byte kappa of a k-block = (2 wl + k / 4) * 16 + (k % 4) * 4 + i  <->  bit 8 i + k of word wl: the order in
// which the transform threads lay out their registers.
// Nibble layout: one B matrix Bn[pass*96 + n][3 nblk * 128]; k-block 3 b + type of block b.  K-byte kappa of an h or l
// k-block <-> coordinate kappa of the block; of a sign k-block: register kappa / 4 = 2 word + parity, byte i = kappa % 4
// <-> coordinate 8 word + 2 i + parity (low nibbles, parity 0, have the value 8 and carry 16 J; high nibbles 128 and J).
struct OperandArgs {
  const float* Qcat;
  int64_t ldq;
  int nqg, dpad, prod;
  Geo g;
  double alpha[8], amax, csum;
  double delta;     // nibble layout: step of the centroid table
  QConst* qc;
  uint8_t* Ba;
  uint8_t* Bs;
};

// 2^e as a double, e in the normal range.
__device__ __forceinline__ double pow2_of(int e) { return __hiloint2double((e + 1023) << 20, 0); }

// Maxima and sums of a rotated query, all threads of a CTA of 256.
__device__ __forceinline__ QConst query_constants(const OperandArgs& a, const float* q) {
  __shared__ double red[4][8];
  __shared__ QConst shared_c;
  double mx1 = 0.0, sm1 = 0.0, mx2 = 0.0, sm2 = 0.0;
  for (int j = threadIdx.x; j < a.g.d; j += 256) {
    const double v = (double)q[j];
    mx1 = fmax(mx1, fabs(v));
    sm1 += v;
    if (a.prod) {
      const double u = (double)q[a.dpad + j];
      mx2 = fmax(mx2, fabs(u));
      sm2 += u;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mx1 = fmax(mx1, __shfl_xor_sync(0xffffffffu, mx1, o));
    mx2 = fmax(mx2, __shfl_xor_sync(0xffffffffu, mx2, o));
    sm1 += __shfl_xor_sync(0xffffffffu, sm1, o);
    sm2 += __shfl_xor_sync(0xffffffffu, sm2, o);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    red[0][warp] = mx1; red[1][warp] = sm1; red[2][warp] = mx2; red[3][warp] = sm2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) {
      mx1 = fmax(mx1, red[0][w]); sm1 += red[1][w];
      mx2 = fmax(mx2, red[2][w]); sm2 += red[3][w];
    }
    // |W| < 2^e with W = 2 alpha q'  ->  |W| 2^(22-e) < 2^22: three signed radix-256 digits hold it.  The same
    // exponent as in the register-fed scan, so that both engines form identical integers and estimates.
    auto expo = [](double wmax) {
      if (!(wmax > 0.0) || !isfinite(wmax)) return 0;
      int e;
      frexp(wmax, &e);
      return 22 - e;
    };
    QConst c;
    c.fa = expo(2.0 * a.amax * mx1);
    c.fs = expo(2.0 * mx2);
    c.sa = (float)ldexp(1.0, -c.fa);
    c.ss = (float)ldexp(1.0, -c.fs);
    c.ca = (float)(a.csum * sm1);
    c.cs = (float)(-sm2);
    c.pad[0] = c.pad[1] = 0;
    shared_c = c;
  }
  __syncthreads();
  return shared_c;
}

// Nibble layout: one warp, the same reductions in the same order as the register-fed engine's (lane-strided maxima in fp32, the
// sum of q'' in fp64 folded by xor shuffles).
__device__ __forceinline__ QConst query_constants_nib(const OperandArgs& a, const float* q) {
  __shared__ QConst shared_c;
  const int lane = threadIdx.x;
  if (threadIdx.x < 32) {
    float mx1 = 0.f, mx2 = 0.f;
    double sm2 = 0.0;
#pragma unroll 8
    for (int j = lane; j < a.g.d; j += 32) {
      mx1 = fmaxf(mx1, fabsf(q[j]));
      const float u = q[a.dpad + j];
      mx2 = fmaxf(mx2, fabsf(u));
      sm2 += (double)u;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, o));
      mx2 = fmaxf(mx2, __shfl_xor_sync(0xffffffffu, mx2, o));
      sm2 += __shfl_xor_sync(0xffffffffu, sm2, o);
    }
    if (lane == 0) {
      const nib::QScale s = nib::make_scale(mx1, mx2);
      const nib::QConst n = nib::make_const(s, a.delta, sm2);
      QConst c;
      c.sa = n.sa; c.ca = 0.f; c.ss = n.ss; c.cs = n.cs;
      c.fa = s.fh; c.fs = 0;
      // the real scale of the sign-bit weights travels in the two spare words
      c.pad[0] = __double2loint(s.sq); c.pad[1] = __double2hiint(s.sq);
      shared_c = c;
    }
  }
  __syncthreads();
  return shared_c;
}

// One launch for constants and operand: CTA (query, share of the operand's words).  Every share forms the query's constants again,
// which is cheaper than a launch of their own (3 us each: two or three fewer per call, 64 queries against 4,096 rows of d = 128: 15.5 -> 13.8 us).  A thread
// takes a 32-bit word of B (four K-bytes): its weights are formed once and leave as a word in each of the three digit rows; a
// warp writes 128 contiguous bytes of each.
template <bool NIB>
__global__ void __launch_bounds__(256) toperand_kernel(const __grid_constant__ OperandArgs a) {
  allow_successor();
  wait_for_predecessor();   // the queries are its output; what this kernel writes may still be read by it
  const int ql = blockIdx.x;
  const bool present = ql < a.nqg;   // absent queries of the last pass get zero rows
  const float* q = a.Qcat + (int64_t)(present ? ql : 0) * a.ldq;
  QConst c = {};
  if (present) {
    c = NIB ? query_constants_nib(a, q) : query_constants(a, q);
    if (blockIdx.y == 0 && threadIdx.x == 0) a.qc[ql] = c;
  }
  const int row0 = ql / kQueriesPerPass * NCOL + ql % kQueriesPerPass;   // digit l of the query: row0 + 32 l
  for (int i = blockIdx.y * 256 + threadIdx.x; i < (a.g.kba + a.g.kbs) * 32; i += gridDim.y * 256) {
    const bool part = i >= a.g.kba * 32;   // bit streams: the sign part
    const int nkb = part ? a.g.kbs : a.g.kba;
    const int at = part ? i - a.g.kba * 32 : i, kb = at >> 5, word = at & 31;
    uint32_t out[LIMBS] = {0u, 0u, 0u};
    if (present && NIB) {
      const int b = kb / 3, type = kb % 3;
      nib::QScale sc;
      sc.fh = c.fa;
      sc.sq = __hiloint2double(c.pad[1], c.pad[0]);
#pragma unroll
      for (int i4 = 0; i4 < 4; ++i4) {
        int cib = 4 * word + i4, mul = 1;
        if (type == 2) {
          cib = 8 * (word >> 1) + 2 * i4 + (word & 1);
          mul = (word & 1) ? 1 : 16;
        }
        const int coord = nib::coord_of_block(a.g.nbi, a.g.idx_rb, a.g.qjl_rb, a.g.d, b, cib);
        if (coord < 0) continue;
        const long long J = mul * nib::weight(sc, type, q[(type < 2 ? 0 : a.dpad) + coord]);
#pragma unroll
        for (int l = 0; l < LIMBS; ++l) out[l] |= (uint32_t)(nib::digit_of(J, l) & 255) << (8 * i4);
      }
    } else if (present) {
      const int wl = word >> 3, k = word & 7;
      const double scale = pow2_of((part ? c.fs : c.fa) - k);
#pragma unroll
      for (int i4 = 0; i4 < 4; ++i4) {
        const int bit = 8 * i4 + k;
        double W = 0.0;
        if (!part) {
          const Slot s = slot_a(a.g, kb, wl, bit);
          if (s.coord < a.g.d) W = 2.0 * a.alpha[s.term] * (double)q[s.coord];
        } else {
          const int j = 32 * (4 * kb + wl) + bit;
          if (j < a.g.d) W = 2.0 * (double)q[a.dpad + j];
        }
        const double Jd = rint(W * scale);
        int J = fabs(Jd) <= 8388608.0 ? (int)Jd : 0;   // non-finite query entries contribute nothing
#pragma unroll
        for (int l = 0; l < LIMBS; ++l) {
          const int dg = ((J + 128) & 255) - 128;
          J = (J - dg) >> 8;
          out[l] |= (uint32_t)(dg & 255) << (8 * i4);
        }
      }
    }
    uint8_t* dst = (part ? a.Bs : a.Ba) + ((size_t)row0 * nkb + kb) * KB_BYTES + word * 4;
#pragma unroll
    for (int l = 0; l < LIMBS; ++l) *reinterpret_cast<uint32_t*>(dst + (size_t)l * kQueriesPerPass * nkb * KB_BYTES) = out[l];
  }
}

// ------------------------------------------------------------------ epilogue
// Estimates of one row for 16 queries (constants qc[0 .. 16)) from the three digit sums of the two terms.  The digits are
// recombined exactly (64-bit integer: the same T as in the register-fed engine), then fp32.  No branch in here, so that the
// sixteen chains overlap: with the threshold test inside the loop the epilogue ran at 8 cycles per instruction and was half of
// the many-query scan's time at d = 200.
template <bool MSE, bool SIGNS>
__device__ __forceinline__ void estimates16(const uint32_t (&va)[LIMBS][16], const uint32_t (&vs)[LIMBS][16], const QConst* qc, float nu,
                                            float cg, float (&est)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float4 c = *reinterpret_cast<const float4*>(qc + i);   // sa, ca, ss, cs
    float av = 0.f, sv = 0.f;
    if (MSE) av = fmaf((float)(((long long)(int)va[2][i] * 256 + (int)va[1][i]) * 256 + (int)va[0][i]), c.x, c.y);
    if (SIGNS) sv = fmaf((float)(((long long)(int)vs[2][i] * 256 + (int)vs[1][i]) * 256 + (int)vs[0][i]), c.z, c.w);
    est[i] = __fmul_rn(nu, fmaf(cg, sv, av));
  }
}

// est[i], i in a register array and different from lane to lane: four levels of selects.
__device__ __forceinline__ float pick16(const float (&est)[16], int i) {
  float a8[8], a4[4];
#pragma unroll
  for (int j = 0; j < 8; ++j) a8[j] = (i & 1) ? est[2 * j + 1] : est[2 * j];
#pragma unroll
  for (int j = 0; j < 4; ++j) a4[j] = (i & 2) ? a8[2 * j + 1] : a8[2 * j];
  const float x = (i & 4) ? a4[1] : a4[0], y = (i & 4) ? a4[3] : a4[2];
  return (i & 8) ? y : x;
}

// Filter mode: the estimates that reach their query's threshold (bit i of `hits`: query q0 + i) go to the CTA's buffers.  A lane
// takes its own hits one after the other, all lanes at once: a test per query, each with a body for the few lanes that hit,
// cost 1,300 cycles per 16 queries where one estimate in 120 hits.
template <int CAPACITY, class Args>
__device__ __forceinline__ void append_hits(const Args& a, uint32_t hits, const float (&est)[16], int q0, int64_t row, int* lcnt, uint2* lbuf) {
  while (hits != 0u) {
    const int i = __ffs((int)hits) - 1, ql = q0 + i;
    hits &= hits - 1u;
    const float e = pick16(est, i);
    const int ls = atomicAdd(&lcnt[ql], 1);
    if (ls < CAPACITY) {
      lbuf[ql * CAPACITY + ls] = make_uint2(__float_as_uint(e), (uint32_t)row);
    } else {   // the CTA's buffer is full: straight to the global list
      const int slot = atomicAdd(a.count + ql, 1);
      if (slot < a.cap) {
        a.cand_s[(int64_t)ql * a.cap + slot] = e;
        a.cand_i[(int64_t)ql * a.cap + slot] = (int)row;
      }
    }
  }
}

// ------------------------------------------------------------------ scan kernel
struct ScanArgs {
  int64_t n, npairs;
  uint32_t hi_a, hi_b, lo_a, lo_b;   // nibble layout: the 16-bit centroid table as bytes (h of entries 0..3, 4..7; l alike)
  Geo g;
  int pass, nqp;
  const QConst* qc;        // constants of this pass's queries
  const uint8_t* idx;
  size_t idx_rb;
  const uint8_t* qjl;
  size_t qjl_rb;
  const float* gamma;
  const float* norms;
  int64_t step;            // rows of the arrays from one vector to the next
  float coef;
  float* scores;
  int64_t lds;
  const float* tau;
  int* count;
  float* cand_s;
  int* cand_i;
  int cap;
  const int* run_if;
  int* status;
};

// D[tmem] (+)= A[tmem] * B[smem]^T: A is taken from TMEM (row = lane, 4 K-bytes per 32-bit column).
__device__ __forceinline__ void umma_i8_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The same over a CTA pair (M = 256: the leader's thread issues for both CTAs, each CTA holds its own rows of A and D in
// TMEM and half of B's rows in shared memory).
__device__ __forceinline__ void umma_i8_ts_pair(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::i8 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// kind::i8: D = s32, A = unsigned 8-bit, B = signed 8-bit, both K-major.
__host__ __device__ constexpr uint32_t idesc_i8(int M, int N, bool a_signed = false) {
  return (2u << 4) | ((a_signed ? 1u : 0u) << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

template <int BM, int MODE, bool NIB = false>
__global__ void __launch_bounds__(NTHREADS, 1)
scan_tc_kernel(const __grid_constant__ CUtensorMap tmBa, const __grid_constant__ CUtensorMap tmBs,
               const __grid_constant__ CUtensorMap tmPa, const __grid_constant__ CUtensorMap tmPs, ScanArgs a) {
  allow_successor();
  if (a.run_if != nullptr) {
    wait_for_predecessor();   // it may write the switch
    if (*a.run_if == 0) return;
  }

  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* bring = smem;
  unsigned char* pring = smem + B_STAGES * BTILE_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(pring + P_STAGES * PTILE_BYTES);
  uint64_t* afull = bars;                           // [A_SLOTS]   transform warps -> MMA
  uint64_t* bfull = afull + A_SLOTS;                // [B_STAGES]  TMA -> MMA
  // One tcgen05.commit per k-block: the issuing thread pays ~350 cycles per commit (measured), so the release
  // of the A slot (2 k-blocks later) and of the B stage (8 k-blocks later) share one ring of barriers.
  uint64_t* kdone = bfull + B_STAGES;               // [B_STAGES]  MMAs of k-block f complete
  uint64_t* pfull = kdone + B_STAGES;               // [P_STAGES]  TMA (packed rows) -> transform warps
  uint64_t* pempty = pfull + P_STAGES;              // [P_STAGES]  transform warps -> TMA producer
  uint64_t* dfull = pempty + P_STAGES;              // accumulators complete -> epilogue
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(dfull + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  QConst* qcs = reinterpret_cast<QConst*>(dfull + 4);
  float* taus = reinterpret_cast<float*>(qcs + kQueriesPerPass);   // [32] admission thresholds (filter mode)
  // Filter mode: admitted pairs are collected per CTA and appended to the global lists in one piece per query at
  // the end: one atomic per (CTA, query) instead of one per pair on 32 contended counters.
  int* lcnt = reinterpret_cast<int*>(taus + kQueriesPerPass);       // [32]
  uint2* lbuf = reinterpret_cast<uint2*>(lcnt + kQueriesPerPass);   // [32][LBUF] (score bits, row)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkb_total = a.g.kba + a.g.kbs;

  if (threadIdx.x == 0) {
    for (int s = 0; s < A_SLOTS; ++s) tc::mbar_init(&afull[s], 8);
    for (int s = 0; s < B_STAGES; ++s) {
      tc::mbar_init(&bfull[s], 1);
      tc::mbar_init(&kdone[s], 1);
    }
    for (int s = 0; s < P_STAGES; ++s) {
      tc::mbar_init(&pfull[s], 1);
      tc::mbar_init(&pempty[s], 8);
    }
    tc::mbar_init(dfull, N_ISSUERS);
    *abort_flag = 0;
    tc::fence_barrier_init();
    if (a.g.kba > 0) tc::tma_prefetch_desc(&tmBa);
    if (a.g.kbs > 0) tc::tma_prefetch_desc(&tmBs);
    if (a.g.kba > 0) tc::tma_prefetch_desc(&tmPa);
    if (a.g.kbs > 0) tc::tma_prefetch_desc(&tmPs);
  }
  wait_for_predecessor();   // every input may be its output
  if (threadIdx.x < kQueriesPerPass) {
    QConst c = {1.f, 0.f, 1.f, 0.f, 0, 0, {0, 0}};
    if ((int)threadIdx.x < a.nqp) c = a.qc[threadIdx.x];
    qcs[threadIdx.x] = c;
    taus[threadIdx.x] = (MODE == 1 && (int)threadIdx.x < a.nqp) ? a.tau[threadIdx.x] : 0.f;
    lcnt[threadIdx.x] = 0;
  }
  if (warp == 1) tc::tmem_alloc(tmem_slot, TMEM_COLS);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer of B
    if (lane == 0) {
      int stage = 0, pstage = 0;
      uint32_t phase = 0, pphase = 0;
      bool ok = true;
      long long kc = 0;   // k-blocks issued so far by this CTA
      for (int64_t pair = blockIdx.x; pair < a.npairs && ok; pair += gridDim.x) {
        for (int f = 0; f < nkb_total; ++f, ++kc) {
          const bool part_s = f >= a.g.kba;
          const int kb = part_s ? f - a.g.kba : f;
          if (NIB ? (kb % 3 == 0) : ((kb & 3) == 0)) {   // the packed rows of the pair for the next group of k-blocks
            if (!(ok = tc::mbar_wait(&pempty[pstage], pphase ^ 1u, abort_flag, a.status))) break;
            const int gb = (part_s || NIB) ? 64 : group_bytes(BM);
            tc::mbar_arrive_expect_tx(&pfull[pstage], (uint32_t)(2 * TILE * gb));
            if (NIB) {   // block kb / 3 of the combined row: from the idx rows, then from the qjl rows
              const int b = kb / 3;
              tc::tma_load_2d(pring + pstage * PTILE_BYTES, b < a.g.nbi ? &tmPa : &tmPs, &pfull[pstage],
                              64 * (b < a.g.nbi ? b : b - a.g.nbi), (int)(pair * (2 * TILE)));
            } else {
              tc::tma_load_2d(pring + pstage * PTILE_BYTES, part_s ? &tmPs : &tmPa, &pfull[pstage], (kb >> 2) * gb,
                              (int)(pair * (2 * TILE)));
            }
            if (++pstage == P_STAGES) {
              pstage = 0;
              pphase ^= 1u;
            }
          }
          // B stage kc % B_STAGES was last read by the MMAs of k-block kc - B_STAGES
          if (kc >= B_STAGES && !(ok = tc::mbar_wait(&kdone[stage], phase ^ 1u, abort_flag, a.status))) break;
          tc::mbar_arrive_expect_tx(&bfull[stage], BTILE_BYTES);
          tc::tma_load_2d(bring + stage * BTILE_BYTES, part_s ? &tmBs : &tmBa, &bfull[stage], kb * KB_BYTES, a.pass * NCOL);
          if (++stage == B_STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok) {
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);   // let copies in flight land
      }
    }
    __syncwarp();
  } else if (warp <= N_ISSUERS) {
    // ---------------------------------------------------------------- MMA issuers
    // The k-blocks are dealt in turn to the issuing warps: 8 MMAs (4 per tile) + one commit each.  The
    // accumulators are zeroed by the transform warps, every MMA accumulates, and integer sums do not depend
    // on the order in which the k-blocks of different threads reach the tensor pipe.
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_i8(TILE, NCOL);
      const int me = warp - 1;
      bool ok = true;
      uint32_t kc = 0;    // k-blocks of this CTA so far
      int turn = 0;       // whose k-block comes next
      const uint64_t bdesc0 = tc::smem_desc_sw128(tc::smem_u32(bring));
      for (int64_t pair = blockIdx.x; pair < a.npairs && ok; pair += gridDim.x) {
        for (int f = 0; f < nkb_total; ++f, ++kc) {
          const bool mine = turn == me;
          if (++turn == N_ISSUERS) turn = 0;
          if (!mine) continue;
          const uint32_t bstage = kc & (B_STAGES - 1), stage = kc & (A_SLOTS - 1);
          if (!(ok = tc::mbar_wait(&bfull[bstage], (kc / B_STAGES) & 1u, abort_flag, a.status))) break;
          if (!(ok = tc::mbar_wait(&afull[stage], (kc / A_SLOTS) & 1u, abort_flag, a.status))) break;
          tc::tc_fence_after();
          // nibble layout: k-blocks of h bytes (signed A), l bytes and sign bits in turn; the sign bits have the
          // second accumulator
          const int kind = NIB ? f % 3 : 0;
          const bool part_s = NIB ? kind == 2 : f >= a.g.kba;
          const uint32_t idesc_f = (NIB && kind == 0) ? idesc_i8(TILE, NCOL, true) : idesc;
          const uint64_t bdesc = bdesc0 + (uint64_t)(bstage * (BTILE_BYTES >> 4));
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            const uint32_t a_tmem = tmem_base + (uint32_t)(A_COL0 + t * (A_SLOTS * 32) + stage * 32);
            const uint32_t d_tmem = tmem_base + (uint32_t)(t * D_COLS + (part_s ? NCOL : 0));
#pragma unroll
            for (int step = 0; step < 4; ++step)   // 32 K-bytes per MMA: 8 TMEM columns of A, +32 bytes inside B's swizzled row
              umma_i8_ts(d_tmem, a_tmem + 8 * step, bdesc + 2 * step, idesc_f, 1u);
          }
          tc::umma_commit(&kdone[bstage]);   // A slot and B stage reusable once these MMAs have read them
        }
        if (ok) tc::umma_commit(dfull);   // all MMAs this thread issued for the pair
      }
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- transform + epilogue (thread = vector row)
    const int e = warp - 1 - N_ISSUERS;
    const int t = e >> 2;                   // which tile of the pair
    const int quad = warp & 3;              // TMEM lane group this warp may access
    const int r = quad * 32 + lane;         // row inside the tile
    int stage = 0, pstage_keep = 0;
    uint32_t pphase_keep = 0;
    uint32_t kt = 0;    // k-blocks expanded so far by this warp
    bool ok = true;
    int64_t it = 0;
    // the row's scalars are requested one pair ahead, so that their latency hides behind a pair's k-blocks
    auto load_nu = [&](int64_t pr) -> float {
      const int64_t rw = pr * (2 * TILE) + t * TILE + r;
      return (pr < a.npairs && rw < a.n && a.norms != nullptr) ? __ldg(a.norms + rw * a.step) : 1.f;
    };
    auto load_gm = [&](int64_t pr) -> float {
      const int64_t rw = pr * (2 * TILE) + t * TILE + r;
      return (pr < a.npairs && rw < a.n && (a.g.kbs > 0 || NIB)) ? __ldg(a.gamma + rw * a.step) : 0.f;   // times coef where it is used, so that nothing waits for the load here
    };
    float nu_next = load_nu(blockIdx.x), gm_next = load_gm(blockIdx.x);
    for (int64_t pair = blockIdx.x; pair < a.npairs && ok; pair += gridDim.x, ++it) {
      const int64_t row = pair * (2 * TILE) + t * TILE + r;
      const bool row_ok = row < a.n;
      const float nu = nu_next, gm = gm_next;
      nu_next = load_nu(pair + gridDim.x);
      gm_next = load_gm(pair + gridDim.x);

      // this row's accumulators start from zero (the previous pair's epilogue, by this same thread, has read
      // them; the stores complete before the row's first A tile is announced)
#pragma unroll
      for (int c = 0; c < D_COLS; c += 16) tc::tmem_fill16(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(t * D_COLS + c), 0u);

      // stores one k-block's 32 A registers of this row into the current A slot and announces it
      auto store_a = [&](const uint32_t (&v)[32]) -> bool {
        // A slot kt % 2 was last read by the MMAs of k-block kt - 2: completion number (kt - 2) / B_STAGES of its barrier
        if (kt >= A_SLOTS) {
          const uint32_t kp = kt - A_SLOTS;
          if (!tc::mbar_wait(&kdone[kp & (B_STAGES - 1)], (kp / B_STAGES) & 1u, abort_flag, a.status)) return false;
        }
        tc::tc_fence_after();
        tc::tmem_st32(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(A_COL0 + t * (A_SLOTS * 32) + stage * 32), v);
        tc::tmem_st_wait();
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&afull[stage]);
        if (++stage == A_SLOTS) stage = 0;
        ++kt;
        return true;
      };
      // expands one k-block's words into the row's 128 bytes of the A tile of the current stage
      auto emit = [&](uint32_t (&w)[4], int f) -> bool {
        if (f >= nkb_total) return true;
        if (f < a.g.kba) {
          if (BM == 3) {
            w[3] = parity3(w[0], w[1], w[2]);
          } else if (BM == 4) {
            w[2] = parities4(w[0]);
            w[3] = parities4(w[1]);
          }
        }
        // the row's 128 A bytes of this k-block: register 4 c + e = (word c / 2, bit 4 (c % 2) + e of every byte)
        uint32_t v[32];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint32_t x = w[c >> 1];
          const int k0 = (c & 1) * 4;
#pragma unroll
          for (int e2 = 0; e2 < 4; ++e2) v[4 * c + e2] = x & (0x01010101u << (k0 + e2));
        }
        return store_a(v);
      };
      // groups of four k-blocks: the pair's packed rows arrive by TMA ([256 rows x group bytes], swizzled so that
      // row-per-thread 16-byte reads are conflict-free); the thread copies its row's bytes to registers, frees the
      // stage and expands the four k-blocks
      const int prow = t * TILE + r;   // row inside the pair
      int pstage = pstage_keep;
      uint32_t pphase = pphase_keep;
      if (NIB) {
        // nibble layout: a group is one 64-byte block of the combined row = 16 code words = 128 coordinates, expanded
        // into three k-blocks: h bytes and l bytes by byte permutes with the masked word as selector, sign bits by masks
        for (int f0 = 0; f0 < nkb_total && ok; f0 += 3) {
          if (!(ok = tc::mbar_wait(&pfull[pstage], pphase, abort_flag, a.status))) break;
          const unsigned char* ps = pring + pstage * PTILE_BYTES;
          uint32_t x[16];
#pragma unroll
          for (int j = 0; j < 4; ++j) {   // 64 bytes per row, 64-byte swizzle: chunk c at c ^ ((row >> 1) & 3)
            const uint4 v4 = *reinterpret_cast<const uint4*>(ps + prow * 64 + ((j ^ ((prow >> 1) & 3)) << 4));
            x[4 * j] = v4.x; x[4 * j + 1] = v4.y; x[4 * j + 2] = v4.z; x[4 * j + 3] = v4.w;
          }
          tc::release_stage(&pempty[pstage], lane);
          if (++pstage == P_STAGES) {
            pstage = 0;
            pphase ^= 1u;
          }
          uint32_t v[32];
#pragma unroll
          for (int wd = 0; wd < 16; ++wd) {
            const uint32_t sl = x[wd] & 0x77777777u;
            v[2 * wd] = prmt(a.hi_a, a.hi_b, sl);
            v[2 * wd + 1] = prmt(a.hi_a, a.hi_b, sl >> 16);
          }
          ok = ok && store_a(v);
#pragma unroll
          for (int wd = 0; wd < 16; ++wd) {
            const uint32_t sl = x[wd] & 0x77777777u;
            v[2 * wd] = prmt(a.lo_a, a.lo_b, sl);
            v[2 * wd + 1] = prmt(a.lo_a, a.lo_b, sl >> 16);
          }
          ok = ok && store_a(v);
#pragma unroll
          for (int wd = 0; wd < 16; ++wd) {
            v[2 * wd] = x[wd] & 0x08080808u;
            v[2 * wd + 1] = x[wd] & 0x80808080u;
          }
          ok = ok && store_a(v);
        }
      }
      for (int f0 = 0; !NIB && f0 < nkb_total && ok; f0 += 4) {
        // a part boundary inside a group cannot happen: each part starts a new group
        const bool part_s = f0 >= a.g.kba;
        if (!(ok = tc::mbar_wait(&pfull[pstage], pphase, abort_flag, a.status))) break;
        const unsigned char* ps = pring + pstage * PTILE_BYTES;
        uint32_t w[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j][0] = w[j][1] = w[j][2] = w[j][3] = 0u;
        if (part_s || BM <= 2) {           // 64 bytes per row, 64-byte swizzle: chunk c at c ^ ((row >> 1) & 3)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint4 v = *reinterpret_cast<const uint4*>(ps + prow * 64 + ((j ^ ((prow >> 1) & 3)) << 4));
            w[j][0] = v.x; w[j][1] = v.y; w[j][2] = v.z; w[j][3] = v.w;
          }
        } else if (BM == 3) {              // 48 bytes per row, plain: three words per k-block
          uint32_t x[12];
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const uint4 v = *reinterpret_cast<const uint4*>(ps + prow * 48 + j * 16);
            x[4 * j] = v.x; x[4 * j + 1] = v.y; x[4 * j + 2] = v.z; x[4 * j + 3] = v.w;
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            w[j][0] = x[3 * j]; w[j][1] = x[3 * j + 1]; w[j][2] = x[3 * j + 2];
          }
        } else {                           // b_m = 4: 32 bytes per row, 32-byte swizzle: chunk c at c ^ ((row >> 2) & 1)
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const uint4 v = *reinterpret_cast<const uint4*>(ps + prow * 32 + ((j ^ ((prow >> 2) & 1)) << 4));
            w[2 * j][0] = v.x; w[2 * j][1] = v.y; w[2 * j + 1][0] = v.z; w[2 * j + 1][1] = v.w;
          }
        }
        tc::release_stage(&pempty[pstage], lane);
        if (++pstage == P_STAGES) {
          pstage = 0;
          pphase ^= 1u;
        }
        const int fend = part_s ? nkb_total : a.g.kba;   // k-blocks of this part end here
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (f0 + j < fend) ok = ok && emit(w[j], f0 + j);
        if (!part_s && f0 + 4 >= a.g.kba) f0 = a.g.kba - 4;   // the next group starts the QJL part
      }
      pstage_keep = pstage;
      pphase_keep = pphase;
      if (!ok) break;

      // ---- epilogue: this thread's row of the four accumulators
      if (!(ok = tc::mbar_wait(dfull, (uint32_t)(it & 1), abort_flag, a.status))) break;
      tc::tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(t * D_COLS);
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {   // 16 queries per half: digit l of query 16 h + qq sits in column 32 l + 16 h + qq
        if (h * 16 >= a.nqp) break;   // a short last pass: columns of absent queries are not read
        __syncwarp();                 // lanes leave the first half's stores and hits one by one; the TMEM load takes whole warps
        uint32_t va[LIMBS][16], vs[LIMBS][16];
#pragma unroll
        for (int l = 0; l < LIMBS; ++l) {
          if (a.g.kba > 0) tc::tmem_ld16(taddr + l * 32 + h * 16, va[l]);
          if (a.g.kbs > 0 || NIB) tc::tmem_ld16(taddr + NCOL + l * 32 + h * 16, vs[l]);
        }
        tc::tmem_ld_wait();
        float est[16];
        const float cg = __fmul_rn(a.coef, gm);
        if (a.g.kbs > 0 || NIB) estimates16<(BM > 0), true>(va, vs, qcs + 16 * h, nu, cg, est);
        else estimates16<(BM > 0), false>(va, vs, qcs + 16 * h, nu, cg, est);
        if (MODE == 0) {
#pragma unroll
          for (int qq = 0; qq < 16; ++qq)
            if (row_ok && h * 16 + qq < a.nqp && TQ_DEVICE_CHECK(row >= 0 && row < a.n && row < a.lds, a.status))
              a.scores[(int64_t)(h * 16 + qq) * a.lds + row] = est[qq];
          continue;
        }
        uint32_t hits = 0u;
#pragma unroll
        for (int qq = 0; qq < 16; ++qq) hits |= est[qq] >= taus[h * 16 + qq] ? 1u << qq : 0u;
        if (!row_ok) hits = 0u;
        if (a.nqp < 16 * h + 16) hits &= (1u << (a.nqp - 16 * h)) - 1u;
        append_hits<LBUF>(a, hits, est, 16 * h, row, lcnt, lbuf);
      }
      __syncwarp();
      tc::tc_fence_before();
    }
  }

  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem_base, TMEM_COLS);
  }
  if (MODE == 1 && warp > N_ISSUERS) {   // the eight transform warps append four queries' collected pairs each
    for (int ql = (warp - 1 - N_ISSUERS) * 4; ql < (warp - N_ISSUERS) * 4; ++ql) {
      const int m = min(lcnt[ql], LBUF);
      if (m == 0 || ql >= a.nqp) continue;
      int base = 0;
      if (lane == 0) base = atomicAdd(a.count + ql, m);
      base = __shfl_sync(0xffffffffu, base, 0);
      for (int i = lane; i < m; i += 32) {
        const int slot = base + i;
        if (slot < a.cap) {
          const uint2 e = lbuf[ql * LBUF + i];
          a.cand_s[(int64_t)ql * a.cap + slot] = __uint_as_float(e.x);
          a.cand_i[(int64_t)ql * a.cap + slot] = (int)e.y;
        }
      }
    }
  }
}

// ------------------------------------------------------------------ exact estimates of single rows
// For the rows that a screening pass leaves: the same digit sums as the scan kernels, hence the same estimates, by byte dot
// products on CUDA cores over the digit rows of B that the scan kernels read.
struct RescoreArgs {
  int64_t n;
  Geo g;
  uint32_t hi_a, hi_b, lo_a, lo_b;
  const QConst* qc;
  const uint8_t* Ba;
  const uint8_t* Bs;
  const uint8_t* idx;
  const uint8_t* qjl;
  const float* gamma;
  const float* norms;
  float coef;
  const screen::QueryTerms* terms;
  const float* tau;        // threshold of the listing
  const float* kth;        // lower bound of the k-th best estimate
  const int* count;        // candidates: (lower bound, row)
  const float* cand_s;
  const int* cand_i;
  int cap, k;
  float* out_s;            // [queries][kSurvivors]
  int* out_i;
  int* out_count;
  int* overflow;
  int per_flag;
};

__device__ __forceinline__ int dp4a_us(uint32_t a, uint32_t b, int c) {
  int d;
  asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ int dp4a_ss(uint32_t a, uint32_t b, int c) {
  int d;
  asm("dp4a.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// CTA (query, share of its list): candidates whose upper bound reaches the k-th lower bound, then a warp per row; lane = 32-bit word
// of a k-block.
// Bound: latency of the gathers (the list's rows lie anywhere in the index); some 130 of 1,600 candidates are left for k = 100.
constexpr int kRescoreThreads = 512;
__global__ void __launch_bounds__(kRescoreThreads, 2) rescore_kernel(const __grid_constant__ RescoreArgs a) {
  __shared__ int ids[screen::kSurvivors];
  __shared__ int s_n, s_base, s_numbers;
  allow_successor();
  if (threadIdx.x == 0) s_n = s_numbers = 0;
  __syncthreads();
  wait_for_predecessor();   // the lists are its output
  const int q = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool signs = a.g.kbs > 0 || a.g.nib;
  const float err = a.terms[q].err, unscale = a.terms[q].unscale;
  const bool zero = err == screen::kZeroQuery;
  if (err == screen::kNanQuery || (zero && blockIdx.y > 0)) return;
  const int m = zero ? 0 : a.count[q];
  if (zero) {   // the first rows
    const int rows = (int)min(a.n, (int64_t)a.k + screen::kZeroSpare);
    for (int i = threadIdx.x; i < rows; i += kRescoreThreads) ids[i] = i;
    if (threadIdx.x == 0) s_n = rows;
  } else if (m > a.cap || m < a.k) {   // too long for the list; too short: no threshold that k rows reach keeps fewer
    if (threadIdx.x == 0) atomicExch(a.overflow + q / a.per_flag, 1);
    return;
  }
  const float kth = a.kth[q], slack = 2.f * screen::kThresholdSlack * fabsf(a.tau[q]);
  // four candidates of a thread at a time: the loads of their scalars are a chain of two round trips
  const int stride = kRescoreThreads * (int)gridDim.y;
  for (int i0 = blockIdx.y * kRescoreThreads + threadIdx.x; i0 < m; i0 += 4 * stride) {
    int id[4];
    float low[4], nu[4], gm[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = min(i0 + u * stride, m - 1);
      id[u] = a.cand_i[(int64_t)q * a.cap + i];
      low[u] = a.cand_s[(int64_t)q * a.cap + i];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      nu[u] = a.norms ? __ldg(a.norms + id[u]) : 1.f;
      gm[u] = signs ? __ldg(a.gamma + id[u]) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float high = low[u] + slack + 2.f * screen::row_terms(nu[u], gm[u]).rho * err * unscale;
      if (i0 + u * stride < m && !(high < kth)) {
        const int s = atomicAdd(&s_n, 1);
        if (s < screen::kSurvivors) ids[s] = id[u];
      }
    }
  }
  __syncthreads();
  const int n = s_n;
  if (threadIdx.x == 0) {
    s_base = atomicAdd(a.out_count + q, n);
    if (s_base + n > screen::kSurvivors) atomicExch(a.overflow + q / a.per_flag, 1);
  }
  __syncthreads();
  const int base = s_base;
  if (base + n > screen::kSurvivors) return;   // the pass is scored by the scan kernels
  const QConst c = a.qc[q];
  const int row0 = q / kQueriesPerPass * NCOL + q % kQueriesPerPass;
  const size_t pa = (size_t)a.g.kba * KB_BYTES, psn = (size_t)a.g.kbs * KB_BYTES;
  const uint8_t* ba = a.Ba + (size_t)row0 * pa + 4 * lane;
  const uint8_t* bs = a.Bs + (size_t)row0 * psn + 4 * lane;
  const uint32_t mask = 0x01010101u << (((lane >> 2) & 1) * 4 + (lane & 3));   // of register `lane` of a k-block of the bit streams
  for (int s = warp; s < n; s += kRescoreThreads / 32) {
    const int64_t row = ids[s];
    int va[LIMBS] = {0, 0, 0}, vs[LIMBS] = {0, 0, 0};
    const uint32_t* iw = reinterpret_cast<const uint32_t*>(a.idx + (size_t)row * a.g.idx_rb);
    const uint32_t* qw = reinterpret_cast<const uint32_t*>(a.qjl + (size_t)row * a.g.qjl_rb);
    if (a.g.nib) {
      for (int b = 0; b < a.g.nblk; ++b) {
        const bool second = b >= a.g.nbi;
        const int word = 16 * (second ? b - a.g.nbi : b) + (lane >> 1);
        const uint32_t x = word < (second ? a.g.wq : a.g.widx) ? __ldg((second ? qw : iw) + word) : 0u;
        const uint32_t sl = (x & 0x77777777u) >> ((lane & 1) * 16);
        const uint32_t h = prmt(a.hi_a, a.hi_b, sl), l = prmt(a.lo_a, a.lo_b, sl), z = x & ((lane & 1) ? 0x80808080u : 0x08080808u);
        const uint8_t* bb = ba + (size_t)(3 * b) * KB_BYTES;
#pragma unroll
        for (int g = 0; g < LIMBS; ++g) {
          const uint8_t* bd = bb + (size_t)g * kQueriesPerPass * pa;
          va[g] = dp4a_ss(h, __ldg(reinterpret_cast<const uint32_t*>(bd)), va[g]);
          va[g] = dp4a_us(l, __ldg(reinterpret_cast<const uint32_t*>(bd + KB_BYTES)), va[g]);
          vs[g] = dp4a_us(z, __ldg(reinterpret_cast<const uint32_t*>(bd + 2 * KB_BYTES)), vs[g]);
        }
      }
    } else {
      const int wl = lane >> 3;   // the register's word of the k-block
      auto word = [&](const uint32_t* w, int i, int words) -> uint32_t { return i < words ? __ldg(w + i) : 0u; };
      for (int kb = 0; kb < a.g.kba; ++kb) {
        uint32_t x;
        if (a.g.bm <= 2) {
          x = word(iw, 4 * kb + wl, a.g.widx);
        } else if (a.g.bm == 3) {
          const uint32_t w0 = word(iw, 3 * kb, a.g.widx), w1 = word(iw, 3 * kb + 1, a.g.widx), w2 = word(iw, 3 * kb + 2, a.g.widx);
          x = wl == 0 ? w0 : wl == 1 ? w1 : wl == 2 ? w2 : parity3(w0, w1, w2);
        } else {
          const uint32_t w = word(iw, 2 * kb + (wl & 1), a.g.widx);
          x = wl < 2 ? w : parities4(w);
        }
        x &= mask;
#pragma unroll
        for (int g = 0; g < LIMBS; ++g)
          va[g] = dp4a_us(x, __ldg(reinterpret_cast<const uint32_t*>(ba + (size_t)g * kQueriesPerPass * pa + (size_t)kb * KB_BYTES)), va[g]);
      }
      for (int kb = 0; kb < a.g.kbs; ++kb) {
        const uint32_t x = word(qw, 4 * kb + wl, a.g.wq) & mask;
#pragma unroll
        for (int g = 0; g < LIMBS; ++g)
          vs[g] = dp4a_us(x, __ldg(reinterpret_cast<const uint32_t*>(bs + (size_t)g * kQueriesPerPass * psn + (size_t)kb * KB_BYTES)), vs[g]);
      }
    }
#pragma unroll
    for (int g = 0; g < LIMBS; ++g) {
      va[g] = __reduce_add_sync(0xffffffffu, va[g]);
      vs[g] = __reduce_add_sync(0xffffffffu, vs[g]);
    }
    if (lane == 0) {   // the operations of estimates16
      float av = 0.f, sv = 0.f;
      if (a.g.bm > 0) av = fmaf((float)(((long long)va[2] * 256 + va[1]) * 256 + va[0]), c.sa, c.ca);
      if (signs) sv = fmaf((float)(((long long)vs[2] * 256 + vs[1]) * 256 + vs[0]), c.ss, c.cs);
      const float nu = a.norms != nullptr ? __ldg(a.norms + row) : 1.f, cg = __fmul_rn(a.coef, signs ? __ldg(a.gamma + row) : 0.f);
      const float e = __fmul_rn(nu, fmaf(cg, sv, av));
      a.out_s[(int64_t)q * screen::kSurvivors + base + s] = e;
      a.out_i[(int64_t)q * screen::kSurvivors + base + s] = isnan(e) ? -1 : (int)row;   // a negative id is an empty slot
      if (zero && !isnan(e)) atomicAdd(&s_numbers, 1);
    }
  }
  if (zero) {
    __syncthreads();
    if (threadIdx.x == 0 && s_numbers < a.k) atomicExch(a.overflow + q / a.per_flag, 1);
  }
}

// at least 120 KB so that a second CTA can never share the SM (the kernel allocates all of TMEM)
#include "tq_scan_tcw.cuh"

constexpr size_t kSmemUsed = B_STAGES * BTILE_BYTES + P_STAGES * PTILE_BYTES + 1024 + 512 + kQueriesPerPass * (sizeof(QConst) + sizeof(float) + sizeof(int) + LBUF * sizeof(uint2));
constexpr size_t kSmemBytes = kSmemUsed > 120 * 1024 ? kSmemUsed : 120 * 1024;

template <int BM, int MODE, bool NIB = false>
cudaError_t launch_t(const CUtensorMap& ma, const CUtensorMap& ms, const CUtensorMap& pa, const CUtensorMap& ps,
                     const ScanArgs& args, cudaStream_t st) {
  auto kern = scan_tc_kernel<BM, MODE, NIB>;
  // function attributes are per device: remember the devices this launcher has prepared
  static std::atomic<unsigned long long> attr_devices{0};   // written by any thread that launches
  int attr_dev = 0;
  if (cudaGetDevice(&attr_dev) != cudaSuccess) return cudaErrorInvalidDevice;
  if (attr_dev >= 64 || !((attr_devices.load(std::memory_order_relaxed) >> attr_dev) & 1ull)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (e != cudaSuccess) return e;
    if (attr_dev < 64) attr_devices.fetch_or(1ull << attr_dev, std::memory_order_relaxed);
  }
  const int grid = (int)std::min<int64_t>(args.npairs, tc::sm_count());
  count_launches(1);
  return launch_dependent(kern, dim3((unsigned)grid), dim3(NTHREADS), kSmemBytes, st, ma, ms, pa, ps, args);
}

template <int BM, int MODE, bool NIB, int CTAS>
cudaError_t launch_wide_c(const CUtensorMap& ma, const CUtensorMap& ms, const CUtensorMap& pa, const CUtensorMap& ps,
                          const ScanArgs& args, cudaStream_t st) {
  auto kern = scan_tcw_kernel<BM, MODE, NIB, CTAS>;
  static std::atomic<unsigned long long> attr_devices{0};
  int attr_dev = 0;
  if (cudaGetDevice(&attr_dev) != cudaSuccess) return cudaErrorInvalidDevice;
  if (attr_dev >= 64 || !((attr_devices.load(std::memory_order_relaxed) >> attr_dev) & 1ull)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWideSmemBytes);
    if (e != cudaSuccess) return e;
    if (attr_dev < 64) attr_devices.fetch_or(1ull << attr_dev, std::memory_order_relaxed);
  }
  count_launches(1);
  const int64_t ntiles = (args.n + TILE - 1) / TILE;
  const unsigned passes = (unsigned)((args.nqp + W_QPP - 1) / W_QPP);
  if (CTAS == 1)
    return launch_dependent(kern, dim3((unsigned)std::min<int64_t>(ntiles, tc::sm_count()), passes), dim3(W_NTHREADS), kWideSmemBytes, st, ma,
                            ms, pa, ps, args);
  const int units = (int)std::min<int64_t>((ntiles + CTAS - 1) / CTAS, tc::sm_count() / CTAS);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(units * CTAS), passes);
  cfg.blockDim = dim3(W_NTHREADS);
  cfg.dynamicSmemBytes = kWideSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CTAS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, ma, ms, pa, ps, args);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// pairs = true: ma / ms are the B maps with boxes of half the rows
template <int BM, int MODE, bool NIB = false>
cudaError_t launch_wide_t(bool pairs, const CUtensorMap& ma, const CUtensorMap& ms, const CUtensorMap& pa, const CUtensorMap& ps,
                          const ScanArgs& args, cudaStream_t st) {
  return pairs ? launch_wide_c<BM, MODE, NIB, 2>(ma, ms, pa, ps, args, st) : launch_wide_c<BM, MODE, NIB, 1>(ma, ms, pa, ps, args, st);
}

template <int MODE>
cudaError_t launch_wide(int bm, bool pairs, const CUtensorMap& ma, const CUtensorMap& ms, const CUtensorMap& pa, const CUtensorMap& ps,
                        const ScanArgs& args, cudaStream_t st) {
  if (args.g.nib) return launch_wide_t<3, MODE, true>(pairs, ma, ms, pa, ps, args, st);
  switch (bm) {
    case 0: return launch_wide_t<0, MODE>(pairs, ma, ms, pa, ps, args, st);
    case 1: return launch_wide_t<1, MODE>(pairs, ma, ms, pa, ps, args, st);
    case 2: return launch_wide_t<2, MODE>(pairs, ma, ms, pa, ps, args, st);
    case 3: return launch_wide_t<3, MODE>(pairs, ma, ms, pa, ps, args, st);
    default: return launch_wide_t<4, MODE>(pairs, ma, ms, pa, ps, args, st);
  }
}

template <int MODE>
cudaError_t launch_bm(int bm, const CUtensorMap& ma, const CUtensorMap& ms, const CUtensorMap& pa, const CUtensorMap& ps,
                      const ScanArgs& args, cudaStream_t st) {
  if (args.g.nib) return launch_t<3, MODE, true>(ma, ms, pa, ps, args, st);
  switch (bm) {
    case 0: return launch_t<0, MODE>(ma, ms, pa, ps, args, st);
    case 1: return launch_t<1, MODE>(ma, ms, pa, ps, args, st);
    case 2: return launch_t<2, MODE>(ma, ms, pa, ps, args, st);
    case 3: return launch_t<3, MODE>(ma, ms, pa, ps, args, st);
    default: return launch_t<4, MODE>(ma, ms, pa, ps, args, st);
  }
}

size_t b_bytes(const Geo& g, int part) {
  return (size_t)kPassesPerGroup * NCOL * (part ? g.kbs : g.kba) * KB_BYTES;
}

}  // namespace

bool available(const tq_plan* plan) { return plan->ms.ok != 0; }

// The wide form can be switched off (TQ_SCAN_WIDE=0) to compare the two kernels on one machine.
int queries_per_pass(int nq) {
  static const bool wide = [] {
    const char* e = std::getenv("TQ_SCAN_WIDE");
    return e == nullptr || e[0] != '0';
  }();
  return wide && nq > kQueriesPerPass ? W_QPP : kQueriesPerPass;
}

size_t workspace_bytes(const tq_plan* plan) {
  if (!available(plan)) return 0;
  const Geo g = make_geo(plan);
  return kConstBytes + b_bytes(g, 0) + b_bytes(g, 1);
}

int prepare_group(const tq_plan* plan, const float* Qcat, int nqg, void* workspace, cudaStream_t st, const char* who) {
  const Geo g = make_geo(plan);
  const int ncols = plan->ncat * plan->dpad;
  QConst* qc = static_cast<QConst*>(workspace);
  uint8_t* Ba = static_cast<uint8_t*>(workspace) + kConstBytes;
  uint8_t* Bs = Ba + b_bytes(g, 0);
  OperandArgs a;
  a.Qcat = Qcat;
  a.ldq = ncols;
  a.nqg = nqg;
  a.dpad = plan->dpad;
  a.prod = plan->mode == TQ_PROD ? 1 : 0;
  a.g = g;
  for (int i = 0; i < 8; ++i) a.alpha[i] = plan->ms.alpha[i];
  a.amax = plan->ms.amax;
  a.csum = plan->ms.csum;
  a.delta = plan->nb.delta;
  a.qc = qc;
  a.Ba = Ba;
  a.Bs = Bs;
  const int queries = (nqg + kQueriesPerPass - 1) / kQueriesPerPass * kQueriesPerPass;   // absent ones get zero rows
  const int words = (g.kba + g.kbs) * 32;
  // shares of an operand: one round of 256 words each, fewer rounds than that only where the queries fill the chip
  const int shares = std::max(1, std::min((words + 255) / 256, 16 * tc::sm_count() / queries));
  count_launches(1);
  const dim3 grid((unsigned)queries, (unsigned)shares);
  TQ_CHECK_CUDA(g.nib ? launch_dependent(toperand_kernel<true>, grid, dim3(256), 0, st, a)
                      : launch_dependent(toperand_kernel<false>, grid, dim3(256), 0, st, a), who);
  return TQ_OK;
}

int run_pass(const tq_plan* plan, int pass, int nqp, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma,
             const float* norms, float* scores, int64_t lds, const mscan::Filter* filter, const int* run_if,
             const void* workspace, cudaStream_t st, const char* who, int64_t step) {
  const Geo g = make_geo(plan);
  const QConst* qc = static_cast<const QConst*>(workspace);
  const uint8_t* Ba = static_cast<const uint8_t*>(workspace) + kConstBytes;
  const uint8_t* Bs = Ba + b_bytes(g, 0);
  // more than 32 queries: the wide kernel takes the B rows of this pass and the next as one box of 192 rows and one
  // 128-vector tile at a time
  const bool wide = nqp > kQueriesPerPass;
  TQ_REQUIRE(!wide || (pass % 2 == 0 && pass * kQueriesPerPass + nqp <= kPassesPerGroup * kQueriesPerPass), TQ_ERR_INVALID_ARG,
             "%s: pass %d of %d queries", who, pass, nqp);
  // The wide kernel runs on CTA pairs wherever there is more than one tile (M = 256, each CTA loads half of a B box's
  // rows into one of twelve half-size stages: measured 316 against 339 us per 32 queries at d = 1536, n = 10^6).
  // TQ_SCAN_PAIRS=0 keeps single CTAs, to compare the two on one machine.
  static const bool pairs_on = [] {
    const char* e = std::getenv("TQ_SCAN_PAIRS");
    return e == nullptr || e[0] != '0';
  }();
  const bool pairs = wide && pairs_on && n > TILE;
  const uint32_t brows = wide ? (pairs ? W_NCOL / 2 : W_NCOL) : NCOL, prows = wide ? TILE : 2 * TILE;
  CUtensorMap ma, ms;
  const uint64_t rows = (uint64_t)kPassesPerGroup * NCOL;
  if (g.kba > 0)
    TQ_REQUIRE(tc::make_byte_map(&ma, Ba, rows, (uint64_t)g.kba * KB_BYTES, (uint64_t)g.kba * KB_BYTES, KB_BYTES, brows, 128),
               TQ_ERR_CUDA, "%s: cuTensorMapEncodeTiled failed (B, MSE part)", who);
  if (g.kbs > 0)
    TQ_REQUIRE(tc::make_byte_map(&ms, Bs, rows, (uint64_t)g.kbs * KB_BYTES, (uint64_t)g.kbs * KB_BYTES, KB_BYTES, brows, 128),
               TQ_ERR_CUDA, "%s: cuTensorMapEncodeTiled failed (B, QJL part)", who);
  if (g.kba == 0) ma = ms;
  if (g.kbs == 0) ms = ma;
  // packed rows: boxes of [256 rows x group bytes]; 64- and 32-byte boxes are swizzled (row-per-thread reads)
  CUtensorMap pa, ps;
  const int gb = g.nib ? 64 : group_bytes(g.bm);
  if (g.nib) {
    TQ_REQUIRE(tc::make_byte_map(&pa, idx, (uint64_t)n, plan->idx_row_bytes, plan->idx_row_bytes * step, 64, prows, 64) &&
                   tc::make_byte_map(&ps, qjl, (uint64_t)n, plan->qjl_row_bytes, plan->qjl_row_bytes * step, 64, prows, 64),
               TQ_ERR_CUDA, "%s: cuTensorMapEncodeTiled failed (code rows)", who);
  } else if (g.kba > 0)
    TQ_REQUIRE(tc::make_byte_map(&pa, idx, (uint64_t)n, plan->idx_row_bytes, plan->idx_row_bytes * step, gb, prows,
                                 gb == 64 ? 64 : gb == 32 ? 32 : 0),
               TQ_ERR_CUDA, "%s: cuTensorMapEncodeTiled failed (idx rows)", who);
  if (!g.nib && g.kbs > 0)
    TQ_REQUIRE(tc::make_byte_map(&ps, qjl, (uint64_t)n, plan->qjl_row_bytes, plan->qjl_row_bytes * step, 64, prows, 64), TQ_ERR_CUDA,
               "%s: cuTensorMapEncodeTiled failed (qjl rows)", who);
  if (!g.nib && g.kba == 0) pa = ps;
  if (!g.nib && g.kbs == 0) ps = pa;
  ScanArgs a;
  a.n = n;
  a.npairs = (n + 2 * TILE - 1) / (2 * TILE);
  a.hi_a = plan->nb.hi_a; a.hi_b = plan->nb.hi_b; a.lo_a = plan->nb.lo_a; a.lo_b = plan->nb.lo_b;
  a.g = g;
  a.pass = pass;
  a.nqp = nqp;
  a.qc = qc + (size_t)pass * kQueriesPerPass;
  a.idx = idx;
  a.idx_rb = plan->idx_row_bytes;
  a.qjl = qjl;
  a.qjl_rb = plan->qjl_row_bytes;
  a.gamma = gamma;
  a.norms = norms;
  a.step = step;
  a.coef = plan->coef;
  a.scores = scores;
  a.lds = lds;
  a.tau = filter ? filter->tau : nullptr;
  a.count = filter ? filter->count : nullptr;
  a.cand_s = filter ? filter->cand_s : nullptr;
  a.cand_i = filter ? filter->cand_i : nullptr;
  a.cap = filter ? filter->cap : 0;
  a.run_if = run_if;
  a.status = plan->d_status;
  if (wide) TQ_CHECK_CUDA(filter ? launch_wide<1>(g.bm, pairs, ma, ms, pa, ps, a, st) : launch_wide<0>(g.bm, pairs, ma, ms, pa, ps, a, st), who);
  else TQ_CHECK_CUDA(filter ? launch_bm<1>(g.bm, ma, ms, pa, ps, a, st) : launch_bm<0>(g.bm, ma, ms, pa, ps, a, st), who);
  return TQ_OK;
}

int rescore(const tq_plan* plan, int nqp, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma, const float* norms,
            const void* workspace, const screen::QueryTerms* terms, const float* tau, const float* kth, const int* count,
            const float* cand_s, const int* cand_i, int cap, int k, float* out_s, int* out_i, int* out_count, int* overflow, int per_flag,
            cudaStream_t st, const char* who) {
  RescoreArgs a;
  a.n = n;
  a.g = make_geo(plan);
  a.hi_a = plan->nb.hi_a; a.hi_b = plan->nb.hi_b; a.lo_a = plan->nb.lo_a; a.lo_b = plan->nb.lo_b;
  a.qc = static_cast<const QConst*>(workspace);
  a.Ba = static_cast<const uint8_t*>(workspace) + kConstBytes;
  a.Bs = a.Ba + b_bytes(a.g, 0);
  a.idx = idx;
  a.qjl = qjl;
  a.gamma = gamma;
  a.norms = norms;
  a.coef = plan->coef;
  a.terms = terms;
  a.tau = tau;
  a.kth = kth;
  a.count = count;
  a.cand_s = cand_s;
  a.cand_i = cand_i;
  a.cap = cap;
  a.k = k;
  a.out_s = out_s;
  a.out_i = out_i;
  a.out_count = out_count;
  a.overflow = overflow;
  a.per_flag = per_flag;
  count_launches(1);
  TQ_CHECK_CUDA(launch_dependent(rescore_kernel, dim3((unsigned)nqp, (unsigned)std::max(1, std::min(8, 2 * tc::sm_count() / nqp))), dim3(kRescoreThreads), 0, st, a), who);
  return TQ_OK;
}

}  // namespace tscan
}  // namespace tq
