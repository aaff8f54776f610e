// Tensor-core reconstruction (sm_100a): DeQuant_mse / DeQuant_prod of Algorithms 1 and 2,
//   Xhat = nu (c[idx] Pi + coef gamma z S),   z = +-1 from the sign bits,
// as one tcgen05 GEMM [n, d] = [c[idx] | z] [Pi ; S] whose A operand is expanded from the packed codes in shared memory
// and whose B operand (limbs of Pi^T and S^T, made once per plan) arrives by TMA.
//
// fp32 fidelity on fp16 tensor cores.  A value v is held as hi + lo, two fp16 numbers (11-bit significands, lo signed):
// the pair keeps v to 2^-24 |v|, as fp32 does.  Pi, S and the codebook are scaled by powers of two so that their largest
// entries lie in [2^13, 2^14): the limbs of everything down to 2^-16 of the largest entry are normal numbers, smaller
// ones are exact to 2^-39 of it.  c[idx] Pi takes the three products hi hi + hi lo + lo hi (the dropped lo lo is 2^-24
// relative), z S only two: z is exact.  bf16 limbs (the quantiser's) would keep 17 bits only.
// The tensor cores add into their fp32 accumulator with truncation (measured through a library GEMM: a bias of
// 1.3e-6 of the result after 96 accumulations, 2e-7 after 16), so an accumulator holds a few k-blocks of one of the
// two terms; the worker warps drain it into fp32 registers with round-to-nearest additions while the tensor
// pipe fills the other accumulator.  That is also where gamma, one number per row, multiplies the z S term.
//
// Bound: tensor pipe, 5 MMA passes of 2 n d^2 flops (3 for TQ_MSE); the codes and Xhat are 0.05 of that time.  Measured at
// n = 50,000, d = 1536, TQ_PROD b = 4: 11.80 ms as an fp32 GEMM on CUDA cores (40 TFLOP/s of 4 n d^2), 1.14 ms here (414).
// What keeps it from the 0.72 ms of five passes at the bf16 rate: the power cap (1.3 GHz in a loop) and the workers' chain
// per k-block (expansion 350 cycles, proxy fence 190, a drain 1,300 per chunk) against 1,280 cycles of MMAs.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <vector>

#include <cuda_fp16.h>

#include "tq_dequant_tc.h"
#include "tq_quantize_tc.h"
#include "tq_tc.cuh"

namespace tq {
namespace dq {

using namespace tq::tc;

namespace {

constexpr int BM = 128;             // rows of codes per CTA = TMEM lanes
constexpr int BK = 64;              // coordinates per k-block: fp16 elements of one 128-byte swizzled row
constexpr int NWORK = 16;           // worker warps: they expand codes ahead of the MMAs and drain accumulators behind them
constexpr int kWork0 = 2;           // after the TMA warp and the MMA warp
constexpr int NTHREADS = 32 * (kWork0 + NWORK);
constexpr int kMapRows = 64;        // rows of a B box

template <int BN, int CTAS>
struct Cfg {
  static constexpr int kBRows = BN / CTAS;                       // rows of B this CTA loads
  static constexpr int kABytes = BM * BK * 2;                    // one A limb
  static constexpr int kBBytes = kBRows * BK * 2;                // one B limb
  static constexpr int kStageBytes = 2 * kABytes + 2 * kBBytes;
  static constexpr int kStages = BN == 64 ? 4 : 3;
  static constexpr int kTmemCols = 2 * BN;
  static constexpr int kColsPerWarp = BN / 4;                    // accumulator columns of one worker warp
  static constexpr int kStoreBytes = NWORK * 2048;               // [32 rows x 16 columns] fp32 per worker warp
  static constexpr int kSmemBytes = kStages * kStageBytes + 1024 + 512 + kStoreBytes;
};

struct Args {
  int64_t n;
  int d, num_kb;                    // k-blocks of 64 coordinates
  int chunk;                        // k-blocks per accumulation
  int tiles_m, tiles_n;
  int split;                        // CTAs of a cluster that share one tile's K (1: none; more only where every CTA has one tile)
  const uint8_t* idx;
  const uint8_t* qjl;
  const float* gamma;               // nullptr: no z term
  const float* norms;               // nullable
  int idx_rb, qjl_rb;
  int bits;                         // b_m; 0: no centroid term
  int nibble;                       // TQ_LAYOUT_NIBBLE
  uint32_t tab[4][4];               // bytes of the fp16 limbs of the codebook: hi low byte, hi high byte, lo low, lo high; 16 entries each
  // Weights of the accumulators, powers of two but for coef.  They are applied as the accumulators are drained, so that the sums
  // are in the units of the result and any norm and gamma of an fp32 result's range may multiply them.
  float oscale;                     // 2^-(eP + ec): centroid term
  float gscale;                     // coef 2^-eS: sign term, per unit of gamma
  float* out;
  int64_t ldo;
  int tma_store;                    // Xhat rows are 16-byte aligned: boxes leave by TMA
  int* status;
};

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) { return __byte_perm(a, b, sel); }

// Eight b-bit codes (low bits of x) as eight nibbles.
__device__ __forceinline__ uint32_t spread3(uint32_t x) {
  x = (x & 0x00000fffu) | ((x & 0x00fff000u) << 4);
  x = (x & 0x003f003fu) | ((x & 0x0fc00fc0u) << 2);
  return (x & 0x07070707u) | ((x & 0x38383838u) << 1);
}
__device__ __forceinline__ uint32_t spread2(uint32_t x) {
  x = (x & 0x000000ffu) | ((x & 0x0000ff00u) << 8);
  x = (x & 0x000f000fu) | ((x & 0x00f000f0u) << 4);
  return (x & 0x03030303u) | ((x & 0x0c0c0c0cu) << 2);
}
__device__ __forceinline__ uint32_t spread1(uint32_t x) {
  x = (x & 0x0fu) | ((x & 0xf0u) << 12);
  x = (x & 0x00030003u) | ((x & 0x000c000cu) << 6);
  return (x & 0x01010101u) | ((x & 0x02020202u) << 3);
}

// Word w (32 bits) of a packed row of rb bytes; zero past its end.
__device__ __forceinline__ uint32_t row_word(const uint8_t* row, int rb, int w) {
  return 4 * w < rb ? __ldg(reinterpret_cast<const uint32_t*>(row) + w) : 0u;
}

// Sixteen coordinates (part `part` of k-block kb) as raw packed words; unpack_* turns them into nibbles where they are used.
__device__ __forceinline__ void load_part(const Args& a, int64_t row, int kb, int part, int term, uint32_t (&w)[2]) {
  if (a.nibble) {   // eight bytes of the combined row, wholly in one of its two arrays (16-byte multiples)
    const int off = kb * 32 + 8 * part;
    uint2 v = make_uint2(0u, 0u);
    if (off < a.idx_rb) v = __ldg(reinterpret_cast<const uint2*>(a.idx + (size_t)row * a.idx_rb + off));
    else if (off - a.idx_rb < a.qjl_rb) v = __ldg(reinterpret_cast<const uint2*>(a.qjl + (size_t)row * a.qjl_rb + (off - a.idx_rb)));
    w[0] = v.x;
    w[1] = v.y;
    return;
  }
  const int bits = term == 0 ? a.bits : 1;
  const uint8_t* r = term == 0 ? a.idx + (size_t)row * a.idx_rb : a.qjl + (size_t)row * a.qjl_rb;
  const int rb = term == 0 ? a.idx_rb : a.qjl_rb;
  const int bit = (kb * 64 + 16 * part) * bits, word = bit >> 5;   // 16 bits codes start on a 16-bit boundary
  w[0] = row_word(r, rb, word);
  w[1] = bits > 2 ? row_word(r, rb, word + 1) : 0u;
  if (bit & 16) {
    w[0] = __funnelshift_r(w[0], w[1], 16);
    w[1] >>= 16;
  }
}

// The sixteen codes as two words of eight nibbles.
__device__ __forceinline__ void unpack_indices(const Args& a, const uint32_t (&w)[2], uint32_t (&nib)[2]) {
  if (a.nibble || a.bits == 4) { nib[0] = w[0]; nib[1] = w[1]; }
  else if (a.bits == 3) { nib[0] = spread3(w[0]); nib[1] = spread3(__funnelshift_r(w[0], w[1], 24)); }
  else if (a.bits == 2) { nib[0] = spread2(w[0]); nib[1] = spread2(w[0] >> 16); }
  else { nib[0] = spread1(w[0]); nib[1] = spread1(w[0] >> 8); }
}
// The sixteen sign bits at the tops of the nibbles of two words.
__device__ __forceinline__ void unpack_signs(const Args& a, const uint32_t (&w)[2], uint32_t (&nib)[2]) {
  if (a.nibble) { nib[0] = w[0]; nib[1] = w[1]; }
  else { nib[0] = spread1(w[0]) << 3; nib[1] = spread1(w[0] >> 8) << 3; }
}

// The limbs of sixteen centroids into one row of the two A tiles: eight coordinates = one 16-byte piece of each limb's row.
// Four codes are four selectors of a byte permute over a table of eight bytes.
__device__ __forceinline__ void expand_indices(const Args& a, const uint32_t (&w)[2], unsigned char* dst, int lo_offset, uint32_t piece, uint32_t swz) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t four = h == 0 ? w[q] : w[q] >> 16;
      const uint32_t sel = four & 0x7777u;
      uint32_t byte[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) byte[p] = prmt(a.tab[p][0], a.tab[p][1], sel);
      if (a.bits == 4) {   // sixteen centroids: the upper half of the table where bit 3 of the code is set
        const uint32_t up = prmt(0x0000ff00u, 0u, (four >> 3) & 0x1111u);
#pragma unroll
        for (int p = 0; p < 4; ++p) byte[p] = (byte[p] & ~up) | (prmt(a.tab[p][2], a.tab[p][3], sel) & up);
      }
      hi[2 * h] = prmt(byte[0], byte[1], 0x5140u);
      hi[2 * h + 1] = prmt(byte[0], byte[1], 0x7362u);
      lo[2 * h] = prmt(byte[2], byte[3], 0x5140u);
      lo[2 * h + 1] = prmt(byte[2], byte[3], 0x7362u);
    }
    const uint32_t off = ((piece + (uint32_t)q) ^ swz) << 4;
    *reinterpret_cast<uint4*>(dst + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(dst + lo_offset + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

// Sixteen signs as fp16 +-1: -1.0 (0xbc00) with the sign flipped where the bit is set.
__device__ __forceinline__ void expand_signs(const uint32_t (&w)[2], unsigned char* dst, uint32_t piece, uint32_t swz) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    uint32_t z[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {   // coordinates 2 p and 2 p + 1
      const uint32_t x = w[q] >> (8 * p);
      z[p] = 0xbc00bc00u ^ ((x << 12) & 0x8000u) ^ ((x << 24) & 0x80000000u);
    }
    *reinterpret_cast<uint4*>(dst + (((piece + (uint32_t)q) ^ swz) << 4)) = make_uint4(z[0], z[1], z[2], z[3]);
  }
}

// A warp's 32 rows x NC columns leave through its 2 KB of shared memory in pieces of 16 columns: by TMA where Xhat's rows are
// 16-byte aligned (64-byte swizzle: piece p of row y at p ^ ((y >> 1) & 3)), else as 64-byte row pieces.
template <int NC>
__device__ __forceinline__ void store_sums(const Args& a, const CUtensorMap& map, const float (&r)[NC], float scale, int64_t row0,
                                           int col0, unsigned char* buf, int lane) {
#pragma unroll
  for (int q = 0; q < NC / 16; ++q) {
    const int c0 = col0 + 16 * q;
    if (c0 >= a.d) break;
    if (lane == 0) tma_store_wait_read();
    __syncwarp();
    const uint32_t sw = (uint32_t)((lane >> 1) & 3);
#pragma unroll
    for (int p = 0; p < 4; ++p)
      *reinterpret_cast<float4*>(buf + lane * 64 + ((p ^ sw) << 4)) =
          make_float4(r[16 * q + 4 * p] * scale, r[16 * q + 4 * p + 1] * scale, r[16 * q + 4 * p + 2] * scale, r[16 * q + 4 * p + 3] * scale);
    if (a.tma_store) {
      fence_proxy_async();
      __syncwarp();
      if (lane == 0 && row0 < a.n) {
        tma_store_2d(&map, buf, c0, (int)row0);   // clipped at row n and column d
        tma_store_commit();
      }
    } else {
      __syncwarp();
      const int cc = lane & 15;
      for (int y = lane >> 4; y < 32; y += 2) {
        const float v = *reinterpret_cast<const float*>(buf + y * 64 + ((((uint32_t)cc >> 2) ^ ((y >> 1) & 3)) << 4) + (cc & 3) * 4);
        if (row0 + y < a.n && c0 + cc < a.d && TQ_DEVICE_CHECK(c0 + cc < a.ldo, a.status)) a.out[(row0 + y) * a.ldo + c0 + cc] = v;
      }
      __syncwarp();
    }
  }
}

template <int BN, int CTAS>
__global__ void __launch_bounds__(NTHREADS, 1)
dequant_kernel(const __grid_constant__ CUtensorMap tmP1, const __grid_constant__ CUtensorMap tmP2,
               const __grid_constant__ CUtensorMap tmS1, const __grid_constant__ CUtensorMap tmS2,
               const __grid_constant__ CUtensorMap tmO, const __grid_constant__ Args a) {
  using C = Cfg<BN, CTAS>;
  const int rank = CTAS == 2 ? (int)cluster_ctarank() : 0;
  const int split = CTAS == 2 ? 1 : a.split, krank = CTAS == 2 || split == 1 ? 0 : (int)cluster_ctarank();
  const int64_t unit = blockIdx.x / (CTAS * split), nunits = gridDim.x / (CTAS * split);
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kStages * C::kStageBytes);
  uint64_t* full_b = bars;                      // [kStages]  TMA -> MMA (the leader's)
  uint64_t* full_a = bars + C::kStages;         // [kStages]  code expansion -> MMA (the leader's)
  uint64_t* empty = bars + 2 * C::kStages;      // [kStages]  MMA -> TMA and code expansion
  uint64_t* tfull = bars + 3 * C::kStages;      // [2]        MMA -> epilogue
  uint64_t* tempty = tfull + 2;                 // [2]        epilogue -> MMA (the leader's)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  unsigned char* stg = reinterpret_cast<unsigned char*>(bars) + 512;   // [NWORK][2048]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t num_tiles = (int64_t)a.tiles_m * a.tiles_n;
  const int kChunk = a.chunk, all_chunks = (a.num_kb + kChunk - 1) / kChunk;
  // chunks of this CTA: all of them, or its share of the tile's K
  const int c_begin = min(all_chunks, (all_chunks + split - 1) / split * krank), c_end = min(all_chunks, (all_chunks + split - 1) / split * (krank + 1));
  // every tile runs, per chunk of coordinates, the k-blocks of the centroid term and then those of the sign term
  const int first_term = a.bits > 0 ? 0 : 1, last_term = a.gamma != nullptr ? 1 : 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(&full_b[s], 1);
      mbar_init(&full_a[s], NWORK * CTAS);
      mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], NWORK * CTAS);
    }
    *abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmP1);
    tma_prefetch_desc(&tmP2);
    tma_prefetch_desc(&tmS1);
    tma_prefetch_desc(&tmS2);
  }
  if (warp == 1) {
    if (CTAS == 2) tmem_alloc_pair(tmem_slot, C::kTmemCols);
    else tmem_alloc(tmem_slot, C::kTmemCols);
  }
  tc_fence_before();
  if (CTAS == 2) cluster_sync();
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (B limbs)
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int64_t t = unit; t < num_tiles && ok; t += nunits) {
        const int n0 = (int)(t % a.tiles_n) * BN + rank * C::kBRows;
        for (int c = c_begin; c < c_end && ok; ++c)
          for (int term = first_term; term <= last_term && ok; ++term)
            for (int kb = c * kChunk; kb < min((c + 1) * kChunk, a.num_kb); ++kb) {
              if (!(ok = mbar_wait_suspended(&empty[stage], phase ^ 1u, abort_flag, a.status))) break;
              unsigned char* sb = smem + stage * C::kStageBytes + 2 * C::kABytes;
              const CUtensorMap* m1 = term == 0 ? &tmP1 : &tmS1;
              const CUtensorMap* m2 = term == 0 ? &tmP2 : &tmS2;
              if (CTAS == 2) {
                if (rank == 0) mbar_arrive_expect_tx(&full_b[stage], 2 * 2 * C::kBBytes);
#pragma unroll
                for (int r = 0; r < C::kBRows; r += kMapRows) {
                  tma_load_2d_pair(sb + r * BK * 2, m1, &full_b[stage], kb * BK, n0 + r);
                  tma_load_2d_pair(sb + C::kBBytes + r * BK * 2, m2, &full_b[stage], kb * BK, n0 + r);
                }
              } else {
                mbar_arrive_expect_tx(&full_b[stage], 2 * C::kBBytes);
#pragma unroll
                for (int r = 0; r < C::kBRows; r += kMapRows) {
                  tma_load_2d(sb + r * BK * 2, m1, &full_b[stage], kb * BK, n0 + r);
                  tma_load_2d(sb + C::kBBytes + r * BK * 2, m2, &full_b[stage], kb * BK, n0 + r);
                }
              }
              if (++stage == C::kStages) {
                stage = 0;
                phase ^= 1u;
              }
            }
      }
      if (!ok) {
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);   // copies in flight land before the shared memory is given up
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0 && rank == 0) {
      // fp16 x fp16 -> fp32, both K-major: as instr_desc_bf16 with the operand formats 0
      constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)((BM * CTAS) >> 4) << 24);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      uint32_t it = 0;
      for (int64_t t = unit; t < num_tiles && ok; t += nunits)
        for (int c = c_begin; c < c_end && ok; ++c)
          for (int term = first_term; term <= last_term && ok; ++term, ++it) {
            const uint32_t acc = it & 1u, acc_phase = (it >> 1) & 1u;
            if (!(ok = mbar_wait_suspended(&tempty[acc], acc_phase ^ 1u, abort_flag, a.status))) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + acc * BN;
            uint32_t accumulate = 0u;
            for (int kb = c * kChunk; kb < min((c + 1) * kChunk, a.num_kb); ++kb) {
              if (!(ok = mbar_wait_suspended(&full_b[stage], phase, abort_flag, a.status))) break;
              if (!(ok = mbar_wait_suspended(&full_a[stage], phase, abort_flag, a.status))) break;
              tc_fence_after();
              const uint32_t sa = smem_u32(smem + stage * C::kStageBytes);
              const uint64_t a1 = smem_desc_sw128(sa), a2 = smem_desc_sw128(sa + C::kABytes);
              const uint64_t b1 = smem_desc_sw128(sa + 2 * C::kABytes), b2 = smem_desc_sw128(sa + 2 * C::kABytes + C::kBBytes);
              auto mma = [&](uint64_t ad, uint64_t bd) {
                if (CTAS == 2) umma_bf16_pair(d_tmem, ad, bd, idesc, accumulate);
                else umma_bf16(d_tmem, ad, bd, idesc, accumulate);
                accumulate = 1u;
              };
#pragma unroll
              for (int k = 0; k < BK / 16; ++k) {   // the small products first: fewer additions truncate a full-size sum
                const uint64_t off = (uint64_t)(k * 2);   // 32 bytes per K step
                mma(a1 + off, b2 + off);                            // hi lo, or z lo
                if (term == 0) mma(a2 + off, b1 + off);             // lo hi
              }
#pragma unroll
              for (int k = 0; k < BK / 16; ++k) mma(a1 + (uint64_t)(k * 2), b1 + (uint64_t)(k * 2));   // hi hi, or z hi
              if (CTAS == 2) umma_commit_pair(&empty[stage]);
              else umma_commit(&empty[stage]);
              if (++stage == C::kStages) {
                stage = 0;
                phase ^= 1u;
              }
            }
            if (ok) {
              if (CTAS == 2) umma_commit_pair(&tfull[acc]);
              else umma_commit(&tfull[acc]);
            }
          }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ workers: expansion ahead of the MMAs, drain behind them
    // A warp owns 32 rows (its TMEM lane group lg) x one quarter: sixteen of a k-block's 64 coordinates when it expands,
    // a quarter of the tile's columns when it drains.  Chunk by chunk it expands chunk j and then drains chunk j - 1, so
    // that the MMAs of chunk j find their operand while the workers wait for chunk j - 1.  (Waiting for a stage while
    // expanding chunk j needs MMAs of chunk j at most, whose accumulator was drained as chunk j - 2: no cycle.)
    constexpr int NC = C::kColsPerWarp;
    const int lg = warp & 3, part = (warp - kWork0) >> 2;
    const int rt = lg * 32 + lane;
    const uint32_t swz = (uint32_t)(rt & 7);
    unsigned char* buf = stg + (warp - kWork0) * 2048;
    const int nterms = last_term - first_term + 1;
    const int jobs = (c_end - c_begin) * nterms;       // accumulations of a tile
    bool ok = true;
    int stage = 0;
    uint32_t phase = 0, it = 0;
    float r[NC];
    for (int64_t t = unit; t < num_tiles && ok; t += nunits) {
      const int64_t row0 = ((t / a.tiles_n) * CTAS + rank) * BM + lg * 32, row = row0 + lane;
      const int col0 = (int)(t % a.tiles_n) * BN + part * NC;
      const bool row_ok = row < a.n;
      const int64_t src_row = row_ok ? row : a.n - 1;   // rows past the end repeat the last one
      const float g = (a.gamma != nullptr && row_ok) ? a.gscale * __ldg(a.gamma + row) : 0.f;
      const float nu = (a.norms != nullptr && row_ok) ? __ldg(a.norms + row) : 1.f;
#pragma unroll
      for (int i = 0; i < NC; ++i) r[i] = 0.f;
      uint32_t nxt[2];
      load_part(a, src_row, c_begin * kChunk, part, first_term, nxt);
      for (int j = 0; j <= jobs; ++j) {
        if (j < jobs) {
          const int c = c_begin + j / nterms, term = first_term + j % nterms;
          const int kb_end = min((c + 1) * kChunk, a.num_kb);
          for (int kb = c * kChunk; kb < kb_end; ++kb) {
            uint32_t w[2] = {nxt[0], nxt[1]}, nib[2];
            // the codes of the next k-block are requested before this one is expanded
            if (kb + 1 < kb_end) load_part(a, src_row, kb + 1, part, term, nxt);
            else if (j + 1 < jobs) load_part(a, src_row, (c_begin + (j + 1) / nterms) * kChunk, part, first_term + (j + 1) % nterms, nxt);
            if (term == 0) unpack_indices(a, w, nib);
            else unpack_signs(a, w, nib);
            if (!(ok = mbar_wait_suspended(&empty[stage], phase ^ 1u, abort_flag, a.status))) break;
            unsigned char* dst = smem + stage * C::kStageBytes + rt * 128;
            if (term == 0) expand_indices(a, nib, dst, C::kABytes, 2u * part, swz);
            else expand_signs(nib, dst, 2u * part, swz);
            // The tensor core of this SM reads what these threads wrote, in a pair too (each SM reads its own rows of A):
            // the proxy fence orders the writes, the arrival only tells the leader's issuer.  A cluster-scope release
            // here and acquire there took 1,200-1,400 cycles per k-block and bound the kernel (1.62 against 1.30 ms at n = 50,000, d = 1536).
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
              if (CTAS == 2) mbar_arrive_leader(&full_a[stage]);
              else mbar_arrive(&full_a[stage]);
            }
            if (++stage == C::kStages) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (!ok) break;
        }
        if (j == 0) continue;
        const uint32_t acc = it & 1u, acc_phase = (it >> 1) & 1u;
        const int drained_term = first_term + (j - 1) % nterms;
        ++it;
        if (!(ok = mbar_wait_suspended(&tfull[acc], acc_phase, abort_flag, a.status))) break;
        tc_fence_after();
        const float s = drained_term == 0 ? a.oscale : g;
        const uint32_t base = tmem_base + ((uint32_t)(lg * 32) << 16) + acc * BN + part * NC;
#pragma unroll
        for (int q = 0; q < NC / 16; ++q) {
          uint32_t v[16];
          tmem_ld16(base + 16 * q, v);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) r[16 * q + i] = fmaf(s, __uint_as_float(v[i]), r[16 * q + i]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (CTAS == 2) mbar_arrive_leader(&tempty[acc]);
          else mbar_arrive(&tempty[acc]);
        }
      }
      if (!ok) break;
      if (split > 1) break;   // one tile per CTA: the sums of the cluster meet below
      store_sums<NC>(a, tmO, r, nu, row0, col0, buf, lane);
    }
    if constexpr (CTAS == 1) {
      if (split > 1) {
#pragma unroll
        for (int i = 0; i < NC; i += 4) *reinterpret_cast<float4*>(buf + lane * 64 + 4 * i) = make_float4(r[i], r[i + 1], r[i + 2], r[i + 3]);
      }
    }
    if (lane == 0) tma_store_wait_all();   // this warp's stores have completed before the CTA gives up its shared memory
    __syncwarp();
  }

  if constexpr (CTAS == 1) {
    if (split > 1) {
      // The sums of worker warp w are added up, in rank order, by the CTA of rank w mod split, which also stores them.
      cluster_sync();
      const int w = warp - kWork0;
      if (w >= 0 && w % split == krank) {
        constexpr int NC = C::kColsPerWarp;
        const int lg = warp & 3;
        const int64_t row0 = unit / a.tiles_n * BM + lg * 32, row = row0 + lane;
        unsigned char* buf = stg + w * 2048;
        float r[NC];
#pragma unroll
        for (int i = 0; i < NC; ++i) r[i] = 0.f;
        for (int p = 0; p < split; ++p) {
          uint32_t peer;
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(smem_u32(buf + lane * 64)), "r"(p));
#pragma unroll
          for (int i = 0; i < NC; i += 4) {
            float4 v;
            asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(peer + 4 * i) : "memory");
            r[i] += v.x; r[i + 1] += v.y; r[i + 2] += v.z; r[i + 3] += v.w;
          }
        }
        __syncwarp();
        const float nu = (a.norms != nullptr && row < a.n) ? __ldg(a.norms + row) : 1.f;
        store_sums<NC>(a, tmO, r, nu, row0, (int)(unit % a.tiles_n) * BN + (w >> 2) * NC, buf, lane);
        if (lane == 0) tma_store_wait_all();
        __syncwarp();
      }
      cluster_sync();   // nobody leaves while its sums may still be read
    }
  }

  tc_fence_before();
  if (CTAS == 2) cluster_sync();
  else __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    if (CTAS == 2) tmem_dealloc_pair(tmem_base, C::kTmemCols);
    else tmem_dealloc(tmem_base, C::kTmemCols);
  }
}

// ---------------------------------------------------------------- plan set-up
// out_hi/lo[i][j] = fp16 limbs of M[j][i] * scale (the transpose of a d x d matrix), row pitch `pitch`.
__global__ void transpose_limbs_kernel(const float* __restrict__ M, int d, int64_t ldm, float scale, __half* __restrict__ hi,
                                       __half* __restrict__ lo, int64_t pitch) {
  __shared__ float tile[32][33];
  const int j0 = blockIdx.y * 32, i0 = blockIdx.x * 32;
  for (int y = threadIdx.y; y < 32; y += blockDim.y)
    tile[y][threadIdx.x] = (j0 + y < d && i0 + (int)threadIdx.x < d) ? M[(int64_t)(j0 + y) * ldm + i0 + threadIdx.x] * scale : 0.f;
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += blockDim.y) {
    const int i = i0 + y, j = j0 + threadIdx.x;
    if (i >= d || j >= pitch) continue;
    const float v = j < d ? tile[threadIdx.x][y] : 0.f;
    const __half h = __float2half_rn(v);
    hi[(int64_t)i * pitch + j] = h;
    lo[(int64_t)i * pitch + j] = __float2half_rn(v - __half2float(h));
  }
}

// Exponent e with 2^13 <= max 2^e < 2^14 (0 for an all-zero matrix).
int limb_exponent(double mx) { return mx > 0.0 ? 13 - std::ilogb(mx) : 0; }

template <int BN, int CTAS>
cudaError_t launch(const tq_plan* plan, const CUtensorMap& out_map, Args& a, cudaStream_t st) {
  using C = Cfg<BN, CTAS>;
  auto kern = dequant_kernel<BN, CTAS>;
  static std::atomic<unsigned long long> attr_devices{0};   // devices whose function attribute has been set
  const int dev = plan->device;
  if (dev >= 64 || !((attr_devices.load(std::memory_order_relaxed) >> dev) & 1ull)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
    if (e != cudaSuccess) return e;
    if (dev < 64) attr_devices.fetch_or(1ull << dev, std::memory_order_relaxed);
  }
  a.tiles_m = (int)((a.n + BM * CTAS - 1) / (BM * CTAS));
  a.tiles_n = (a.d + BN - 1) / BN;
  const int64_t tiles = (int64_t)a.tiles_m * a.tiles_n;
  const int units = (int)std::min<int64_t>(tiles, sm_count() / CTAS);
  // few rows leave most of the chip idle: clusters of up to eight CTAs share a tile's K (at least two k-blocks each)
  a.split = 1;
  while (CTAS == 1 && a.split < 8 && tiles * a.split * 2 <= sm_count() && a.num_kb >= 4 * a.split) a.split *= 2;
  if (BN == 64) a.chunk = std::min(a.chunk, 2);   // four stages: two chunks in flight
  const int cluster = CTAS * a.split;
  const auto& m = plan->dq;
  const CUtensorMap &s1 = plan->mode == TQ_PROD ? m.map_s_hi : m.map_p_hi, &s2 = plan->mode == TQ_PROD ? m.map_s_lo : m.map_p_lo;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(units * cluster));
  cfg.blockDim = dim3(NTHREADS);
  cfg.dynamicSmemBytes = C::kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 1 : 0;
  count_launches(1);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, m.map_p_hi, m.map_p_lo, s1, s2, out_map, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t plan_init(tq_plan* plan, const float* Pi, const float* S) {
  auto& m = plan->dq;
  m.ok = 0;
  const int d = plan->d;
  if (!tc::supported(d)) return cudaSuccess;
  m.pitch = plan->dpad;
  const size_t count = (size_t)d * m.pitch;
  auto max_abs = [&](const float* M) {
    double mx = 0.0;
    for (size_t i = 0; i < (size_t)d * d; ++i) mx = std::max(mx, std::fabs((double)M[i]));
    return mx;
  };
  double cmax = 0.0;
  const int levels = plan->mse_bits > 0 ? 1 << plan->mse_bits : 0;
  for (int i = 0; i < levels; ++i) cmax = std::max(cmax, std::fabs((double)plan->cb.c[i]));
  const double pmax = max_abs(Pi), smax = S ? max_abs(S) : 0.0;
  if (!std::isfinite(pmax) || !std::isfinite(smax)) return cudaSuccess;   // the CUDA-core path carries such values through
  const int eP = limb_exponent(pmax), eS = limb_exponent(smax), ec = limb_exponent(cmax);
  for (int e : {eP, eS, ec, eP + ec})
    if (e > 100 || e < -100) return cudaSuccess;
  m.gscale = (float)std::ldexp(1.0, -eS) * plan->coef;
  m.oscale = (float)std::ldexp(1.0, -(eP + ec));
  for (int p = 0; p < 4; ++p)
    for (int q = 0; q < 4; ++q) m.tab[p][q] = 0u;
  for (int i = 0; i < levels; ++i) {
    const float v = (float)std::ldexp((double)plan->cb.c[i], ec);
    const __half_raw h = __half(__float2half_rn(v));
    const __half_raw l = __half(__float2half_rn(v - __half2float(__half(h))));
    const uint32_t bytes[4] = {(uint32_t)h.x & 255u, (uint32_t)h.x >> 8, (uint32_t)l.x & 255u, (uint32_t)l.x >> 8};
    for (int p = 0; p < 4; ++p) m.tab[p][i >> 2] |= bytes[p] << (8 * (i & 3));
  }
  const dim3 grid((d + 31) / 32, (m.pitch + 31) / 32), block(32, 8);
  for (int which = 0; which < (S ? 2 : 1); ++which) {
    __half** hi = which == 0 ? &m.p_hi : &m.s_hi;
    __half** lo = which == 0 ? &m.p_lo : &m.s_lo;
    cudaError_t e = cudaMalloc(hi, count * 2);
    if (e == cudaSuccess) e = cudaMalloc(lo, count * 2);
    if (e != cudaSuccess) return e;
    // dRotCat: rows of Pi, then (from row dpad) rows of S
    transpose_limbs_kernel<<<grid, block>>>(plan->dRotCat + (which == 0 ? 0 : (size_t)plan->dpad * plan->dpad), d, plan->dpad,
                                            (float)std::ldexp(1.0, which == 0 ? eP : eS), *hi, *lo, m.pitch);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (!tc::make_half_map(which == 0 ? &m.map_p_hi : &m.map_s_hi, *hi, d, d, m.pitch, kMapRows) ||
        !tc::make_half_map(which == 0 ? &m.map_p_lo : &m.map_s_lo, *lo, d, d, m.pitch, kMapRows))
      return cudaErrorInvalidValue;
  }
  m.ok = 1;
  return cudaSuccess;
}

void plan_free(tq_plan* plan) {
  cudaFree(plan->dq.p_hi);
  cudaFree(plan->dq.p_lo);
  cudaFree(plan->dq.s_hi);
  cudaFree(plan->dq.s_lo);
}

int dequantize(const tq_plan* plan, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma, const float* norms,
               float* Xhat, int64_t ldxh, cudaStream_t st, const char* who) {
  const auto& m = plan->dq;
  const bool prod = plan->mode == TQ_PROD;
  Args a;
  a.d = plan->d;
  a.num_kb = (plan->d + BK - 1) / BK;
  // A longer accumulation drains less often and truncates more: measured rms error per result at 1 / 2 / 4 k-blocks
  // 2.5e-7 / 5e-7 / 9e-7, time 1.64 / 1.30 / 1.12 ms (n = 50,000, d = 1536, TQ_PROD).  An fp32 chain over the same K errs by
  // 2e-7 at K = 128, 4.3e-7 at 580, 7e-7 at 1536, 1.2e-6 at 3072: each K gets the longest one that errs no more.
  const int64_t total_k = (int64_t)plan->ncat * plan->dpad;
  a.chunk = total_k < 1024 ? 1 : total_k < 3072 ? 2 : 4;
  a.idx_rb = (int)plan->idx_row_bytes;
  a.qjl_rb = (int)plan->qjl_row_bytes;
  a.bits = plan->mse_bits;
  a.nibble = plan->layout == TQ_LAYOUT_NIBBLE ? 1 : 0;
  for (int p = 0; p < 4; ++p)
    for (int q = 0; q < 4; ++q) a.tab[p][q] = m.tab[p][q];
  a.gscale = m.gscale;
  a.oscale = m.oscale;
  a.ldo = ldxh;
  a.tma_store = ldxh % 4 == 0;
  a.status = plan->d_status;
  constexpr int64_t kMaxRows = (int64_t)1 << 30;   // row coordinates of the store map are 32-bit
  for (int64_t r0 = 0; r0 < n; r0 += kMaxRows) {
    a.n = std::min(kMaxRows, n - r0);
    a.idx = idx ? idx + (size_t)r0 * plan->idx_row_bytes : nullptr;
    a.qjl = prod ? qjl + (size_t)r0 * plan->qjl_row_bytes : nullptr;
    a.gamma = prod ? gamma + r0 : nullptr;
    a.norms = norms ? norms + r0 : nullptr;
    a.out = Xhat + r0 * ldxh;
    CUtensorMap om = m.map_p_hi;   // any valid map where the rows do not leave by TMA
    if (a.tma_store)
      TQ_REQUIRE(tc::make_store_map_f32(&om, a.out, a.n, plan->d, ldxh), TQ_ERR_CUDA, "%s: cuTensorMapEncodeTiled failed", who);
    // 256 x 256 tiles on CTA pairs or 128 x 64 tiles on single CTAs, whichever needs less time in whole waves: a wave of the
    // former took 1.6 times as long as one of the latter (d = 1536: 76 against 48 us), with eleven times the work in it.
    const int64_t big = ((a.n + 2 * BM - 1) / (2 * BM)) * ((plan->d + 255) / 256), pairs = sm_count() / 2;
    const int64_t small = ((a.n + BM - 1) / BM) * ((plan->d + 63) / 64), singles = sm_count();
    const bool pair = 8 * ((big + pairs - 1) / pairs) <= 5 * ((small + singles - 1) / singles);
    if (pair) TQ_CHECK_CUDA((launch<256, 2>(plan, om, a, st)), who);
    else TQ_CHECK_CUDA((launch<64, 1>(plan, om, a, st)), who);
  }
  return TQ_OK;
}

}  // namespace dq
}  // namespace tq
