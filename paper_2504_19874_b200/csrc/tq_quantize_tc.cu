// Tensor-core quantisation path (sm_100a): the rotation y = Pi u and the QJL projection
// z = S' e as tcgen05 GEMMs fed by TMA, with the nearest-centroid search, bit packing,
// residual and sign extraction fused into the epilogue that reads the accumulators from TMEM.
//
// fp32 fidelity on bf16 tensor cores: every fp32 operand is split into two bf16 limbs
// (v = hi + lo + O(2^-17 |v|)), and each product is formed as hi*hi + hi*lo + lo*hi with fp32
// accumulation (3 MMA passes).  The dropped terms are ~2^-17 relative per product, i.e.
// ~1e-7 on a rotated coordinate of a unit vector at d = 1536 -- far inside the 1e-5 window in
// which a nearest-centroid decision may legitimately differ from exact arithmetic.
//
// Two forms of the GEMM kernel: one CTA per tile of 128 rows, and (the usual one at d > 128) a pair of CTAs of one
// cluster per tile of 256 rows (tcgen05 cta_group::2), which halves what every SM reads of B from shared memory.  The
// tiles are up to 256 columns wide; few rows take narrower ones, so that every SM has one (pick_tile).
#include <atomic>
#include <cfloat>
#include <cstdlib>
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "tq_quantize_tc.h"
#include "tq_tc.cuh"

namespace tq {
namespace tc {

namespace {

constexpr int BM = 128;          // rows of X per tile = TMEM lanes
constexpr int BK = 64;           // bf16 elements per 128-byte swizzled row
constexpr int UMMA_K = 16;
constexpr int NSPLIT = 2;        // spare warps beside the GEMM: the next block's operand limbs (see SplitTask), gamma (MODE 2)

// CTAS = 2: two CTAs of a cluster share one 256-row tile (tcgen05 cta_group::2).  Each loads its own 128 rows of A and
// its own half of B's rows, so a k-block costs each SM 64 KB of shared-memory writes instead of 96 and its MMAs read
// half of B from the partner: the shared-memory bandwidth that caps the one-CTA kernel (158 bytes per clock wanted,
// 128 available) drops to 104.
struct Tile { int bn, ctas; };   // columns of a tile, CTAs that share it

template <int BN, int CTAS>
struct Cfg {
  // epilogue warps per TMEM lane group: each takes 1/kEps of the tile's columns, 64 (32 where the tile is the whole row)
  static constexpr int kEps = CTAS == 1 && BN == 128 ? 4 : BN / 64;
  static constexpr int kThreads = 32 * (2 + 4 * kEps + NSPLIT);             // warp 0: TMA, warp 1: MMA + TMEM owner, epilogue, spare
  static constexpr int kBRows = BN / CTAS;                                  // rows of B this CTA loads
  static constexpr int kStageBytes = 2 * BM * BK * 2 + 2 * kBRows * BK * 2; // A hi/lo + B hi/lo
  static constexpr int kStages = CTAS == 2 ? (BN == 128 ? 4 : 3) : (BN == 128 ? 3 : 4);
  static constexpr int kAccCols = BN == 192 ? 256 : BN;                     // TMEM columns from one accumulator to the next
  static constexpr int kTmemCols = 2 * kAccCols;                            // two accumulators
  static constexpr int kStoreBytes = 4 * kEps * 2048;  // MODE 1: one [32 rows x 64 B] box per epilogue warp, staged for a TMA store
  // bf16 rows have one limb: smaller stages, more of them in the same bytes
  static constexpr int kStageBytes1 = kStageBytes - BM * BK * 2;
  static constexpr int kStages1 = kStages * kStageBytes / kStageBytes1;
  static_assert((2 * kStages1 + 4) * 8 + 8 <= 192, "barriers");
  static constexpr int kSmemBytes = kStages * kStageBytes + 1024 /*alignment slack*/ + 512 /*barriers, centroids*/ + kStoreBytes;
};

struct GemmArgs {
  int64_t M;             // valid rows
  int N, K;              // = d, d
  int tiles_m, tiles_n;
  Codebook cb;
  uint8_t* out;          // packed idx (MODE 0/1) or qjl (MODE 2) rows
  size_t out_rb;
  __nv_bfloat16* E1;     // MODE 1: residual limbs, pitch ldE
  __nv_bfloat16* E2;
  const CUtensorMap* store_e1;   // host pointers to the TMA store maps of E1 / E2 (box 32 rows x 32 columns, 64-byte swizzle);
  const CUtensorMap* store_e2;   // the launcher passes them on as kernel arguments
  int64_t ldE;
  float* gpart;          // MODE 1: [parts][Mpad] partial sums of e^2, one per epilogue warp's columns; MODE 2: gamma from them
  float* gamma;          // MODE 2
  int parts;
  int64_t Mpad;
  const float* nu;       // per-row norm (MODE 1: a row with nu == 0 has residual 0; one_limb: see RowScale); nullable
  int one_limb;          // MODE 0, 1: the rows came in bf16, A is one limb of x 2^-e: two MMA passes, the accumulators are scaled
  // TQ_LAYOUT_NIBBLE (BITS = 3 with MODE 1, and MODE 2): the codes of 32 coordinates are four words of the combined
  // row [idx row | qjl row], nibble = index | sign << 3.  MODE 1 writes them with the sign bits clear, MODE 2 ORs
  // the sign bits in.
  int nibble;
  // Operand preparation of the NEXT block of rows (nu = ||x||, u = x / nu, bf16 limbs of u), done by NSPLIT spare
  // warps of every CTA while this launch's GEMM runs: the GEMM is bound by the tensor pipe and shared memory, the
  // preparation by HBM and a little issue bandwidth.  The rotate launch of TQ_MSE plans (MODE 0) carries one where it pays,
  // see quantize().
  struct SplitTask {
    const float* X;      // first row of the next block
    int64_t ldx, rows;   // rows == 0: nothing to do
    int d, dpad, normalize;
    __nv_bfloat16* L1;
    __nv_bfloat16* L2;
    float* norms;        // nullable
  } split;
  uint8_t* nib_idx;      // idx rows (stride nib_idx_rb) and qjl rows (stride nib_qjl_rb) of this block of rows
  uint8_t* nib_qjl;
  size_t nib_idx_rb, nib_qjl_rb;
  int* status;
};

// Rows of bf16 enter the rotation as they are but for a power of two, exactly: A = x down with |A| in [1, 2), and y = back * acc.
// (u = x / nu takes two limbs, that is a third MMA pass and half again the preparation: 1,001 rows of d = 3072, prod b = 2, took
// 118 us, 96 with one limb.)  A zero row, and one whose norm is not finite, becomes what x times 0 is.
struct RowScale {
  float down, back;
};
__device__ __forceinline__ RowScale row_scale(float nu) {
  if (!(nu > 0.f) || !(nu <= FLT_MAX)) return {0.f, 0.f};
  const float down = ldexpf(1.f, -max(-126, min(126, ilogbf(nu))));
  return {down, 1.f / (nu * down)};
}

// Bit i of the low byte of x at bit 4 i + 3.
__device__ __forceinline__ uint32_t spread_to_nibble_tops(uint32_t x) {
  x &= 0xffu;
  x = (x | (x << 12)) & 0x000f000fu;
  x = (x | (x << 6)) & 0x03030303u;
  x = (x | (x << 3)) & 0x11111111u;
  return x << 3;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// fp32 rows, 16-byte aligned, of at most 2048 NV / 16 elements per segment: a segment is held in registers (NV x 16
// bytes per lane, all loads in flight at once); a row of one segment is read once, longer rows a second time (from L2)
// after the norm is known.  NV follows d, so that short rows do not pay for sixteen mostly empty rounds (at d = 200 the
// kernel was bound by the issue of predicated-off instructions, 2.6 TB/s).  The sums are those of NV = 16: the rounds
// left out added fma(0, 0, s) = s.
template <bool NORMALIZE, int NV>
__device__ __forceinline__ void split_rows_vec(const float* __restrict__ X, int64_t ldx, int64_t n, int d, int dpad,
                                               __nv_bfloat16* __restrict__ L1, __nv_bfloat16* __restrict__ L2,
                                               float* __restrict__ norms, int64_t warp, int64_t nwarps, int lane) {
  const int nseg = (d + 128 * NV - 1) / (128 * NV);
  if (NV < 16) {
    // short rows (one segment): 16 / NV rows of a warp are in flight at once -- a single row of 800 bytes per warp
    // does not keep enough bytes in flight to fill the memory pipe
    constexpr int RB = 16 / NV;
    for (int64_t r0 = warp * RB; r0 < n; r0 += nwarps * RB) {
      float4 v[RB][NV];
#pragma unroll
      for (int k = 0; k < RB; ++k) {
        const float4* row4 = reinterpret_cast<const float4*>(X + min(r0 + k, n - 1) * ldx);
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          const int c = lane + 32 * i;
          v[k][i] = (4 * c < d) ? __ldg(row4 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
#pragma unroll
      for (int k = 0; k < RB; ++k) {
        const int64_t r = r0 + k;
        if (r >= n) break;
        float inv = 1.f;
        if (NORMALIZE) {
          float s = 0.f;
#pragma unroll
          for (int i = 0; i < NV; ++i)
            s = fmaf(v[k][i].x, v[k][i].x, fmaf(v[k][i].y, v[k][i].y, fmaf(v[k][i].z, v[k][i].z, fmaf(v[k][i].w, v[k][i].w, s))));
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          const float nu = sqrtf(s);
          inv = (nu > 0.f) ? 1.f / nu : 0.f;
          if (lane == 0 && norms != nullptr) norms[r] = nu;
        }
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          const int c = lane + 32 * i;
          if (4 * c >= d) continue;
          const float u0 = v[k][i].x * inv, u1 = v[k][i].y * inv, u2 = v[k][i].z * inv, u3 = v[k][i].w * inv;
          const float h0 = __bfloat162float(__float2bfloat16_rn(u0)), h1 = __bfloat162float(__float2bfloat16_rn(u1));
          const float h2 = __bfloat162float(__float2bfloat16_rn(u2)), h3 = __bfloat162float(__float2bfloat16_rn(u3));
          *reinterpret_cast<uint2*>(L1 + r * dpad + 4 * c) = make_uint2(pack_bf16x2(h0, h1), pack_bf16x2(h2, h3));
          *reinterpret_cast<uint2*>(L2 + r * dpad + 4 * c) = make_uint2(pack_bf16x2(u0 - h0, u1 - h1), pack_bf16x2(u2 - h2, u3 - h3));
        }
      }
    }
    return;
  }
  for (int64_t r = warp; r < n; r += nwarps) {
    const float4* row4 = reinterpret_cast<const float4*>(X + r * ldx);
    float4 v[NV];
    auto load_seg = [&](int seg) {
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int c = seg * 32 * NV + lane + 32 * i;
        v[i] = (4 * c < d) ? __ldg(row4 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    };
    float inv = 1.f;
    load_seg(0);
    if (NORMALIZE) {
      float s = 0.f;
      for (int seg = 0; seg < nseg; ++seg) {
        if (seg > 0) load_seg(seg);
#pragma unroll
        for (int i = 0; i < NV; ++i) s = fmaf(v[i].x, v[i].x, fmaf(v[i].y, v[i].y, fmaf(v[i].z, v[i].z, fmaf(v[i].w, v[i].w, s))));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const float nu = sqrtf(s);
      inv = (nu > 0.f) ? 1.f / nu : 0.f;
      if (lane == 0 && norms != nullptr) norms[r] = nu;
    }
    for (int seg = 0; seg < nseg; ++seg) {
      if (nseg > 1 && (seg > 0 || NORMALIZE)) load_seg(seg);   // registers hold the last segment read
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int c = seg * 32 * NV + lane + 32 * i;
        if (4 * c >= d) continue;
        const float u0 = v[i].x * inv, u1 = v[i].y * inv, u2 = v[i].z * inv, u3 = v[i].w * inv;
        const float h0 = __bfloat162float(__float2bfloat16_rn(u0)), h1 = __bfloat162float(__float2bfloat16_rn(u1));
        const float h2 = __bfloat162float(__float2bfloat16_rn(u2)), h3 = __bfloat162float(__float2bfloat16_rn(u3));
        *reinterpret_cast<uint2*>(L1 + r * dpad + 4 * c) = make_uint2(pack_bf16x2(h0, h1), pack_bf16x2(h2, h3));
        *reinterpret_cast<uint2*>(L2 + r * dpad + 4 * c) = make_uint2(pack_bf16x2(u0 - h0, u1 - h1), pack_bf16x2(u2 - h2, u3 - h3));
      }
    }
  }
}

__host__ __device__ __forceinline__ bool vec_rows(const float* X, int64_t ldx, int d, int dpad) {
  return (d & 3) == 0 && (ldx & 3) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0 && dpad == d;
}

// One warp per row: nu = ||x|| (optional), u = x / nu, u = hi + lo in bf16.  Rows warp, warp + nwarps, ...
template <bool NORMALIZE>
__device__ __forceinline__ void split_rows(const float* __restrict__ X, int64_t ldx, int64_t n, int d, int dpad,
                                           __nv_bfloat16* __restrict__ L1, __nv_bfloat16* __restrict__ L2,
                                           float* __restrict__ norms, int64_t warp, int64_t nwarps, int lane) {
  if (vec_rows(X, ldx, d, dpad)) {
    if (d <= 256) split_rows_vec<NORMALIZE, 2>(X, ldx, n, d, dpad, L1, L2, norms, warp, nwarps, lane);
    else if (d <= 512) split_rows_vec<NORMALIZE, 4>(X, ldx, n, d, dpad, L1, L2, norms, warp, nwarps, lane);
    else if (d <= 1024) split_rows_vec<NORMALIZE, 8>(X, ldx, n, d, dpad, L1, L2, norms, warp, nwarps, lane);
    else split_rows_vec<NORMALIZE, 16>(X, ldx, n, d, dpad, L1, L2, norms, warp, nwarps, lane);
    return;
  }
  // Other rows: a lane adds its squares over j = lane, lane + 32, ... with sixteen loads in flight, then converts eight
  // neighbouring elements at a time.
  for (int64_t r = warp; r < n; r += nwarps) {
    const float* row = X + r * ldx;
    float inv = 1.f;
    if (NORMALIZE) {
      float s = 0.f;
      for (int j0 = lane; j0 < d; j0 += 512) {
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = j0 + 32 * i < d ? row[j0 + 32 * i] : 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) s = fmaf(v[i], v[i], s);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const float nu = sqrtf(s);
      inv = (nu > 0.f) ? 1.f / nu : 0.f;
      if (lane == 0 && norms != nullptr) norms[r] = nu;
    }
#pragma unroll 2
    for (int j0 = lane * 8; j0 < dpad; j0 += 256) {
      float u[8];
#pragma unroll
      for (int p = 0; p < 8; ++p) u[p] = j0 + p < d ? row[j0 + p] : 0.f;
      uint32_t h[4], l[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float u0 = u[2 * p] * inv, u1 = u[2 * p + 1] * inv;
        const float h0 = __bfloat162float(__float2bfloat16_rn(u0));
        const float h1 = __bfloat162float(__float2bfloat16_rn(u1));
        h[p] = pack_bf16x2(h0, h1);
        l[p] = pack_bf16x2(u0 - h0, u1 - h1);
      }
      *reinterpret_cast<uint4*>(L1 + r * dpad + j0) = make_uint4(h[0], h[1], h[2], h[3]);
      *reinterpret_cast<uint4*>(L2 + r * dpad + j0) = make_uint4(l[0], l[1], l[2], l[3]);
    }
  }
}

template <bool NORMALIZE>
__global__ void __launch_bounds__(256) split_rows_kernel(const float* __restrict__ X, int64_t ldx, int64_t n, int d, int dpad,
                                                         __nv_bfloat16* __restrict__ L1, __nv_bfloat16* __restrict__ L2,
                                                         float* __restrict__ norms) {
  allow_successor();        // (every kernel behind waits for this one, and so for those ahead of it, before it writes or reads)
  wait_for_predecessor();   // it may write X, or read the limb buffers
  split_rows<NORMALIZE>(X, ldx, n, d, dpad, L1, L2, norms, (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5),
                        (int64_t)gridDim.x * (blockDim.x >> 5), threadIdx.x & 31);
}

// Rows of bf16, one warp per row: nu = ||x|| (optional) and the row's only limb.  Bound: HBM, 4 bytes per element (6 with the two
// limbs of x / nu).  Rows of at most 256 NV elements stay in registers between the two, all their loads in flight at once; longer
// rows are read a second time.  VEC: 16-byte loads (rows on the 16-byte grid).
template <int NV, bool VEC>
__global__ void __launch_bounds__(256) scale_rows_kernel(const __nv_bfloat16* __restrict__ X, int64_t ldx, int64_t n, int d, int dpad,
                                                         __nv_bfloat16* __restrict__ L1, float* __restrict__ norms) {
  allow_successor();
  wait_for_predecessor();   // it may write X, or read the limb buffer
  const int lane = threadIdx.x & 31;
  const int nseg = (dpad + 256 * NV - 1) / (256 * NV);
  for (int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < n; r += (int64_t)gridDim.x * (blockDim.x >> 5)) {
    const __nv_bfloat16* row = X + r * ldx;
    uint4 v[NV];
    auto load_seg = [&](int seg) {
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int j = (seg * NV + i) * 256 + lane * 8;
        if (VEC && j + 8 <= d) {
          v[i] = __ldg(reinterpret_cast<const uint4*>(row + j));
        } else {
          uint32_t w[4];
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            const uint32_t lo = j + 2 * p < d ? __bfloat16_as_ushort(row[j + 2 * p]) : 0u;
            const uint32_t hi = j + 2 * p + 1 < d ? __bfloat16_as_ushort(row[j + 2 * p + 1]) : 0u;
            w[p] = lo | (hi << 16);
          }
          v[i] = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
    };
    auto low = [](uint32_t w) { return __uint_as_float(w << 16); };
    auto high = [](uint32_t w) { return __uint_as_float(w & 0xffff0000u); };
    float down = 1.f;
    load_seg(0);
    if (norms != nullptr) {
      float s = 0.f;
      for (int seg = 0; seg < nseg; ++seg) {
        if (seg > 0) load_seg(seg);
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
          for (int p = 0; p < 4; ++p) s = fmaf(low(w[p]), low(w[p]), fmaf(high(w[p]), high(w[p]), s));
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const float nu = sqrtf(s);
      down = row_scale(nu).down;
      if (lane == 0) norms[r] = nu;
    }
    for (int seg = 0; seg < nseg; ++seg) {
      if (nseg > 1 && (seg > 0 || norms != nullptr)) load_seg(seg);   // registers hold the last segment read
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int j = (seg * NV + i) * 256 + lane * 8;
        if (j >= dpad) continue;
        const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
        uint32_t o[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) o[p] = pack_bf16x2(low(w[p]) * down, high(w[p]) * down);
        *reinterpret_cast<uint4*>(L1 + r * dpad + j) = make_uint4(o[0], o[1], o[2], o[3]);
      }
    }
  }
}

// MODE 0: idx.  MODE 1: idx + residual limbs + partial ||e||^2.  MODE 2: sign bits.  ONE: A has one limb.  (An instance of its own: with
// number, size and offsets of the stages at run time, calls of fp32 rows were slower, 300 rows of d = 384 mse b = 2 10.0 -> 10.4 us.)
template <int BN, int MODE, int BITS, int CTAS, bool ONE>
__global__ void __launch_bounds__(Cfg<BN, CTAS>::kThreads, 1)
quantize_gemm_kernel(const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmA2,
                     const __grid_constant__ CUtensorMap tmB1, const __grid_constant__ CUtensorMap tmB2,
                     const __grid_constant__ CUtensorMap tmE1, const __grid_constant__ CUtensorMap tmE2, GemmArgs a) {
  using C = Cfg<BN, CTAS>;
  constexpr int EPS = C::kEps;
  const int rank = CTAS == 2 ? (int)cluster_ctarank() : 0;   // CTA of the pair; rank 0 issues the MMAs
  const int64_t unit = blockIdx.x / CTAS, nunits = gridDim.x / CTAS;   // a unit = one CTA or one pair
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int stages = ONE ? C::kStages1 : C::kStages, stage_bytes = ONE ? C::kStageBytes1 : C::kStageBytes;
  constexpr int b_off = ONE ? BM * BK * 2 : 2 * BM * BK * 2;           // B's limbs in a stage
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kStages * C::kStageBytes);
  uint64_t* full = bars;                    // [stages]   TMA -> MMA
  uint64_t* empty = bars + stages;          // [stages]   MMA -> TMA
  uint64_t* tfull = bars + 2 * stages;      // [2]        MMA -> epilogue
  uint64_t* tempty = tfull + 2;             // [2]        epilogue -> MMA
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  // the centroids in shared memory: indexed by the code they are one wavefront per load, where the same index into
  // the kernel's constant arguments is replayed once per distinct code of the warp
  float* cs = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(bars) + 192);   // [16]
  unsigned char* stg = reinterpret_cast<unsigned char*>(bars) + 512;                    // [4 EPS][2048], 512-byte aligned
  if (MODE == 1 && threadIdx.x < 16) cs[threadIdx.x] = a.cb.c[threadIdx.x];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int num_kb = (a.K + BK - 1) / BK;
  const int64_t num_tiles = (int64_t)a.tiles_m * a.tiles_n;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 4 * EPS * CTAS);   // the leader's: the epilogue warps of both CTAs arrive
    }
    *abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmA1);
    tma_prefetch_desc(&tmA2);
    tma_prefetch_desc(&tmB1);
    tma_prefetch_desc(&tmB2);
  }
  if (warp == 1) {
    if (CTAS == 2) tmem_alloc_pair(tmem_slot, C::kTmemCols);
    else tmem_alloc(tmem_slot, C::kTmemCols);
  }
  tc_fence_before();
  if (CTAS == 2) cluster_sync();   // the partner's barriers exist before anything arrives on them
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  wait_for_predecessor();   // the operands are outputs of the kernel ahead; the outputs may be inputs of it
  allow_successor();        // (only now: a scan's successor may start reading the codes, see nscan::run)

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int64_t t = unit; t < num_tiles && ok; t += nunits) {
        const int m0 = ((int)(t / a.tiles_n) * CTAS + rank) * BM, n0 = (int)(t % a.tiles_n) * BN + rank * C::kBRows;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!(ok = mbar_wait_suspended(&empty[stage], phase ^ 1u, abort_flag, a.status))) break;
          unsigned char* sa = smem + stage * stage_bytes;
          if (CTAS == 2) {
            // both CTAs' bytes are counted on the leader's barrier, which the leader arms for both
            if (rank == 0) mbar_arrive_expect_tx(&full[stage], 2 * stage_bytes);
            tma_load_2d_pair(sa, &tmA1, &full[stage], kb * BK, m0);
            if (!ONE) tma_load_2d_pair(sa + BM * BK * 2, &tmA2, &full[stage], kb * BK, m0);
            tma_load_2d_pair(sa + b_off, &tmB1, &full[stage], kb * BK, n0);
            tma_load_2d_pair(sa + b_off + C::kBRows * BK * 2, &tmB2, &full[stage], kb * BK, n0);
          } else {
            mbar_arrive_expect_tx(&full[stage], stage_bytes);
            tma_load_2d(sa, &tmA1, &full[stage], kb * BK, m0);
            if (!ONE) tma_load_2d(sa + BM * BK * 2, &tmA2, &full[stage], kb * BK, m0);
            tma_load_2d(sa + b_off, &tmB1, &full[stage], kb * BK, n0);
            tma_load_2d(sa + b_off + BN * BK * 2, &tmB2, &full[stage], kb * BK, n0);
          }
          if (++stage == stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok) {
        // let copies already in flight land before the CTA's shared memory is given up
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc = instr_desc_bf16(BM * CTAS, BN);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      int64_t it = 0;
      for (int64_t t = unit; t < num_tiles && ok; t += nunits, ++it) {
        const uint32_t acc = (uint32_t)(it & 1), acc_phase = (uint32_t)((it >> 1) & 1);
        if (!(ok = mbar_wait_suspended(&tempty[acc], acc_phase ^ 1u, abort_flag, a.status))) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * C::kAccCols;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!(ok = mbar_wait_suspended(&full[stage], phase, abort_flag, a.status))) break;
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + stage * stage_bytes);
          const uint64_t a1 = smem_desc_sw128(sa), a2 = smem_desc_sw128(sa + BM * BK * 2);
          const uint64_t b1 = smem_desc_sw128(sa + b_off);
          const uint64_t b2 = smem_desc_sw128(sa + b_off + C::kBRows * BK * 2);
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k) {
            const uint64_t off = (uint64_t)((k * UMMA_K * 2) >> 4);   // 32 bytes per K step
            if (CTAS == 2) {
              umma_bf16_pair(d_tmem, a1 + off, b2 + off, idesc, (kb | k) != 0 ? 1u : 0u);   // hi * lo
              if (!ONE) umma_bf16_pair(d_tmem, a2 + off, b1 + off, idesc, 1u);              // lo * hi
              umma_bf16_pair(d_tmem, a1 + off, b1 + off, idesc, 1u);                        // hi * hi
            } else {
              umma_bf16(d_tmem, a1 + off, b2 + off, idesc, (kb | k) != 0 ? 1u : 0u);
              if (!ONE) umma_bf16(d_tmem, a2 + off, b1 + off, idesc, 1u);
              umma_bf16(d_tmem, a1 + off, b1 + off, idesc, 1u);
            }
          }
          // frees the stage (in both CTAs of a pair) once these MMAs have read it
          if (CTAS == 2) umma_commit_pair(&empty[stage]);
          else umma_commit(&empty[stage]);
          if (++stage == stages) {
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
  } else if (warp >= 2 + 4 * EPS) {
    // ------------------------------------------------------------ spare warps
    if (MODE == 2) {   // gamma = ||e|| from the rotate launch's partial sums, in the order of the columns
      // (eight rows of a lane at a time: with one, the loads' latency made this the longest part of the kernel at d = 128)
      const int64_t step = (int64_t)gridDim.x * NSPLIT * 32;
      for (int64_t r = ((int64_t)blockIdx.x * NSPLIT + (warp - 2 - 4 * EPS)) * 32 + lane; r < a.M; r += 8 * step) {
        float g2[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int t = 0; t < a.parts; ++t) {
#pragma unroll
          for (int i = 0; i < 8; ++i) g2[i] += r + i * step < a.M ? __ldcg(a.gpart + (int64_t)t * a.Mpad + r + i * step) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (r + i * step < a.M) a.gamma[r + i * step] = sqrtf(g2[i]);
      }
    }
    if constexpr (MODE == 0) {   // operand limbs of the next block of rows
      const GemmArgs::SplitTask& t = a.split;
      if (t.rows > 0) {
        const int64_t sw = (int64_t)blockIdx.x * NSPLIT + (warp - 2 - 4 * EPS), nsw = (int64_t)gridDim.x * NSPLIT;
        if (t.normalize) split_rows<true>(t.X, t.ldx, t.rows, t.d, t.dpad, t.L1, t.L2, t.norms, sw, nsw, lane);
        else split_rows<false>(t.X, t.ldx, t.rows, t.d, t.dpad, t.L1, t.L2, t.norms, sw, nsw, lane);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (4 x EPS warps: 4 TMEM lane groups x EPS column parts)
    const int lg = warp & 3;   // TMEM lane group this warp may read
    const int half = (warp - 2) >> 2;   // which part (of EPS) of the tile's columns this warp takes
    bool ok = true;
    int64_t it = 0;
    for (int64_t t = unit; t < num_tiles && ok; t += nunits, ++it) {
      const uint32_t acc = (uint32_t)(it & 1), acc_phase = (uint32_t)((it >> 1) & 1);
      const int tm = (int)(t / a.tiles_n), tn = (int)(t % a.tiles_n);
      const int64_t row = (int64_t)(tm * CTAS + rank) * BM + lg * 32 + lane;
      const int n0 = tn * BN;
      if (!(ok = mbar_wait_suspended(&tfull[acc], acc_phase, abort_flag, a.status))) break;
      tc_fence_after();
      const bool row_ok = row < a.M;
      bool zero_row = false;
      float back = 1.f;
      if ((MODE == 1 || ONE) && a.nu != nullptr && row_ok) {
        const float nu = __ldg(a.nu + row);
        zero_row = nu == 0.f;
        if (ONE) back = row_scale(nu).back;
      }
      float gsum = 0.f;
      uint32_t* out_row = reinterpret_cast<uint32_t*>(a.out + (size_t)(row_ok ? row : 0) * a.out_rb);
      const size_t row_words = a.out_rb / 4;
#pragma unroll 1
      for (int c = half * (BN / 32 / EPS); c < (half + 1) * (BN / 32 / EPS); ++c) {
        const int col0 = n0 + c * 32;
        if (col0 >= a.N) break;   // uniform across the CTA: nothing but zero padding beyond
        uint32_t v[32];
        tmem_ld32(tmem_base + ((uint32_t)(lg * 32) << 16) + acc * C::kAccCols + c * 32, v);
        tmem_ld_wait();
        if (MODE == 2) {
          uint32_t word = 0;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const bool bit = (__uint_as_float(v[i]) >= 0.f) && (col0 + i < a.N);
            word |= (bit ? 1u : 0u) << i;
          }
          const size_t w = (size_t)(col0 >> 5);
          if (a.nibble) {
            const size_t off = 16 * w;   // the group's four words of the combined row
            if (row_ok && off < a.nib_idx_rb + a.nib_qjl_rb) {
              uint4* dst = reinterpret_cast<uint4*>(off < a.nib_idx_rb ? a.nib_idx + (size_t)row * a.nib_idx_rb + off
                                                                       : a.nib_qjl + (size_t)row * a.nib_qjl_rb + (off - a.nib_idx_rb));
              uint4 cur = *dst;   // written by the rotate launch of the same block of rows
              cur.x |= spread_to_nibble_tops(word);
              cur.y |= spread_to_nibble_tops(word >> 8);
              cur.z |= spread_to_nibble_tops(word >> 16);
              cur.w |= spread_to_nibble_tops(word >> 24);
              *dst = cur;
            }
          } else if (row_ok && w < row_words) {
            out_row[w] = word;
          }
        } else {
          constexpr int NB = (1 << BITS) - 1;
          unsigned long long bitbuf = 0;
          int nb = 0, nw = 0;
          uint32_t words[BITS > 0 ? BITS : 1];
          uint32_t nibw[4] = {0u, 0u, 0u, 0u};
          uint32_t e1[16], e2[16];
#pragma unroll
          for (int i2 = 0; i2 < 16; ++i2) {
            float ehi[2] = {0.f, 0.f}, elo[2] = {0.f, 0.f};
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const int i = 2 * i2 + q;
              const float y = ONE ? __uint_as_float(v[i]) * back : __uint_as_float(v[i]);
              const bool col_ok = (col0 + i < a.N);
              int code = 0;
#pragma unroll
              for (int tix = 0; tix < NB; ++tix) code += (y > a.cb.t[tix]) ? 1 : 0;
              if (!col_ok) code = 0;
              if (BITS == 3 && MODE == 1) nibw[i >> 3] |= (uint32_t)code << (4 * (i & 7));
              if (BITS > 0) {
                bitbuf |= (unsigned long long)code << nb;
                nb += BITS;
                if (nb >= 32) {
                  words[nw++] = (uint32_t)bitbuf;
                  bitbuf >>= 32;
                  nb -= 32;
                }
              }
              if (MODE == 1) {
                const float e = (col_ok && !zero_row) ? (y - cs[code]) : 0.f;
                gsum = fmaf(e, e, gsum);
                ehi[q] = __bfloat162float(__float2bfloat16_rn(e));
                elo[q] = e - ehi[q];
              }
            }
            if (MODE == 1) {
              e1[i2] = pack_bf16x2(ehi[0], ehi[1]);
              e2[i2] = pack_bf16x2(elo[0], elo[1]);
            }
          }
          if (BITS == 3 && MODE == 1 && a.nibble) {
            const size_t off = 16 * (size_t)(col0 >> 5);
            if (row_ok && off < a.nib_idx_rb + a.nib_qjl_rb) {
              uint4* dst = reinterpret_cast<uint4*>(off < a.nib_idx_rb ? a.nib_idx + (size_t)row * a.nib_idx_rb + off
                                                                       : a.nib_qjl + (size_t)row * a.nib_qjl_rb + (off - a.nib_idx_rb));
              *dst = make_uint4(nibw[0], nibw[1], nibw[2], nibw[3]);
            }
          } else if (BITS > 0 && row_ok) {
            const size_t w0 = (size_t)(col0 >> 5) * BITS;
#pragma unroll
            for (int q = 0; q < BITS; ++q)
              if (w0 + q < row_words) out_row[w0 + q] = words[q];
          }
          if (MODE == 1) {
            // The warp's 32 rows x 32 columns of each residual limb go out as one TMA store: a row per thread, staged in
            // shared memory in the 64-byte swizzle (16-byte piece q of row r at q ^ ((r >> 1) & 3): four wavefronts per
            // instruction, the minimum for 512 bytes).  Stores straight from the registers were 16 bytes per lane at the
            // matrix's row stride, 32 lines per instruction, and cost a tenth of the whole quantiser.  Rows past M and
            // columns past N hold zeros or scratch inside the buffer's padding; the map clips columns past ldE.
            unsigned char* buf = stg + (warp - 2) * 2048;
            const int64_t row0 = row - lane;
            {   // (the map is Mpad rows high: a tile that overhangs the buffer is clipped by the store itself)
              const uint32_t sw = (uint32_t)((lane >> 1) & 3);
#pragma unroll
              for (int limb = 0; limb < 2; ++limb) {
                if (lane == 0) tma_store_wait_read();   // the previous box has left the buffer
                __syncwarp();
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  const uint32_t* e = limb == 0 ? e1 : e2;
                  *reinterpret_cast<uint4*>(buf + lane * 64 + ((q ^ sw) << 4)) = make_uint4(e[4 * q], e[4 * q + 1], e[4 * q + 2], e[4 * q + 3]);
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                  tma_store_2d(limb == 0 ? &tmE1 : &tmE2, buf, col0, (int)row0);
                  tma_store_commit();
                }
              }
            }
          }
        }
      }
      // accumulator fully read: hand the TMEM buffer back to the MMA warp
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CTAS == 2) mbar_arrive_leader(&tempty[acc]);
        else mbar_arrive(&tempty[acc]);
      }
      if (MODE == 1 && row_ok && EPS * tn + half < a.parts && TQ_DEVICE_CHECK(row < a.Mpad && tn < a.tiles_n, a.status))
        a.gpart[(int64_t)(EPS * tn + half) * a.Mpad + row] = gsum;
      // pad words past the last tile's columns (rows whose stride exceeds the tiles' coverage)
      if (a.nibble && tn == a.tiles_n - 1 && half == EPS - 1 && row_ok) {
        if (MODE == 1) {   // words of the combined row that no group of 32 coordinates owns
          const size_t wi = a.nib_idx_rb / 4, wq = a.nib_qjl_rb / 4;
          for (size_t w = (size_t)((a.N + 31) >> 5) * 4; w < wi + wq; ++w)
            (w < wi ? reinterpret_cast<uint32_t*>(a.nib_idx + (size_t)row * a.nib_idx_rb)[w]
                    : reinterpret_cast<uint32_t*>(a.nib_qjl + (size_t)row * a.nib_qjl_rb)[w - wi]) = 0u;
        }
      } else if (tn == a.tiles_n - 1 && half == EPS - 1 && row_ok) {
        constexpr int kBitsPerCoord = (MODE == 2) ? 1 : BITS;
        if (kBitsPerCoord > 0) {
          const size_t covered = (size_t)((a.N + 31) >> 5) * kBitsPerCoord;
          for (size_t w = covered; w < row_words; ++w) out_row[w] = 0u;
        }
      }
    }
    if (MODE == 1) {   // the residual stores of this warp have completed before the CTA gives up its shared memory
      if (lane == 0) tma_store_wait_all();
      __syncwarp();
    }
  }

  tc_fence_before();
  if (CTAS == 2) cluster_sync();   // neither CTA leaves while the partner may still arrive on its barriers or read its rows
  else __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    if (CTAS == 2) tmem_dealloc_pair(tmem_base, C::kTmemCols);
    else tmem_dealloc(tmem_base, C::kTmemCols);
  }
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// bf16 matrix [rows, cols] with row pitch `pitch` elements; box = 64 columns x box_rows, 128B swizzle.
bool make_map(CUtensorMap* map, const __nv_bfloat16* base, int64_t rows, int cols, int64_t pitch, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch * 2};
  const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// bf16 matrix [rows, cols] with row pitch `pitch` elements, for TMA stores of [32 rows x 32 columns] boxes staged in
// shared memory in the 64-byte swizzle.
bool make_store_map(CUtensorMap* map, __nv_bfloat16* base, int64_t rows, int64_t cols, int64_t pitch) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch * 2};
  const cuuint32_t box[2] = {32, 32};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Byte matrix [rows, row_bytes] with row pitch `pitch` bytes; box = box_bytes x box_rows; `swizzle` = 0 (plain
// rows in shared memory) or 32 / 64 / 128 (that swizzle span; box_bytes must not exceed it).
bool make_byte_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t row_bytes, uint64_t pitch,
                   uint32_t box_bytes, uint32_t box_rows, int swizzle) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)row_bytes, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch};
  const cuuint32_t box[2] = {(cuuint32_t)box_bytes, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUtensorMapSwizzle sw = swizzle == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                : swizzle == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                : swizzle == 32 ? CU_TENSOR_MAP_SWIZZLE_32B
                                                : CU_TENSOR_MAP_SWIZZLE_NONE;
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_half_map(CUtensorMap* map, const __half* base, int64_t rows, int cols, int64_t pitch, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch * 2};
  const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_store_map_f32(CUtensorMap* map, float* base, int64_t rows, int64_t cols, int64_t pitch) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch * 4};
  const cuuint32_t box[2] = {16, 32};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int sm_count() {
  static std::atomic<int> cached{0};   // all devices of a process are taken to be alike
  int sms = cached.load(std::memory_order_relaxed);
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cached.store(sms, std::memory_order_relaxed);
  }
  return sms;
}

namespace {

template <int BN, int MODE, int BITS, int CTAS, bool ONE>
cudaError_t launch_gemm_t(const CUtensorMap& a1, const CUtensorMap& a2, const CUtensorMap& b1, const CUtensorMap& b2,
                          const GemmArgs& args, cudaStream_t st) {
  auto kern = quantize_gemm_kernel<BN, MODE, BITS, CTAS, ONE>;
  using C = Cfg<BN, CTAS>;
  // function attributes are per device: remember the devices this launcher has prepared
  static std::atomic<unsigned long long> attr_devices{0};   // written by any thread that launches
  int attr_dev = 0;
  if (cudaGetDevice(&attr_dev) != cudaSuccess) return cudaErrorInvalidDevice;
  if (attr_dev >= 64 || !((attr_devices.load(std::memory_order_relaxed) >> attr_dev) & 1ull)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
    if (e != cudaSuccess) return e;
    if (attr_dev < 64) attr_devices.fetch_or(1ull << attr_dev, std::memory_order_relaxed);
  }
  const int64_t tiles = (int64_t)args.tiles_m * args.tiles_n;   // tiles_m counts rows of BM * CTAS
  const int units = (int)std::min<int64_t>(tiles, sm_count() / CTAS);
  count_launches(1);
  // the store maps of the residual limbs (MODE 1); any valid map otherwise
  const CUtensorMap& e1 = args.store_e1 ? *args.store_e1 : a1;
  const CUtensorMap& e2 = args.store_e2 ? *args.store_e2 : a2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(units * CTAS));
  cfg.blockDim = dim3(C::kThreads);
  cfg.dynamicSmemBytes = C::kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CTAS;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CTAS == 1 ? 1 : 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, a1, a2, b1, b2, e1, e2, args);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int BN, int MODE, int CTAS, bool ONE>
cudaError_t launch_gemm_bits(int bits, const CUtensorMap& a1, const CUtensorMap& a2, const CUtensorMap& b1,
                             const CUtensorMap& b2, const GemmArgs& args, cudaStream_t st) {
  if constexpr (MODE == 2) {
    return launch_gemm_t<BN, 2, 1, CTAS, false>(a1, a2, b1, b2, args, st);
  } else {
    switch (bits) {
      case 0: return launch_gemm_t<BN, MODE, 0, CTAS, ONE>(a1, a2, b1, b2, args, st);
      case 1: return launch_gemm_t<BN, MODE, 1, CTAS, ONE>(a1, a2, b1, b2, args, st);
      case 2: return launch_gemm_t<BN, MODE, 2, CTAS, ONE>(a1, a2, b1, b2, args, st);
      case 3: return launch_gemm_t<BN, MODE, 3, CTAS, ONE>(a1, a2, b1, b2, args, st);
      default: return launch_gemm_t<BN, MODE, 4, CTAS, ONE>(a1, a2, b1, b2, args, st);
    }
  }
}

template <int MODE, bool ONE = false>
cudaError_t launch_gemm(const Tile& t, int bits, const CUtensorMap& a1, const CUtensorMap& a2, const MatrixLimbs& b,
                        const GemmArgs& args, cudaStream_t st) {
  if constexpr (MODE != 2 && !ONE)
    if (args.one_limb) return launch_gemm<MODE, true>(t, bits, a1, a2, b, args, st);
  const int box = t.bn / t.ctas / 32 - 1;   // maps by the rows of B that a CTA loads
  const CUtensorMap &b1 = b.map_hi[box], &b2 = b.map_lo[box];
  if (t.ctas == 1) {
    if (t.bn == 128) return launch_gemm_bits<128, MODE, 1, ONE>(bits, a1, a2, b1, b2, args, st);
    return launch_gemm_bits<64, MODE, 1, ONE>(bits, a1, a2, b1, b2, args, st);
  }
  switch (t.bn) {
    case 128: return launch_gemm_bits<128, MODE, 2, ONE>(bits, a1, a2, b1, b2, args, st);
    case 192: return launch_gemm_bits<192, MODE, 2, ONE>(bits, a1, a2, b1, b2, args, st);
    default: return launch_gemm_bits<256, MODE, 2, ONE>(bits, a1, a2, b1, b2, args, st);
  }
}

}  // namespace

bool supported(int d) { return d >= 128 && encode_fn() != nullptr; }

cudaError_t build_matrix_limbs(const float* dM, int rows, int d, int dpad, MatrixLimbs* out) {
  out->hi = out->lo = nullptr;
  const size_t bytes = (size_t)rows * dpad * sizeof(__nv_bfloat16);
  cudaError_t e = cudaMalloc(&out->hi, bytes);
  if (e != cudaSuccess) return e;
  e = cudaMalloc(&out->lo, bytes);
  if (e != cudaSuccess) return e;
  const int blocks = std::min((rows + 7) / 8, sm_count() * 8);
  split_rows_kernel<false><<<blocks, 256>>>(dM, d, rows, d, dpad, out->hi, out->lo, nullptr);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  for (int i = 0; i < kBoxes; ++i)
    if (!make_map(&out->map_hi[i], out->hi, rows, d, dpad, 32 * (i + 1)) || !make_map(&out->map_lo[i], out->lo, rows, d, dpad, 32 * (i + 1)))
      return cudaErrorInvalidValue;
  return cudaSuccess;
}

void free_matrix_limbs(MatrixLimbs* m) {
  cudaFree(m->hi);
  cudaFree(m->lo);
  m->hi = m->lo = nullptr;
}

// CTA pairs can be switched off (TQ_GEMM_PAIRS=0) to compare the two kernels on one machine.
bool pair_tiles_enabled() {
  static const bool on = [] {
    const char* e = std::getenv("TQ_GEMM_PAIRS");
    return e == nullptr || e[0] != '0';
  }();
  return on;
}

// Tile of a block of rows: the one with the least waves x time.  Every output is the same sum in the same order on all of them,
// so the codes do not depend on it.  Time of a k-block of 64 in units of 10 ns, all SMs busy (d = 768 to 3072): 62 for 128 x 64
// on one CTA, and on a pair 68, 93 and 120 for 256 x 128, 192 and 256 (the rule takes a little more for the narrow ones: under
// the power limit of a long call they lose 5 to 20 %).  The wider the tile, the fewer operand bytes per MMA, so 256 columns win
// wherever there are waves enough, and narrower tiles where a wave would leave SMs idle (TQ_PROD, us: d = 3072, 1,000 rows: 145,
// 113 and 129 with 128, 192 and 256 columns; 50,000 rows: 4,287, 3,963 and 3,813; d = 1536, 128 rows: 42 with 64 columns, 62
// with 256).  d <= 128: one tile is the whole row.  *time: waves x time.
Tile pick_tile(int64_t rows, int d, int64_t* time = nullptr) {
  if (d <= 128) return {128, 1};
  static constexpr struct { Tile t; int time; } kChoices[] = {{{256, 2}, 120}, {{192, 2}, 96}, {{128, 2}, 72}, {{64, 1}, 64}};
  Tile best = {64, 1};
  int64_t least = INT64_MAX;
  for (const auto& c : kChoices) {
    if (c.t.ctas == 2 && !pair_tiles_enabled()) continue;
    const int64_t tiles = ((rows + BM * c.t.ctas - 1) / (BM * c.t.ctas)) * ((d + c.t.bn - 1) / c.t.bn);
    const int units = sm_count() / c.t.ctas;
    const int64_t cost = (tiles + units - 1) / units * c.time;
    if (cost < least) {
      least = cost;
      best = c.t;
    }
  }
  if (time != nullptr) *time = least;
  return best;
}

// Partial sums of e^2 per row: room for four per 256 columns.
int gamma_parts(int d) { return 4 * ((d + 255) / 256); }

size_t scratch_bytes_per_row(const tq_plan* plan) {
  size_t per = (size_t)plan->dpad * 2 * 2 + sizeof(float);                            // X limbs + nu
  if (plan->mode == TQ_PROD) per += (size_t)plan->dpad * 2 * 2 + (size_t)gamma_parts(plan->d) * sizeof(float);  // E limbs + partial sums
  return per;
}

int quantize(const tq_plan* plan, const void* X, int x_dtype, int64_t n, int64_t ldx, uint8_t* idx, uint8_t* qjl,
             float* gamma, float* norms, void* scratch, size_t scratch_bytes, cudaStream_t st, const char* who) {
  const int d = plan->d, dpad = plan->dpad;
  const bool prod = plan->mode == TQ_PROD;
  const size_t per_row = scratch_bytes_per_row(plan);
  int64_t R = (int64_t)(scratch_bytes / per_row) / BM * BM;
  R = std::min<int64_t>(R, round_up64(n, BM));
  TQ_REQUIRE(R >= BM, TQ_ERR_WORKSPACE, "%s: scratch of %zu bytes cannot hold one block of %d rows", who, scratch_bytes, BM);
  // TQ_MSE: the operand limbs of block i + 1 may be prepared by spare warps of the rotate launch of block i; the scratch is then
  // used as two half-size sets written and read in turn (when the data spans more than one block and each half still holds a
  // tile).
  // Two warps per CTA keep up only while the GEMM gives them time: its work per row grows with d^2, theirs with d.
  // Measured per 10^6 rows with the CTA-pair GEMMs: TQ_MSE d = 1536 10.1 ms with them against 10.6 without; beside the project
  // launch of TQ_PROD they lost (d = 1536: 22.1 against 21.5 ms, d = 3072 alike), so it has none; at d = 1024 and below the
  // spare warps were the critical path for both.
  // Rows of bf16 or off the 16-byte grid are the critical path at every d (11,734 bf16 rows of d = 1536: 167 us and more with
  // the spare warps, 136 with a launch of their own).
  const bool overlap = !prod && d >= 1536 && x_dtype == TQ_F32 && vec_rows(static_cast<const float*>(X), ldx, d, dpad);
  // A call that fits one block is cut in two for this where the half of the preparation that it hides (at 6 TB/s) takes longer
  // than the waves that it adds and a launch (5 us): 300 rows of d = 1536 in two halves took 94 us, 20 in one.
  auto halves_pay = [&] {
    int64_t one = 0, half = 0;
    pick_tile(R, d, &one);
    pick_tile(R / 2 / BM * BM, d, &half);
    return 0.01 * (double)((d + BK - 1) / BK) * (double)(2 * half - one) + 5.0 < 0.5 * (double)n * d * 8 / 6e6;
  };
  const bool pingpong = overlap && n > R / 2 / BM * BM && R / 2 >= BM && (n > R || halves_pay());
  const int64_t Rbuf = R;   // rows the carved buffers hold in all
  if (pingpong) R = R / 2 / BM * BM;
  // carve the scratch (every part is a multiple of 256 bytes because Rbuf is a multiple of 128)
  char* p = static_cast<char*>(scratch);
  __nv_bfloat16* XL1 = reinterpret_cast<__nv_bfloat16*>(p); p += (size_t)Rbuf * dpad * 2;
  __nv_bfloat16* XL2 = reinterpret_cast<__nv_bfloat16*>(p); p += (size_t)Rbuf * dpad * 2;
  __nv_bfloat16 *EL1 = nullptr, *EL2 = nullptr;
  float* gpart = nullptr;
  if (prod) {
    EL1 = reinterpret_cast<__nv_bfloat16*>(p); p += (size_t)Rbuf * dpad * 2;
    EL2 = reinterpret_cast<__nv_bfloat16*>(p); p += (size_t)Rbuf * dpad * 2;
    gpart = reinterpret_cast<float*>(p); p += (size_t)Rbuf * gamma_parts(d) * sizeof(float);
  }
  // limb buffers of block number b
  auto limbs1 = [&](int64_t b) { return XL1 + (pingpong && (b & 1) ? (size_t)R * dpad : 0); };
  auto limbs2 = [&](int64_t b) { return XL2 + (pingpong && (b & 1) ? (size_t)R * dpad : 0); };
  const size_t xsz = (x_dtype == TQ_F32) ? 4 : 2;
  auto launch_split = [&](int64_t r0, cudaStream_t s) -> cudaError_t {
    const int64_t rows = std::min(R, n - r0);
    const void* Xc = static_cast<const char*>(X) + (size_t)r0 * ldx * xsz;
    float* nu_out = norms ? norms + r0 : nullptr;
    const int blocks = (int)std::min<int64_t>((rows + 7) / 8, (int64_t)sm_count() * 8);
    __nv_bfloat16 *L1 = limbs1(r0 / R), *L2 = limbs2(r0 / R);
    // A grid of more than one wave is launched plainly: as a programmatic dependent its first blocks settle wherever the kernel
    // ahead drains first, and the uneven rest costs more than the launch gap saves (200,000 rows of d = 200: 135 us a call, 123
    // plain).
    auto go = [&](auto kern, auto... args) -> cudaError_t {
      if (blocks <= 2 * sm_count()) return launch_dependent(kern, dim3((unsigned)blocks), dim3(256), 0, s, args...);
      kern<<<blocks, 256, 0, s>>>(args...);
      return cudaGetLastError();
    };
    cudaError_t e;
    if (x_dtype == TQ_F32) {
      const float* x = static_cast<const float*>(Xc);
      e = norms ? go(split_rows_kernel<true>, x, ldx, rows, d, dpad, L1, L2, nu_out) : go(split_rows_kernel<false>, x, ldx, rows, d, dpad, L1, L2, nu_out);
    } else {
      const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(Xc);
      const bool vec = ldx % 8 == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0;
      auto pick = [&](auto nv) {
        constexpr int NV = decltype(nv)::value;
        return vec ? go(scale_rows_kernel<NV, true>, x, ldx, rows, d, dpad, L1, nu_out) : go(scale_rows_kernel<NV, false>, x, ldx, rows, d, dpad, L1, nu_out);
      };
      e = d <= 256 ? pick(std::integral_constant<int, 1>()) : d <= 1024 ? pick(std::integral_constant<int, 4>()) : pick(std::integral_constant<int, 12>());
    }
    count_launches(1);
    return e;
  };
  for (int64_t r0 = 0; r0 < n; r0 += R) {
    const int64_t rows = std::min(R, n - r0);
    float* nu_out = norms ? norms + r0 : nullptr;
    // 1. nu, u = x / nu, bf16 limbs of u: by a launch of its own, or by the spare warps of the previous block's rotate launch
    if (r0 == 0 || !pingpong) TQ_CHECK_CUDA(launch_split(r0, st), who);
    __nv_bfloat16 *XLc1 = limbs1(r0 / R), *XLc2 = limbs2(r0 / R);
    auto next_block_task = [&](GemmArgs& ga) {
      ga.split.X = static_cast<const float*>(X) + (r0 + R) * ldx;
      ga.split.ldx = ldx;
      ga.split.rows = std::min(R, n - (r0 + R));
      ga.split.d = d;
      ga.split.dpad = dpad;
      ga.split.normalize = norms ? 1 : 0;
      ga.split.L1 = limbs1(r0 / R + 1);
      ga.split.L2 = limbs2(r0 / R + 1);
      ga.split.norms = norms ? norms + r0 + R : nullptr;
    };

    CUtensorMap mA1, mA2;
    TQ_REQUIRE(make_map(&mA1, XLc1, rows, d, dpad, BM) && make_map(&mA2, XLc2, rows, d, dpad, BM), TQ_ERR_CUDA,
               "%s: cuTensorMapEncodeTiled failed", who);
    GemmArgs g;
    g.M = rows;
    g.N = d;
    g.K = d;
    const Tile tile = pick_tile(rows, d);
    g.tiles_m = (int)((rows + BM * tile.ctas - 1) / (BM * tile.ctas));
    g.tiles_n = (d + tile.bn - 1) / tile.bn;
    g.cb = plan->cb;
    g.out = idx ? idx + (size_t)r0 * plan->idx_row_bytes : nullptr;
    g.out_rb = plan->idx_row_bytes;
    g.E1 = EL1;
    g.E2 = EL2;
    g.ldE = dpad;
    CUtensorMap sE1, sE2;
    g.store_e1 = g.store_e2 = nullptr;
    if (prod) {
      TQ_REQUIRE(make_store_map(&sE1, EL1, R, dpad, dpad) && make_store_map(&sE2, EL2, R, dpad, dpad), TQ_ERR_CUDA,
                 "%s: cuTensorMapEncodeTiled failed (residual stores)", who);
      g.store_e1 = &sE1;
      g.store_e2 = &sE2;
    }
    g.gpart = gpart;
    g.gamma = gamma ? gamma + r0 : nullptr;
    g.parts = d <= 128 ? 4 : (d + 63) / 64;   // per epilogue warp: 32 columns of a tile that is the whole row, else 64
    g.Mpad = R;
    g.nu = nu_out;
    g.one_limb = x_dtype == TQ_F32 ? 0 : 1;
    g.split.rows = 0;
    g.nibble = (plan->layout == TQ_LAYOUT_NIBBLE) ? 1 : 0;
    g.nib_idx = idx ? idx + (size_t)r0 * plan->idx_row_bytes : nullptr;
    g.nib_qjl = qjl ? qjl + (size_t)r0 * plan->qjl_row_bytes : nullptr;
    g.nib_idx_rb = plan->idx_row_bytes;
    g.nib_qjl_rb = plan->qjl_row_bytes;
    g.status = plan->d_status;
    // 2. y = Pi u, idx (+ residual limbs and partial norms)
    if (!prod) {
      if (pingpong && r0 + R < n) next_block_task(g);
      TQ_CHECK_CUDA(launch_gemm<0>(tile, plan->mse_bits, mA1, mA2, plan->pi_limbs, g, st), who);
      continue;
    }
    TQ_CHECK_CUDA(launch_gemm<1>(tile, plan->mse_bits, mA1, mA2, plan->pi_limbs, g, st), who);
    // 3. qjl = sign(S' e), gamma = ||e||
    CUtensorMap mE1, mE2;
    TQ_REQUIRE(make_map(&mE1, EL1, rows, d, dpad, BM) && make_map(&mE2, EL2, rows, d, dpad, BM), TQ_ERR_CUDA,
               "%s: cuTensorMapEncodeTiled failed", who);
    g.out = qjl + (size_t)r0 * plan->qjl_row_bytes;
    g.out_rb = plan->qjl_row_bytes;
    TQ_CHECK_CUDA(launch_gemm<2>(tile, 1, mE1, mE2, plan->sp_limbs, g, st), who);
  }
  return TQ_OK;
}

}  // namespace tc
}  // namespace tq
