// Quantiser for short vectors (d = 32, 64, 96; the channel groups of a KV cache): Quant_mse / Quant_prod of Algorithms 1 and 2 in ONE
// launch.  A CTA takes 64 rows through the whole chain -- norm, rotation, nearest centroid, packing, residual, gamma, QJL
// projection, signs -- with the rows, the residuals and both matrices in shared memory.
//
// Every sum is an fp32 chain in the order of the CUDA-core GEMM and the row-norm kernel that other small dimensions use
// (products added in ascending order; a lane's squares, then the xor butterfly), so the codes are the same bits.  A version on
// fp16 limbs and mma.sync took 42 us for the prompt below, but its codes differed in a few coordinates at the boundaries, and
// forming those rows again with these chains brought it to 73 us.
//
// Bound: instruction issue (0.69 per scheduler and cycle), two thirds of it the 2 (TQ_MSE 1) n d^2 FMAs.  A thread owns 8 rows x
// 4 columns: per four k, 8 + 4 16-byte reads for 128 FMAs, the reads of a warp's two row groups being broadcasts.  Measured, n =
// 32,768, d = 64, bf16: TQ_PROD b_m = 2 48 -> 20 us, TQ_MSE b = 3 34 -> 13 us; the four calls of a 4,096-token prompt 229 -> 68.
// No gain: pairs of FMAs in one instruction (fma.rn.f32x2), calls scheduled ahead as programmatic dependents.
#include <algorithm>
#include <atomic>

#include "tq_quantize_small.h"
#include "tq_quantize_tc.h"

namespace tq {
namespace sq {

namespace {

constexpr int RT = 64;                                    // rows per CTA
template <int D>
struct Cfg {
  static constexpr int kThreads = 8 * (D / 4);            // ty = 0..7 x one thread per four columns
  static constexpr int kStride = D + 4;                   // floats between rows: the row groups of a warp fall into different banks
  static constexpr int smem(bool prod) { return (RT * kStride + (prod ? 2 : 1) * D * D + 2 * RT) * (int)sizeof(float); }
};

struct Args {
  const void* X;
  int64_t n, ldx;
  int vec;                          // rows are 16-byte aligned
  const float* backt;               // [D, ncols]: row k holds Pi[:, k]
  int ncols;
  const float* spt;                 // [D, D]: row k holds S'[:, k]
  Codebook cb;
  uint8_t* idx;
  uint8_t* qjl;
  float* gamma;
  float* norms;                     // nullable: rows are taken as unit-norm
  int idx_rb, qjl_rb;
};

template <bool BF16>
__device__ __forceinline__ float element(const void* X, int64_t at) {
  if (BF16) return __bfloat162float(static_cast<const __nv_bfloat16*>(X)[at]);
  return __ldg(static_cast<const float*>(X) + at);
}
// Sum of squares of one row of xs by four threads (j = 0..3 of a lane quad), added as a warp with element 32 w + l in lane l
// would: per lane in ascending order, then the xor butterfly over lane distances 16, 8, 4, 2, 1.  Whole quads call it.
template <int D>
__device__ __forceinline__ float row_squares(const float* row, int j) {
  float s[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    s[m] = 0.f;
#pragma unroll
    for (int w = 0; w < D / 32; ++w) {
      const float x = row[32 * w + 4 * m + j];
      s[m] = fmaf(x, x, s[m]);
    }
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1)
#pragma unroll
    for (int m = 0; m < o; ++m) s[m] += s[m + o];
  s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
  return s[0] + __shfl_xor_sync(0xffffffffu, s[0], 1);
}
// Four BITS-bit codes of coordinates 4 t .. 4 t + 3 (t = lane & 7) of a group of 32 -> the group's BITS words.  Returns one word
// and its number in `which` (-1: this lane has none).
template <int BITS>
__device__ __forceinline__ uint32_t group_words(uint32_t four, int t, int& which) {
  if (BITS == 3) {   // pairs of lanes hold 24 bits; word k = bits of pairs k and k + 1
    const uint32_t other = __shfl_xor_sync(0xffffffffu, four, 1);
    const uint32_t pair = (t & 1) ? other | (four << 12) : four | (other << 12);
    const uint32_t next = __shfl_down_sync(0xffffffffu, pair, 2);
    const int k = t >> 1;
    which = (t & 1) == 0 && k < 3 ? k : -1;
    return (pair >> (8 * k)) | (next << ((24 - 8 * k) & 31));
  }
  constexpr int LANES = 8 / BITS;   // lanes of one word
  uint32_t v = four << (4 * BITS * (t & (LANES - 1)));
#pragma unroll
  for (int o = 1; o < LANES; o <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
  which = (t & (LANES - 1)) == 0 ? t / LANES : -1;
  return v;
}

template <int D, int BITS, bool PROD, bool BF16>
__global__ void __launch_bounds__(Cfg<D>::kThreads) small_quantize_kernel(Args a) {
  constexpr int T = Cfg<D>::kThreads, TX = D / 4, S = Cfg<D>::kStride;
  extern __shared__ __align__(16) float smem[];
  float* xs = smem;                        // [RT][S]  rows, later the residuals
  float* bs = xs + RT * S;                 // [D][D]   Pi^T
  float* ss = bs + D * D;                  // [D][D]   S'^T (PROD)
  float* vs = bs + (PROD ? 2 : 1) * D * D; // [RT]     nu as the comparisons take it (1 for a zero row)
  float* is = vs + RT;                     // [RT]     1 / nu (-1 for a zero row; 0 where the norm has overflowed)
  const int tid = threadIdx.x, lane = tid & 31;
  const int tx = tid % TX, ty = tid / TX, t8 = lane & 7;
  const int64_t row0 = (int64_t)blockIdx.x * RT;
  {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(bs);
    for (int i = tid; i < D * TX; i += T)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * i), "l"(a.backt + (size_t)(i / TX) * a.ncols + 4 * (i % TX)) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (PROD) {   // wanted only after the first product
      for (int i = tid; i < D * TX; i += T)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 4 * D * D + 16 * i), "l"(a.spt + 4 * i) : "memory");
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
  }
  // ---- rows to shared memory, then their norms
  constexpr int PE = BF16 ? 8 : 4;   // elements of a 16-byte piece
#pragma unroll
  for (int p = tid; p < RT * D / PE; p += T) {
    const int r = p / (D / PE), c = PE * (p % (D / PE));
    const int64_t at = min(row0 + r, a.n - 1) * a.ldx + c;   // rows past the end repeat the last one
    float x[PE];
    if (a.vec) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(a.X) + at * (16 / PE)));
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (BF16) {
          x[2 * i] = __uint_as_float(w[i] << 16);
          x[(2 * i + 1) % PE] = __uint_as_float(w[i] & 0xffff0000u);
        } else {
          x[i] = __uint_as_float(w[i]);
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < PE; ++i) x[i] = element<BF16>(a.X, at + i);
    }
#pragma unroll
    for (int i = 0; i < PE; i += 4) *reinterpret_cast<float4*>(xs + r * S + c + i) = make_float4(x[i], x[i + 1], x[i + 2], x[i + 3]);
  }
  __syncthreads();
#pragma unroll
  for (int r = tid >> 2; r < RT; r += T / 4) {   // whole warps
    float nu = 1.f;
    if (a.norms != nullptr) nu = sqrtf(row_squares<D>(xs + r * S, tid & 3));
    if ((tid & 3) == 0) {
      if (a.norms != nullptr && row0 + r < a.n) a.norms[row0 + r] = nu;
      vs[r] = nu > 0.f ? nu : 1.f;
      is[r] = nu > 0.f ? 1.f / nu : -1.f;
    }
  }
  if (PROD) asm volatile("cp.async.wait_group 1;" ::: "memory");
  else asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();

  // acc[i][c] = sum_k xs[8 i + ty][k] m[k][4 tx + c], k ascending
  float acc[8][4];
  auto product = [&](const float* m) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][c] = 0.f;
#pragma unroll 2
    for (int k = 0; k < D; k += 4) {
      float4 b[4];
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) b[kk] = *reinterpret_cast<const float4*>(m + (k + kk) * D + 4 * tx);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 x = *reinterpret_cast<const float4*>(xs + (8 * i + ty) * S + k);
        const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          acc[i][0] = fmaf(xv[kk], b[kk].x, acc[i][0]);
          acc[i][1] = fmaf(xv[kk], b[kk].y, acc[i][1]);
          acc[i][2] = fmaf(xv[kk], b[kk].z, acc[i][2]);
          acc[i][3] = fmaf(xv[kk], b[kk].w, acc[i][3]);
        }
      }
    }
  };
  product(bs);
  if (PROD) __syncthreads();   // the rows are read: residuals may take their place

  // ---- nearest centroid, packed codes, residual
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = 8 * i + ty;
    const int64_t row = row0 + r;
    const float v = vs[r], inv = is[r];
    uint32_t four = 0u;
    float e[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float y = acc[i][c];
      int code = 0;
      float cent = a.cb.c[0];
#pragma unroll
      for (int t = 0; t < (1 << BITS) - 1; ++t) {
        const bool above = y > a.cb.t[t] * v;
        code += above ? 1 : 0;
        if (PROD) cent = above ? a.cb.c[t + 1] : cent;
      }
      four |= (uint32_t)code << (BITS * c);
      if (PROD) e[c] = inv >= 0.f ? fmaf(y, inv, -cent) : 0.f;
    }
    if (BITS > 0) {
      int which;
      const uint32_t word = group_words<BITS == 0 ? 1 : BITS>(four, t8, which);
      uint32_t* dst = reinterpret_cast<uint32_t*>(a.idx + (size_t)row * a.idx_rb);
      if (row < a.n) {
        if (which >= 0) dst[(tx >> 3) * BITS + which] = word;
        if (D * BITS / 32 + tx < a.idx_rb / 4) dst[D * BITS / 32 + tx] = 0u;   // pad words (fewer than four)
      }
    }
    if (PROD) *reinterpret_cast<float4*>(xs + r * S + 4 * tx) = make_float4(e[0], e[1], e[2], e[3]);
  }
  if constexpr (PROD) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    // ---- gamma = |r|, then z = sign(S' r)
#pragma unroll
    for (int r = tid >> 2; r < RT; r += T / 4) {
      const float s = row_squares<D>(xs + r * S, tid & 3);
      if ((tid & 3) == 0 && row0 + r < a.n) a.gamma[row0 + r] = sqrtf(s);
    }
    product(ss);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int64_t row = row0 + 8 * i + ty;
      uint32_t four = 0u;
#pragma unroll
      for (int c = 0; c < 4; ++c) four |= acc[i][c] >= 0.f ? 1u << c : 0u;
      int which;
      const uint32_t word = group_words<1>(four, t8, which);
      uint32_t* dst = reinterpret_cast<uint32_t*>(a.qjl + (size_t)row * a.qjl_rb);
      if (row < a.n) {
        if (which == 0) dst[tx >> 3] = word;
        if (D / 32 + tx < a.qjl_rb / 4) dst[D / 32 + tx] = 0u;
      }
    }
  }
}

template <int D, int BITS, bool PROD, bool BF16>
cudaError_t launch(const Args& a, cudaStream_t st, int device) {
  auto kern = small_quantize_kernel<D, BITS, PROD, BF16>;
  constexpr int smem = Cfg<D>::smem(PROD);
  if (smem > 48 * 1024) {
    static std::atomic<unsigned long long> attr_devices{0};   // devices whose function attribute has been set
    if (device >= 64 || !((attr_devices.load(std::memory_order_relaxed) >> device) & 1ull)) {
      const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e != cudaSuccess) return e;
      if (device < 64) attr_devices.fetch_or(1ull << device, std::memory_order_relaxed);
    }
  }
  const int64_t ctas = (a.n + RT - 1) / RT;
  if (ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  kern<<<(unsigned)ctas, Cfg<D>::kThreads, smem, st>>>(a);
  count_launches(1);
  return cudaGetLastError();
}

template <int D, bool PROD, bool BF16>
cudaError_t launch_bits(const Args& a, int bits, cudaStream_t st, int device) {
  switch (bits) {
    case 0: return launch<D, 0, true, BF16>(a, st, device);   // (TQ_MSE has at least one bit)
    case 1: return launch<D, 1, PROD, BF16>(a, st, device);
    case 2: return launch<D, 2, PROD, BF16>(a, st, device);
    case 3: return launch<D, 3, PROD, BF16>(a, st, device);
    default: return launch<D, 4, PROD, BF16>(a, st, device);
  }
}

template <int D>
cudaError_t launch_d(const Args& a, int bits, bool prod, bool bf16, cudaStream_t st, int device) {
  if (prod) return bf16 ? launch_bits<D, true, true>(a, bits, st, device) : launch_bits<D, true, false>(a, bits, st, device);
  return bf16 ? launch_bits<D, false, true>(a, bits, st, device) : launch_bits<D, false, false>(a, bits, st, device);
}

__global__ void transpose_kernel(const float* __restrict__ in, int d, float* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d * d; i += gridDim.x * blockDim.x) out[i] = in[(i % d) * d + i / d];
}

}  // namespace

cudaError_t plan_init(tq_plan* plan) {
  auto& s = plan->sq;
  s.ok = 0;
  const int d = plan->d;
  if (d % 32 != 0 || d > 96) return cudaSuccess;
  if (plan->mode == TQ_PROD) {
    cudaError_t e = cudaMalloc(&s.spt, (size_t)d * d * sizeof(float));
    if (e != cudaSuccess) return e;
    transpose_kernel<<<16, 256>>>(plan->dSp, d, s.spt);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  s.ok = 1;
  return cudaSuccess;
}

void plan_free(tq_plan* plan) { cudaFree(plan->sq.spt); }

int quantize(const tq_plan* plan, const void* X, int x_dtype, int64_t n, int64_t ldx, uint8_t* idx, uint8_t* qjl, float* gamma,
             float* norms, cudaStream_t st, const char* who) {
  Args a;
  a.X = X;
  a.n = n;
  a.ldx = ldx;
  a.vec = (ldx * (x_dtype == TQ_F32 ? 4 : 2)) % 16 == 0;
  a.backt = plan->dBackT;
  a.ncols = plan->ncat * plan->dpad;
  a.spt = plan->sq.spt;
  a.cb = plan->cb;
  a.idx = idx;
  a.qjl = qjl;
  a.gamma = gamma;
  a.norms = norms;
  a.idx_rb = (int)plan->idx_row_bytes;
  a.qjl_rb = (int)plan->qjl_row_bytes;
  const bool prod = plan->mode == TQ_PROD, bf16 = x_dtype == TQ_BF16;
  cudaError_t e;
  switch (plan->d) {
    case 32: e = launch_d<32>(a, plan->mse_bits, prod, bf16, st, plan->device); break;
    case 64: e = launch_d<64>(a, plan->mse_bits, prod, bf16, st, plan->device); break;
    default: e = launch_d<96>(a, plan->mse_bits, prod, bf16, st, plan->device); break;
  }
  TQ_CHECK_CUDA(e, who);
  return TQ_OK;
}

}  // namespace sq
}  // namespace tq
