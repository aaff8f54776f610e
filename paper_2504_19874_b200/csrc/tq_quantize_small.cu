// Quantiser for short vectors (d = 32, 64, 96, 128; the channel groups of a KV cache): Quant_mse / Quant_prod of Algorithms 1 and 2
// in ONE launch that keeps a row in the registers of four lanes from its load to its packed codes -- norm, rotation, nearest
// centroid, residual, gamma, QJL projection, signs.  The accumulator fragment of the rotation is, lane for lane, the A fragment
// that the projection needs, so the residual never leaves the registers.  (mma.sync, not tcgen05: at K = N = 64 the whole job
// is 0.1 of an MMA tile pipeline's start-up, and the register layout is what makes the fusion free.)
//
// fp32 fidelity: operands are pairs of fp16 limbs (hi + lo keeps a value to 2^-24), rows scaled by the power of two that
// brings their largest element to [2^12, 2^13), matrices likewise; hi hi + hi lo + lo hi in fp32.  bf16 input is exact in
// one limb and takes two products.
//
// Bound: memory latency and launch (n = 32,768 rows of 64: 5 MB).  Before: row norms, an fp32 GEMM on CUDA cores per
// product and a clearing of the rows, three to five launches per call.  Measured per call, n = 32,768, d = 64, bf16:
// TQ_PROD b_m = 2 48 -> 12 us, TQ_MSE b = 3 34 -> 8 us; the four calls of a 4,096-token prompt 229 -> 42 us.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <vector>

#include "tq_quantize_small.h"
#include "tq_quantize_tc.h"

namespace tq {
namespace sq {

namespace {

constexpr int NW = 8;               // warps per CTA, 16 rows each

// Bytes between matrix rows in shared memory: a multiple of 64 that is 64 mod 128, so that the 16-byte fragment loads of
// eight lanes (two matrix rows x four pieces) fall into distinct banks.
__host__ __device__ constexpr int row_stride(int d) { return 2 * d + ((2 * d) % 128 == 0 ? 64 : 0); }
__host__ __device__ constexpr int image_bytes(int d) { return 2 * d * row_stride(d); }   // hi rows, then lo rows

struct Args {
  const void* X;
  int64_t n, ldx;
  int vec;                          // rows are 16-byte aligned
  const uint4* pi_img;
  const uint4* sp_img;
  float pi_unscale;                 // 2^-eP
  Codebook cb;
  uint8_t* idx;
  uint8_t* qjl;
  float* gamma;
  float* norms;                     // nullable: rows are taken as unit-norm
  int idx_rb, qjl_rb;
};

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_half2(float a, float b) {
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// hi and lo limbs of two values
__device__ __forceinline__ void limbs(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(a, b);
  const float2 f = __half22float2(h);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = pack_half2(a - f.x, b - f.y);
}
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}
__device__ __forceinline__ float quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ uint32_t quad_or(uint32_t v) {
  v |= __shfl_xor_sync(0xffffffffu, v, 1);
  return v | __shfl_xor_sync(0xffffffffu, v, 2);
}
// 2^e that brings a row's largest magnitude into [2^12, 2^13), and its inverse (1 and 1 for an all-zero row)
__device__ __forceinline__ void row_scale(float amax, float& up, float& down) {
  const int e = (int)((__float_as_uint(amax) >> 23) & 255u) - 127;
  const int s = amax > 0.f ? max(-100, min(100, 12 - e)) : 0;
  up = __uint_as_float((uint32_t)(s + 127) << 23);
  down = __uint_as_float((uint32_t)(127 - s) << 23);
}

// Packs the codes of a row pair: thread (g, q) holds for tile j the codes of coordinates 8 j + 2 q, + 1 (low bits of `pair`,
// BITS each); `words` collects the row's words over the tiles, the four lanes of a quad are combined at the end.
template <int BITS>
__device__ __forceinline__ void put_codes(uint32_t* words, int j, int q, uint32_t pair) {
  constexpr int per_tile = 8 * BITS;
  const int base = (j * per_tile) >> 5, off = (j * per_tile) & 31;
  if (BITS == 3) {
    const unsigned long long v = (unsigned long long)pair << (off + 6 * q);
    words[base] |= (uint32_t)v;
    if (off > 8) words[base + 1] |= (uint32_t)(v >> 32);   // off = 8: at most 8 + 18 + 6 = 32 bits
  } else {
    words[base] |= pair << (off + 2 * BITS * q);
  }
}
template <int NWORDS>
__device__ __forceinline__ void store_words(uint8_t* row, int rb, uint32_t (&words)[NWORDS], int q, bool ok) {
#pragma unroll
  for (int w = 0; w < NWORDS; ++w) {
    const uint32_t v = quad_or(words[w]);
    if (ok && (w & 3) == q) reinterpret_cast<uint32_t*>(row)[w] = v;
  }
  for (int w = NWORDS + ((q - NWORDS) & 3); w < rb / 4; w += 4)   // pad words
    if (ok) reinterpret_cast<uint32_t*>(row)[w] = 0u;
}

template <int D, int BITS, bool PROD, bool BF16>
__global__ void __launch_bounds__(32 * NW) small_quantize_kernel(Args a) {
  constexpr int KB = D / 32, NT = D / 8, STRIDE = row_stride(D);
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float cs[16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
  {
    constexpr int pieces = image_bytes(D) / 16;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(smem);
    auto copy = [&](uint32_t to, const uint4* from) {
      for (int i = threadIdx.x; i < pieces; i += 32 * NW)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + 16 * i), "l"(from + i) : "memory");
    };
    copy(dst, a.pi_img);
    if (PROD) copy(dst + image_bytes(D), a.sp_img);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (threadIdx.x < 16) cs[threadIdx.x] = a.cb.c[threadIdx.x];
  }
  const unsigned char* bp = smem + g * STRIDE + q * 16;   // this lane's piece of row g of a tile
  constexpr int LO = D * STRIDE, SP = image_bytes(D);

  const int64_t tiles = (a.n + 15) / 16;
  // rows g and g + 8 of tile t: lane q holds elements 32 b + 8 q .. + 7 of block b
  float x[2][KB][8];
  auto load_rows = [&](int64_t t) {
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      const int64_t row = min(t * 16 + g + 8 * y, a.n - 1);   // rows past the end repeat the last one
#pragma unroll
      for (int b = 0; b < KB; ++b) {
        const int64_t at = row * a.ldx + 32 * b + 8 * q;
        if (BF16) {
          const __nv_bfloat16* p = static_cast<const __nv_bfloat16*>(a.X) + at;
          if (a.vec) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(p));
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              x[y][b][2 * i] = __uint_as_float(w[i] << 16);
              x[y][b][2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
            }
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[y][b][i] = __bfloat162float(p[i]);
          }
        } else {
          const float* p = static_cast<const float*>(a.X) + at;
          if (a.vec) {
            const float4 u = __ldg(reinterpret_cast<const float4*>(p)), v = __ldg(reinterpret_cast<const float4*>(p) + 1);
            x[y][b][0] = u.x; x[y][b][1] = u.y; x[y][b][2] = u.z; x[y][b][3] = u.w;
            x[y][b][4] = v.x; x[y][b][5] = v.y; x[y][b][6] = v.z; x[y][b][7] = v.w;
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[y][b][i] = __ldg(p + i);
          }
        }
      }
    }
  };
  int64_t t = (int64_t)blockIdx.x * NW + warp;
  if (t < tiles) load_rows(t);   // while the matrices arrive
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  for (; t < tiles; t += (int64_t)gridDim.x * NW) {
    const bool ok[2] = {t * 16 + g < a.n, t * 16 + g + 8 < a.n};
    float rs[2];          // accumulator -> rotated coordinate of the unit vector
    bool zero[2];
    uint32_t ah[KB][2][4], al[BF16 ? 1 : KB][2][4];   // A fragments of k-step (b, s)
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      float ss = 0.f, mx = 0.f;
#pragma unroll
      for (int b = 0; b < KB; ++b)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          ss = fmaf(x[y][b][i], x[y][b][i], ss);
          mx = fmaxf(mx, fabsf(x[y][b][i]));
        }
      const float nu = a.norms != nullptr ? sqrtf(quad_sum(ss)) : 1.f;
      if (a.norms != nullptr && ok[y] && q == 0) a.norms[t * 16 + g + 8 * y] = nu;
      zero[y] = !(nu > 0.f);
      float up, down;
      row_scale(quad_max(mx), up, down);
      rs[y] = zero[y] ? 0.f : down * a.pi_unscale / nu;
#pragma unroll
      for (int b = 0; b < KB; ++b)
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
          for (int h = 0; h < 2; ++h) {   // k slots 2 q, 2 q + 1 (h = 0) and 2 q + 8, 2 q + 9 (h = 1)
            const float v0 = x[y][b][4 * s + 2 * h] * up, v1 = x[y][b][4 * s + 2 * h + 1] * up;
            if (BF16) ah[b][s][2 * h + y] = pack_half2(v0, v1);
            else limbs(v0, v1, ah[b][s][2 * h + y], al[BF16 ? 0 : b][s][2 * h + y]);
          }
    }
    if (D <= 64 && t + (int64_t)gridDim.x * NW < tiles) load_rows(t + (int64_t)gridDim.x * NW);   // (wider rows: the registers are taken)
    // ---- y = Pi u, nearest centroid, residual
    constexpr int IW = D * BITS / 32 > 0 ? D * BITS / 32 : 1;
    uint32_t iw[2][IW];
#pragma unroll
    for (int y = 0; y < 2; ++y)
#pragma unroll
      for (int w = 0; w < IW; ++w) iw[y][w] = 0u;
    float e[PROD ? NT : 1][4];
    float es[2] = {0.f, 0.f}, emax[2] = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      float small[4] = {0.f, 0.f, 0.f, 0.f}, acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int b = 0; b < KB; ++b) {
        const uint4 hi = *reinterpret_cast<const uint4*>(bp + 8 * j * STRIDE + 64 * b);
        const uint4 lo = *reinterpret_cast<const uint4*>(bp + LO + 8 * j * STRIDE + 64 * b);
        mma16816(small, ah[b][0], lo.x, lo.y);
        mma16816(small, ah[b][1], lo.z, lo.w);
        if (!BF16) {
          mma16816(small, al[BF16 ? 0 : b][0], hi.x, hi.y);
          mma16816(small, al[BF16 ? 0 : b][1], hi.z, hi.w);
        }
        mma16816(acc, ah[b][0], hi.x, hi.y);
        mma16816(acc, ah[b][1], hi.z, hi.w);
      }
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        uint32_t pair = 0u;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float v = (acc[2 * y + i] + small[2 * y + i]) * rs[y];
          int code = 0;
#pragma unroll
          for (int k = 0; k < (1 << BITS) - 1; ++k) code += (v > a.cb.t[k]) ? 1 : 0;
          pair |= (uint32_t)code << (BITS * i);
          if (PROD) {
            const float r = zero[y] ? 0.f : v - (BITS > 0 ? cs[code] : a.cb.c[0]);
            e[PROD ? j : 0][2 * y + i] = r;
            es[y] = fmaf(r, r, es[y]);
            emax[y] = fmaxf(emax[y], fabsf(r));
          }
        }
        if (BITS > 0) put_codes<BITS>(iw[y], j, q, pair);
      }
    }
#pragma unroll
    for (int y = 0; y < 2; ++y)
      if (BITS > 0) store_words<IW>(a.idx + (size_t)(t * 16 + g + 8 * y) * a.idx_rb, a.idx_rb, iw[y], q, ok[y]);
    if constexpr (PROD) {
      // ---- gamma, then z = sign(S' e): the tiles' accumulators are the A fragments (k-step p: tiles 2 p, 2 p + 1)
      uint32_t eh[NT / 2][4], el[NT / 2][4];
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        const float gm = sqrtf(quad_sum(es[y]));
        if (q == 0 && ok[y]) a.gamma[t * 16 + g + 8 * y] = gm;
        float up, down;
        row_scale(quad_max(emax[y]), up, down);
#pragma unroll
        for (int p = 0; p < NT / 2; ++p)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            limbs(e[2 * p + h][2 * y] * up, e[2 * p + h][2 * y + 1] * up, eh[p][2 * h + y], el[p][2 * h + y]);
      }
      uint32_t zw[2][D / 32];
#pragma unroll
      for (int y = 0; y < 2; ++y)
#pragma unroll
        for (int w = 0; w < D / 32; ++w) zw[y][w] = 0u;
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        float small[4] = {0.f, 0.f, 0.f, 0.f}, acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int b = 0; b < KB; ++b) {   // (the image of S' has its columns in the order of these k slots)
          const uint4 hi = *reinterpret_cast<const uint4*>(bp + SP + 8 * j * STRIDE + 64 * b);
          const uint4 lo = *reinterpret_cast<const uint4*>(bp + SP + LO + 8 * j * STRIDE + 64 * b);
          mma16816(small, eh[2 * b], lo.x, lo.y);
          mma16816(small, eh[2 * b + 1], lo.z, lo.w);
          mma16816(small, el[2 * b], hi.x, hi.y);
          mma16816(small, el[2 * b + 1], hi.z, hi.w);
          mma16816(acc, eh[2 * b], hi.x, hi.y);
          mma16816(acc, eh[2 * b + 1], hi.z, hi.w);
        }
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          const uint32_t pair = (acc[2 * y] + small[2 * y] >= 0.f ? 1u : 0u) | (acc[2 * y + 1] + small[2 * y + 1] >= 0.f ? 2u : 0u);
          put_codes<1>(zw[y], j, q, pair);
        }
      }
#pragma unroll
      for (int y = 0; y < 2; ++y) store_words<D / 32>(a.qjl + (size_t)(t * 16 + g + 8 * y) * a.qjl_rb, a.qjl_rb, zw[y], q, ok[y]);
    }
    if (D > 64 && t + (int64_t)gridDim.x * NW < tiles) load_rows(t + (int64_t)gridDim.x * NW);
  }
}

template <int D, int BITS, bool PROD, bool BF16>
cudaError_t launch(const Args& a, cudaStream_t st, int device) {
  auto kern = small_quantize_kernel<D, BITS, PROD, BF16>;
  constexpr int smem = image_bytes(D) * (PROD ? 2 : 1);
  if (smem + 64 > 48 * 1024) {   // the centroids are static shared memory
    static std::atomic<unsigned long long> attr_devices{0};   // devices whose function attribute has been set
    if (device >= 64 || !((attr_devices.load(std::memory_order_relaxed) >> device) & 1ull)) {
      const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e != cudaSuccess) return e;
      if (device < 64) attr_devices.fetch_or(1ull << device, std::memory_order_relaxed);
    }
  }
  const int64_t ctas = std::min<int64_t>((a.n + 16 * NW - 1) / (16 * NW), (int64_t)tc::sm_count() * 2);
  kern<<<(unsigned)ctas, 32 * NW, smem, st>>>(a);
  count_launches(1);
  return cudaGetLastError();
}

template <int D, bool PROD, bool BF16>
cudaError_t launch_bits(const Args& a, int bits, cudaStream_t st, int device) {
  switch (bits) {
    case 0: return PROD ? launch<D, 0, true, BF16>(a, st, device) : cudaErrorInvalidValue;   // TQ_MSE has at least one bit
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

}  // namespace

cudaError_t plan_init(tq_plan* plan) {
  auto& s = plan->sq;
  s.ok = 0;
  const int d = plan->d;
  if (d % 32 != 0 || d > 128) return cudaSuccess;
  const size_t dd = (size_t)d * d, stride = row_stride(d) / 2;
  std::vector<float> M(dd);
  std::vector<__half> img(image_bytes(d) / 2, __half(0.f));
  for (int which = 0; which < (plan->mode == TQ_PROD ? 2 : 1); ++which) {
    cudaError_t e = cudaMemcpy(M.data(), which == 0 ? plan->dPi : plan->dSp, dd * sizeof(float), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return e;
    double mx = 0.0;
    for (float v : M) mx = std::max(mx, std::fabs((double)v));
    if (!std::isfinite(mx)) return cudaSuccess;
    const int ex = mx > 0.0 ? std::max(-100, std::min(100, 13 - std::ilogb(mx))) : 0;
    for (int n = 0; n < d; ++n)
      for (int p = 0; p < d; ++p) {   // position p of row n: 32 b + 8 q + 4 s + 2 h + i
        const int b = p >> 5, q = (p >> 3) & 3, s2 = (p >> 2) & 1, h = (p >> 1) & 1, i = p & 1;
        const int k = which == 0 ? p : 32 * b + 16 * s2 + 8 * h + 2 * q + i;
        const float v = (float)std::ldexp((double)M[(size_t)n * d + k], ex);
        const __half hi = __float2half_rn(v);
        img[n * stride + p] = hi;
        img[(d + n) * stride + p] = __float2half_rn(v - __half2float(hi));
      }
    void** dst = which == 0 ? &s.pi_img : &s.sp_img;
    e = cudaMalloc(dst, image_bytes(d));
    if (e == cudaSuccess) e = cudaMemcpy(*dst, img.data(), image_bytes(d), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return e;
    if (which == 0) s.pi_unscale = (float)std::ldexp(1.0, -ex);
  }
  s.ok = 1;
  return cudaSuccess;
}

void plan_free(tq_plan* plan) {
  cudaFree(plan->sq.pi_img);
  cudaFree(plan->sq.sp_img);
}

// d = 128 (canonical layout): the tcgen05 GEMMs take four launches and a scratch round trip of the limbs, this kernel reads both
// matrices from shared memory once per 16 rows.  Measured: n = 100 20 against 29 us, n = 5,000 23 against 30 us, n = 500,000
// bf16 297 against 337 us, n = 10^6 fp32 395 against 353 us (TQ_MSE) and 675 against 663 us (TQ_PROD).
bool preferred(const tq_plan* plan, int x_dtype, int64_t n) {
  return plan->sq.ok && plan->layout == TQ_LAYOUT_CANONICAL && (x_dtype == TQ_BF16 || n < 200000);
}

int quantize(const tq_plan* plan, const void* X, int x_dtype, int64_t n, int64_t ldx, uint8_t* idx, uint8_t* qjl, float* gamma,
             float* norms, cudaStream_t st, const char* who) {
  Args a;
  a.X = X;
  a.n = n;
  a.ldx = ldx;
  a.vec = (ldx * (x_dtype == TQ_F32 ? 4 : 2)) % 16 == 0;
  a.pi_img = static_cast<const uint4*>(plan->sq.pi_img);
  a.sp_img = static_cast<const uint4*>(plan->sq.sp_img);
  a.pi_unscale = plan->sq.pi_unscale;
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
    case 96: e = launch_d<96>(a, plan->mse_bits, prod, bf16, st, plan->device); break;
    default: e = launch_d<128>(a, plan->mse_bits, prod, bf16, st, plan->device); break;
  }
  TQ_CHECK_CUDA(e, who);
  return TQ_OK;
}

}  // namespace sq
}  // namespace tq
