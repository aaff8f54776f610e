// C ABI of libtq: argument checking, plan set-up and kernel dispatch.
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "tq_attend_simt.cuh"
#include "tq_dequant_tc.h"
#include "tq_gemm_simt.cuh"
#include "tq_internal.h"
#include "tq_quantize_small.h"
#include "tq_quantize_tc.h"
#include "tq_scan_mma.h"
#include "tq_scan_nib.h"
#include "tq_scan_simt.cuh"
#include "tq_scan_tc.h"
#include "tq_tc.cuh"

using namespace tq;

namespace {

inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }
inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// S' = S Pi^T in fp64 (set-up, once per plan): out[i][j] = sum_k S[i][k] Pi[j][k].
__global__ void sprime_kernel(const float* __restrict__ S, const float* __restrict__ Pi, float* __restrict__ out, int d) {
  __shared__ double sa[16][17], sb[16][17];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int i = blockIdx.y * 16 + ty, j = blockIdx.x * 16 + tx;
  double acc = 0.0;
  for (int k0 = 0; k0 < d; k0 += 16) {
    const int ia = blockIdx.y * 16 + ty, jb = blockIdx.x * 16 + ty;
    sa[ty][tx] = (ia < d && k0 + tx < d) ? (double)S[(size_t)ia * d + k0 + tx] : 0.0;
    sb[ty][tx] = (jb < d && k0 + tx < d) ? (double)Pi[(size_t)jb * d + k0 + tx] : 0.0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k) acc += sa[ty][k] * sb[tx][k];
    __syncthreads();
  }
  if (i < d && j < d) out[(size_t)i * d + j] = (float)acc;
}

int check_plan(const tq_plan* plan, const char* who) {
  TQ_REQUIRE(plan != nullptr, TQ_ERR_INVALID_ARG, "%s: plan is NULL", who);
  int dev = -1;
  TQ_CHECK_CUDA(cudaGetDevice(&dev), who);
  TQ_REQUIRE(dev == plan->device, TQ_ERR_INVALID_ARG, "%s: plan was created on device %d, current device is %d", who,
             plan->device, dev);
  return TQ_OK;
}

int check_rows(const char* who, const char* name, const void* p, int dtype, int64_t rows, int64_t ld, int d) {
  TQ_REQUIRE(dtype == TQ_F32 || dtype == TQ_BF16, TQ_ERR_UNSUPPORTED, "%s: unknown dtype %d for %s", who, dtype, name);
  TQ_REQUIRE(p != nullptr, TQ_ERR_INVALID_ARG, "%s: %s is NULL", who, name);
  TQ_REQUIRE(ld >= d, TQ_ERR_INVALID_ARG, "%s: row stride of %s (%lld) is smaller than d (%d)", who, name, (long long)ld, d);
  TQ_REQUIRE(aligned(p, 16), TQ_ERR_ALIGNMENT, "%s: %s is not 16-byte aligned", who, name);
  (void)rows;
  return TQ_OK;
}

int check_codes(const tq_plan* plan, const char* who, const uint8_t* idx, const uint8_t* qjl, const float* gamma) {
  if (plan->mse_bits > 0) {
    TQ_REQUIRE(idx != nullptr, TQ_ERR_INVALID_ARG, "%s: idx is NULL", who);
    TQ_REQUIRE(aligned(idx, 16), TQ_ERR_ALIGNMENT, "%s: idx is not 16-byte aligned", who);
  }
  if (plan->mode == TQ_PROD) {
    TQ_REQUIRE(qjl != nullptr && gamma != nullptr, TQ_ERR_INVALID_ARG, "%s: qjl / gamma is NULL for a TQ_PROD plan", who);
    TQ_REQUIRE(aligned(qjl, 16) && aligned(gamma, 4), TQ_ERR_ALIGNMENT, "%s: qjl / gamma is misaligned", who);
  }
  return TQ_OK;
}

simt::Codes make_codes(const tq_plan* plan, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma) {
  simt::Codes c;
  c.idx = idx;
  c.idx_rb = plan->idx_row_bytes;
  c.qjl = (plan->mode == TQ_PROD) ? qjl : nullptr;
  c.qjl_rb = plan->qjl_row_bytes;
  c.gamma = gamma;
  c.cb = plan->cb;
  c.d = plan->d;
  c.dpad = plan->dpad;
  c.coef = plan->coef;
  c.rows = n;
  c.nibble = plan->layout == TQ_LAYOUT_NIBBLE;
  return c;
}

size_t qcat_bytes(const tq_plan* plan, int nq) {
  return align_up((size_t)nq * plan->ncat * plan->dpad * sizeof(float), 256);
}

constexpr int64_t kTensorChunk = 65536;    // rows per launch the tensor-core quantiser asks scratch for
constexpr int64_t kResidualChunk = 16384;  // rows of E kept in flight by tq_quantize_prod (L2-sized)
constexpr int64_t kTopkBlockMin = 4096, kTopkBlockPref = 65536;
constexpr int kFewQueries = 16;  // up to this many queries the code scan is bandwidth-bound
// top-k on the tensor-path scan: candidate pairs kept per query, queries per pass, dense-buffer rows
constexpr int kCandCap = 32768;
constexpr int64_t kFilterMinN = 65536;
constexpr int64_t kDenseRowsMin = 4096;
constexpr int kGroupQueries = tscan::kQueriesPerPass * tscan::kPassesPerGroup;

// The two engines behind the bit-plane scan: register-fed integer MMA (2, 4 or 8 queries per pass) for few queries, tcgen05
// (32 queries per pass, 64 in calls of more than 32 queries) for more.
struct ScanEngine {
  const tq_plan* plan;
  bool tc;
  bool nib;                 // register-fed table-lookup scan of the nibble layout (2 or 8 queries per pass)
  int qpp;                  // queries per pass
  int64_t dense_rows_pref;  // rows of the dense score buffer that keep the rescue pass to a few launches
  size_t ws_bytes;          // engine workspace (constants + B operand)
};

ScanEngine pick_engine(const tq_plan* plan, int nq) {
  ScanEngine e;
  e.plan = plan;
  e.nib = plan->layout == TQ_LAYOUT_NIBBLE;
  // nibble layout (measured at n = 10^6): at d = 1536 a tcgen05 pass costs 0.53 ms against 0.28 ms per pass of the
  // eight-query register-fed shape, so it wins from 15 queries on; where that shape does not fit shared memory
  // (d = 3072: 0.84 ms against 0.35 ms per two-query pass) from five queries on
  // bit streams: a tcgen05 pass costs the same for any number of queries up to 32; the register-fed eight-query shape, where
  // its operand fits shared memory, is cheaper up to eight (whole calls of 8 queries, 10^6 rows: d = 1536 mse b = 2 207 against
  // 301 us, prod b = 3 309 against 440, d = 1024 prod b = 4 336 against 487, d = 200 prod b = 3 93 against 148); two passes of it
  // are not (9 queries and more).  Where only the four-query shape fits (prod b = 4 and mse b = 4 at d = 1536), 4 + 3 queries
  // already cost more than a tcgen05 pass.
  const int tc_from = e.nib ? (nscan::queries_per_pass(plan, 8) == 8 ? 15 : 5) : mscan::queries_per_pass(plan, 8) == 8 ? 9 : 7;
  e.tc = nq >= tc_from && tscan::available(plan);
  e.nib = e.nib && !e.tc;
  e.qpp = e.tc ? tscan::queries_per_pass(nq) : e.nib ? nscan::queries_per_pass(plan, nq) : mscan::queries_per_pass(plan, nq);
  e.dense_rows_pref = 1 << 20;   // n = 10^6: the guarded rescue is one scan + one selection launch per pass
  e.ws_bytes = e.tc ? tscan::workspace_bytes(plan) : e.nib ? nscan::workspace_bytes(plan) : mscan::workspace_bytes(plan, nq);
  return e;
}

// Prepares what the pass starting at query q0 needs (the tcgen05 engine builds 256 queries at a time).
int engine_prepare(const ScanEngine& e, const float* Qcat, int q0, int nq, void* ws, cudaStream_t st, const char* who) {
  const int ncols = e.plan->ncat * e.plan->dpad;
  if (e.nib) return nscan::prepare(e.plan, Qcat + (size_t)q0 * ncols, std::min(e.qpp, nq - q0), ws, st, who);
  if (e.tc) {
    if (q0 % kGroupQueries != 0) return TQ_OK;
    return tscan::prepare_group(e.plan, Qcat + (size_t)q0 * ncols, std::min(kGroupQueries, nq - q0), ws, st, who);
  }
  return mscan::prepare(e.plan, Qcat + (size_t)q0 * ncols, std::min(e.qpp, nq - q0), ws, st, who);
}

int engine_run(const ScanEngine& e, int q0, int nqp, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma,
               const float* norms, float* scores, int64_t lds, const mscan::Filter* filter, const int* run_if, const void* ws,
               cudaStream_t st, const char* who, int64_t step = 1) {
  if (e.nib) return nscan::run(e.plan, nqp, n, idx, qjl, gamma, norms, scores, lds, filter, run_if, ws, true, st, who, step);
  if (e.tc)
    return tscan::run_pass(e.plan, (q0 % kGroupQueries) / tscan::kQueriesPerPass, nqp, n, idx, qjl, gamma, norms, scores, lds,
                           filter, run_if, ws, st, who, step);
  return mscan::run(e.plan, nqp, n, idx, qjl, gamma, norms, scores, lds, filter, run_if, ws, st, who, step);
}

size_t ms_score_fixed(const tq_plan* plan, int nq) { return qcat_bytes(plan, nq) + align_up(pick_engine(plan, nq).ws_bytes, 256); }
size_t ms_topk_fixed(const tq_plan* plan, int nq) {
  return ms_score_fixed(plan, nq) + 1024 /* tau, count, overflow */ + (size_t)pick_engine(plan, nq).qpp * kCandCap * 8;
}

// Samples of a screened search: `dense` rows whose lower bounds are written out give a threshold that k rows reach, `first` rows (0:
// none) are filtered with it and give the threshold of the pass over all rows.  That one then keeps k n / first candidates: a hit
// costs its warp as much as testing 30 estimates, and with one sample of 13,312 of 10^6 rows (one hit in 132) the pass took
// 939 us instead of 130.
// The rows written out are among the first sample's, so that at least k of that one reach the threshold.
struct ScreenSamples {
  int64_t dense, dense_step, first, first_step;
};
ScreenSamples screen_samples(int64_t n, int k, int64_t most) {
  const double expect = 2048.0 / (k + 8);   // rows per sampled row that make a list of 2,048
  const double dense0 = std::max(4096.0, std::min(160.0 * (k + 8), std::max(16384.0, 16.0 * (k + 8))));
  double first = std::max(std::sqrt((double)n * dense0), n / expect), dense = std::max(dense0, first / expect);
  ScreenSamples s;
  if ((double)n <= 16.0 * dense0 && n / dense0 <= expect) {
    first = 0.0;
    dense = dense0;
  }
  s.first = std::min<int64_t>(round_up64((int64_t)first, 256), n);
  s.dense = std::min<int64_t>(round_up64((int64_t)dense, 256), std::min<int64_t>(most / 256 * 256, s.first > 0 ? s.first : n));
  s.first_step = s.first > 0 ? n / s.first : 1;
  s.dense_step = s.first > 0 ? s.first_step * (s.first / s.dense) : n / s.dense;
  return s;
}

// Top-k of many queries over at least kFilterMinN vectors: bounds of the estimates from one fp16 pass per 256 queries, exact estimates only
// for the rows that the bounds leave (tq_screen_tc.cu).  It pays where the exact engine needs several passes of 64 queries, and the
// less so the more rows the samples add and the more k-blocks a row has: with up to 128 queries their issue, not the MMAs, bounds the
// pass, and selecting among the rows written out grows with k.  The line is a fit to 630 searches measured both ways (us, exact /
// screened): d = 200 prod b = 3, 10^6 rows, k = 10, 65 queries 477 / 287, 256 queries 1,289 / 358; d = 768 prod b = 4, 65,536 rows, k = 100,
// 128 queries 223 / 243, 192 queries 304 / 275; d = 3072 prod b = 2, 500,000 rows, k = 10, 128 queries 1,379 / 1,466, 129 queries
// 1,676 / 1,516; d = 1536 mse b = 2, k = 1,024, 256 queries, 10^6 rows 2,821 / 2,356, 65,536 rows 594 / 902.
constexpr int kScreenPass = 64;   // queries of a pass of the exact engine in such calls: they share a flag
bool screens(const tq_plan* plan, int nq, int64_t n, int k) {
  const ScanEngine e = pick_engine(plan, nq);
  if (nq <= kScreenPass || n < kFilterMinN || !e.tc || e.qpp != kScreenPass) return false;
  const ScreenSamples s = screen_samples(n, k, std::max<int64_t>(std::min<int64_t>(n, e.dense_rows_pref) / 4, 16384));
  const double passes = (nq + kScreenPass - 1) / kScreenPass, rows = (double)n + (double)s.first + (double)s.dense + 1e4 + 200.0 * k;
  return passes * (double)n >= rows * (1.0 + screen::k_blocks(plan) / 96.0);
}
// A query's list: 2,048 candidates are expected at most (screen_samples), and two CTAs of the selection fit an SM.
constexpr int kScreenCap = 8192;
// Workspace of a screened pass, between the exact engine's operand and the dense score buffer.
struct ScreenSpace {
  size_t operand, tau, kth, count, count1, left, flag, left_s, left_i, cand_s, cand_i, total;   // byte offsets
};
ScreenSpace screen_space(const tq_plan* plan) {
  ScreenSpace s;
  constexpr size_t Q = screen::kQueries;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t here = at;
    at += align_up(bytes, 256);
    return here;
  };
  s.operand = take(screen::workspace_bytes(plan));
  s.tau = take(Q * 4);
  s.kth = take(Q * 4);
  s.count = take(Q * 4);
  s.count1 = take(Q * 4);
  s.left = take(Q * 4);
  s.flag = take(3 * Q / kScreenPass * 4);
  s.left_s = take(Q * screen::kSurvivors * 4);
  s.left_i = take(Q * screen::kSurvivors * 4);
  s.cand_s = take(Q * kScreenCap * 4);
  s.cand_i = take(Q * kScreenCap * 4);
  s.total = at;
  return s;
}
// Bytes behind the rotated queries that a screened call needs, and those with which its rescue takes few launches.
size_t screen_least(const tq_plan* plan) {
  return align_up(tscan::workspace_bytes(plan), 256) + screen_space(plan).total + (size_t)kDenseRowsMin * screen::kQueries * sizeof(float);
}
size_t screen_pref(const tq_plan* plan, int nq, int64_t n) {
  const ScanEngine e = pick_engine(plan, nq);
  const size_t rescue = (size_t)e.qpp * std::min<int64_t>(n, e.dense_rows_pref), samples = (size_t)screen::kQueries * 16384;
  return align_up(e.ws_bytes, 256) + screen_space(plan).total + align_up(std::max(rescue, samples) * sizeof(float), 256);
}

template <typename T>
cudaError_t launch_row_norm(const T* X, int64_t ld, int64_t n, int d, float* out, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int64_t blocks = std::min<int64_t>((n + 7) / 8, tc::sm_count() * 16);
  scan::row_norm_kernel<T><<<(unsigned)blocks, 256, 0, st>>>(X, ld, n, d, out);
  count_launches(1);
  return cudaGetLastError();
}

// Stage-1 GEMM of both quantisers: Y = X Pi^T with the nearest-centroid epilogue.
template <int BITS, int MODE>
cudaError_t launch_rotate_quantize(const tq_plan* plan, const void* X, int x_dtype, int64_t n, int64_t ldx,
                                   const float* nu, uint8_t* idx, float* E, int64_t ldE, cudaStream_t st) {
  simt::EpQuantize<BITS, MODE> ep;
  ep.cb = plan->cb;
  ep.nu = nu;
  ep.out = idx;
  ep.out_rb = plan->idx_row_bytes;
  ep.E = E;
  ep.ldE = ldE;
  ep.d = plan->d;
  simt::RowsF32 B{plan->dPi, plan->d, plan->d, plan->d};
  if (x_dtype == TQ_F32) {
    simt::RowsF32 A{static_cast<const float*>(X), ldx, n, plan->d};
    return simt::launch_gemm(A, B, ep, n, (int64_t)plan->d, plan->d, st);
  }
  simt::RowsBF16 A{static_cast<const __nv_bfloat16*>(X), ldx, n, plan->d};
  return simt::launch_gemm(A, B, ep, n, (int64_t)plan->d, plan->d, st);
}

template <int MODE>
cudaError_t dispatch_rotate_quantize(const tq_plan* plan, const void* X, int x_dtype, int64_t n, int64_t ldx,
                                     const float* nu, uint8_t* idx, float* E, int64_t ldE, cudaStream_t st) {
  switch (plan->mse_bits) {
    case 0: return launch_rotate_quantize<0, MODE>(plan, X, x_dtype, n, ldx, nu, idx, E, ldE, st);
    case 1: return launch_rotate_quantize<1, MODE>(plan, X, x_dtype, n, ldx, nu, idx, E, ldE, st);
    case 2: return launch_rotate_quantize<2, MODE>(plan, X, x_dtype, n, ldx, nu, idx, E, ldE, st);
    case 3: return launch_rotate_quantize<3, MODE>(plan, X, x_dtype, n, ldx, nu, idx, E, ldE, st);
    default: return launch_rotate_quantize<4, MODE>(plan, X, x_dtype, n, ldx, nu, idx, E, ldE, st);
  }
}

cudaError_t compute_norms(const void* X, int x_dtype, int64_t n, int64_t ldx, int d, float* norms, cudaStream_t st) {
  if (x_dtype == TQ_F32) return launch_row_norm(static_cast<const float*>(X), ldx, n, d, norms, st);
  return launch_row_norm(static_cast<const __nv_bfloat16*>(X), ldx, n, d, norms, st);
}

// True when the packed rows have bytes that no 32-coordinate group writes.
bool has_pad_words(int d, int bits, size_t row_bytes) {
  return bits > 0 && (size_t)((d + 31) / 32) * bits * 4 < row_bytes;
}

// Few queries: one warp per output column j forms <Rot[j, :], q> for up to 8 queries at a time.  The
// warp's slice of the matrix row goes to registers first, so that its latency overlaps the staging
// of the queries in shared memory; each lane sums its products in fp32, the 32 partial sums are
// added in fp64.  The matrix is read once per 8 queries; its rows are padded with zeros to a multiple of 8 columns, so that
// they are read 16 bytes at a time at every d (element by element, 123 queries of d = 1863 took 162 us and more).
constexpr int kRotQ = 8, kRotChunk = 2048;   // 64 KB of queries per chunk (dynamic shared memory)
constexpr int kRotQPerBlock = 64;            // most queries per CTA (grid.y covers the rest)
// Queries per CTA: 64 (eight rounds, the matrix is read once for all of them) where that still gives every SM two CTAs, else
// fewer rounds in more CTAs: 64 queries of d = 128 took four CTAs 33 us for eight rounds each, 32 CTAs take 3.4 us.
inline int rotate_queries_per_cta(int64_t column_ctas, int nq) {
  int per = kRotQPerBlock;
  while (per > kRotQ && column_ctas * ((nq + per - 1) / per) < 2 * tc::sm_count()) per /= 2;
  return per;
}

template <typename T>
__global__ void __launch_bounds__(256) rotate_queries_kernel(const float* __restrict__ Rot, int nrows, int d, int dpad,
                                                             const T* __restrict__ Q, int64_t ldq, int nq,
                                                             float* __restrict__ Qcat, int64_t ldo, int per_cta, int stride) {
  extern __shared__ __align__(16) float qs_raw[];   // [queries of a round][stride]
  auto qs = [&](int qq, int c) -> float* { return qs_raw + qq * stride + c; };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j = blockIdx.x * 8 + warp;
  const float* row = Rot + (size_t)min(j, nrows - 1) * dpad;
  const int q_begin = blockIdx.y * per_cta, q_end = min(nq, q_begin + per_cta);
  for (int q0 = q_begin; q0 < q_end; q0 += kRotQ) {
    float acc[kRotQ];
#pragma unroll
    for (int qq = 0; qq < kRotQ; ++qq) acc[qq] = 0.f;
    const int nact = min(kRotQ, q_end - q0);   // queries of this round: the others are neither staged nor summed
    for (int c0 = 0; c0 < d; c0 += kRotChunk) {
      const int len = min(kRotChunk, dpad - c0);   // the matrix and the staged queries hold zeros in the columns past d
      float4 r[kRotChunk / 128];
      const float4* row4 = reinterpret_cast<const float4*>(row + c0);
#pragma unroll
      for (int i = 0; i < kRotChunk / 128; ++i) {
        const int c4 = lane + 32 * i;
        r[i] = (4 * c4 < len) ? __ldg(row4 + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      if (q0 == q_begin && c0 == 0) {   // the first piece of the matrix (the plan's) is on its way
        wait_for_predecessor();         // it may write the queries
        allow_successor();              // (only now: a successor may start reading the codes, see nscan::run)
      }
      __syncthreads();
      for (int e = threadIdx.x; e < nact * (stride / 4); e += blockDim.x) {
        const int qq = e / (stride / 4), c = 4 * (e % (stride / 4));
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        const T* src = Q + (int64_t)(q0 + qq) * ldq + c0 + c;
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (c0 + c + t < d) v[t] = scan::to_f32<T>(src[t]);
        *reinterpret_cast<float4*>(qs(qq, c)) = make_float4(v[0], v[1], v[2], v[3]);
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < kRotChunk / 128; ++i) {
        const int c4 = lane + 32 * i;
        if (4 * c4 < len) {
#pragma unroll
          for (int qq = 0; qq < kRotQ; ++qq) {
            if (qq < nact) {
              const float4 v = *reinterpret_cast<const float4*>(qs(qq, 4 * c4));
              acc[qq] = fmaf(r[i].x, v.x, fmaf(r[i].y, v.y, fmaf(r[i].z, v.z, fmaf(r[i].w, v.w, acc[qq]))));
            }
          }
        }
      }
    }
#pragma unroll
    for (int qq = 0; qq < kRotQ; ++qq) {
      if (qq >= nact) break;
      double v = (double)acc[qq];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0 && j < nrows && q0 + qq < q_end) Qcat[(int64_t)(q0 + qq) * ldo + j] = (float)v;
    }
  }
}

// Many queries: the same sums in the same order (a lane adds its products over ascending columns 4 lane + 128 i in
// fp32, the 32 partial sums are added in fp64 by the same butterfly), so a query's rotated form does not depend on
// which kernel formed it -- but a warp holds eight matrix rows against the eight staged queries (64 FMAs per pair of
// 16-byte loads), a CTA of four warps 32 rows, and the queries are read once per 32 output columns instead of once
// per 8.  Three CTAs per SM hide each other's staging.
constexpr int kRmRows = 8, kRmWarps = 4, kRmRowsPerBlock = kRmWarps * kRmRows;
constexpr int kRotManyFrom = 64;   // queries from which the blocked kernel is used

template <typename T>
__global__ void __launch_bounds__(32 * kRmWarps) rotate_many_kernel(const float* __restrict__ Rot, int nrows, int d, int dpad,
                                                                    const T* __restrict__ Q, int64_t ldq, int nq,
                                                                    float* __restrict__ Qcat, int64_t ldo, int per_cta, int stride) {
  extern __shared__ __align__(16) float qs_raw[];   // [queries of a round][stride]
  auto qs = [&](int qq, int c) -> float* { return qs_raw + qq * stride + c; };
  wait_for_predecessor();   // it may write the queries
  allow_successor();        // (only now: a successor may start reading the codes, see nscan::run)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = blockIdx.x * kRmRowsPerBlock + warp * kRmRows;
  const int q_begin = blockIdx.y * per_cta, q_end = min(nq, q_begin + per_cta);
  for (int q0 = q_begin; q0 < q_end; q0 += kRotQ) {
    float acc[kRmRows][kRotQ];
#pragma unroll
    for (int rr = 0; rr < kRmRows; ++rr)
#pragma unroll
      for (int qq = 0; qq < kRotQ; ++qq) acc[rr][qq] = 0.f;
    const int nact = min(kRotQ, q_end - q0);
    for (int c0 = 0; c0 < d; c0 += kRotChunk) {
      const int len = min(kRotChunk, dpad - c0);   // the matrix and the staged queries hold zeros in the columns past d
      __syncthreads();
      for (int e = threadIdx.x; e < nact * (stride / 4); e += blockDim.x) {
        const int qq = e / (stride / 4), c = 4 * (e % (stride / 4));
        if (c >= len) continue;   // columns past the chunk's end are not read below
        const T* src = Q + (int64_t)(q0 + qq) * ldq + c0 + c;
        float v[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) v[t] = c0 + c + t < d ? scan::to_f32<T>(src[t]) : 0.f;
        *reinterpret_cast<float4*>(qs(qq, c)) = make_float4(v[0], v[1], v[2], v[3]);
      }
      __syncthreads();
#pragma unroll 2
      for (int i = 0; i < kRotChunk / 128; ++i) {
        const int c4 = lane + 32 * i;
        if (4 * c4 >= len) break;
        float4 r[kRmRows];
#pragma unroll
        for (int rr = 0; rr < kRmRows; ++rr)
          r[rr] = __ldg(reinterpret_cast<const float4*>(Rot + (size_t)min(j0 + rr, nrows - 1) * dpad + c0) + c4);
#pragma unroll
        for (int qq = 0; qq < kRotQ; ++qq) {
          if (qq < nact) {
            const float4 v = *reinterpret_cast<const float4*>(qs(qq, 4 * c4));
#pragma unroll
            for (int rr = 0; rr < kRmRows; ++rr)
              acc[rr][qq] = fmaf(r[rr].x, v.x, fmaf(r[rr].y, v.y, fmaf(r[rr].z, v.z, fmaf(r[rr].w, v.w, acc[rr][qq]))));
          }
        }
      }
    }
    // The 32 partial sums of each of the warp's 64 outputs are added in fp64 along the tree of the xor butterfly
    // (lanes l and l ^ 16, then ^ 8, 4, 2, 1: every lane of the butterfly ends with the same bits, additions being
    // commutative), but transposed: at each level a lane keeps half of its values and hands the other half to its
    // partner, so that 62 fp64 additions per lane do what 320 would; lane l ends with outputs 2 l and 2 l + 1.
    static_assert(kRmRows * kRotQ == 64, "the transposed reduction is written for 64 outputs per warp");
    const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0, b2 = (lane & 4) != 0, b1 = (lane & 2) != 0, b0 = (lane & 1) != 0;
    double w1[32], w2[16], w3[8], w4[4], w5[2];
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const float lo = acc[k / kRotQ][k % kRotQ], hi = acc[(k + 32) / kRotQ][k % kRotQ];
      const float got = __shfl_xor_sync(0xffffffffu, b4 ? lo : hi, 16);
      w1[k] = (double)(b4 ? hi : lo) + (double)got;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) w2[k] = (b3 ? w1[k + 16] : w1[k]) + __shfl_xor_sync(0xffffffffu, b3 ? w1[k] : w1[k + 16], 8);
#pragma unroll
    for (int k = 0; k < 8; ++k) w3[k] = (b2 ? w2[k + 8] : w2[k]) + __shfl_xor_sync(0xffffffffu, b2 ? w2[k] : w2[k + 8], 4);
#pragma unroll
    for (int k = 0; k < 4; ++k) w4[k] = (b1 ? w3[k + 4] : w3[k]) + __shfl_xor_sync(0xffffffffu, b1 ? w3[k] : w3[k + 4], 2);
#pragma unroll
    for (int k = 0; k < 2; ++k) w5[k] = (b0 ? w4[k + 2] : w4[k]) + __shfl_xor_sync(0xffffffffu, b0 ? w4[k] : w4[k + 2], 1);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int idx = 2 * lane + k, rr = idx / kRotQ, qq = idx % kRotQ;
      if (qq < nact && j0 + rr < nrows) Qcat[(int64_t)(q0 + qq) * ldo + j0 + rr] = (float)w5[k];
    }
  }
}

template <typename T>
cudaError_t launch_rotate_queries(const tq_plan* plan, const T* Q, int64_t ldq, int nq, float* Qcat, cudaStream_t st) {
  const int ncols = plan->ncat * plan->dpad;
  constexpr int smem_max = kRotQ * kRotChunk * (int)sizeof(float);
  const int stride = std::min(plan->dpad, kRotChunk), smem = std::min(nq, kRotQ) * stride * (int)sizeof(float);
  // function attributes are per device: remember the devices this launcher has prepared
  static std::atomic<unsigned long long> attr_devices{0};   // written by any thread that launches
  int attr_dev = 0;
  if (cudaGetDevice(&attr_dev) != cudaSuccess) return cudaErrorInvalidDevice;
  if (attr_dev >= 64 || !((attr_devices.load(std::memory_order_relaxed) >> attr_dev) & 1ull)) {
    cudaError_t e = cudaFuncSetAttribute(rotate_queries_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
    if (e != cudaSuccess) return e;
    if (attr_dev < 64) attr_devices.fetch_or(1ull << attr_dev, std::memory_order_relaxed);
  }
  if (nq >= kRotManyFrom) {
    static std::atomic<unsigned long long> many_devices{0};
    if (attr_dev >= 64 || !((many_devices.load(std::memory_order_relaxed) >> attr_dev) & 1ull)) {
      cudaError_t e = cudaFuncSetAttribute(rotate_many_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
      if (e != cudaSuccess) return e;
      if (attr_dev < 64) many_devices.fetch_or(1ull << attr_dev, std::memory_order_relaxed);
    }
    const int cols = (ncols + kRmRowsPerBlock - 1) / kRmRowsPerBlock, per = rotate_queries_per_cta(cols, nq);
    const dim3 grid((unsigned)cols, (unsigned)((nq + per - 1) / per));
    count_launches(1);
    return launch_dependent(rotate_many_kernel<T>, grid, dim3(32 * kRmWarps), smem, st, plan->dRotCat, ncols, plan->d, plan->dpad, Q, ldq, nq, Qcat,
                            (int64_t)ncols, per, stride);
  }
  const int cols = (ncols + 7) / 8, per = rotate_queries_per_cta(cols, nq);
  const dim3 grid((unsigned)cols, (unsigned)((nq + per - 1) / per));
  count_launches(1);
  return launch_dependent(rotate_queries_kernel<T>, grid, dim3(256), smem, st, plan->dRotCat, ncols, plan->d, plan->dpad, Q, ldq, nq, Qcat, (int64_t)ncols,
                          per, stride);
}

// Q' = Q Pi^T and Q'' = Q S^T side by side: Qcat[nq, ncat*dpad].
cudaError_t prepare_queries(const tq_plan* plan, const void* Q, int q_dtype, int nq, int64_t ldq, float* Qcat,
                            cudaStream_t st) {
  // Both kernels add the same products in the same order, so that a query's rotated form (and hence its
  // estimates) does not depend on how many other queries came with it.
  if (q_dtype == TQ_F32) return launch_rotate_queries(plan, static_cast<const float*>(Q), ldq, nq, Qcat, st);
  return launch_rotate_queries(plan, static_cast<const __nv_bfloat16*>(Q), ldq, nq, Qcat, st);
}

template <int BITS, bool PROD>
cudaError_t launch_scan_few(const scan::ScanArgs& base, int nq, cudaStream_t st) {
  const size_t per_query = (size_t)(PROD ? 2 : 1) * 32 * base.groups * sizeof(float);
  int tile = 8;
  while (tile > 1 && per_query * tile > 200 * 1024) tile >>= 1;
  if (per_query * tile > 220 * 1024) return cudaErrorInvalidConfiguration;
  const int64_t blocks = std::min<int64_t>((base.n + 255) / 256, tc::sm_count() * 2);
  for (int q0 = 0; q0 < nq; q0 += tile) {
    scan::ScanArgs a = base;
    a.q0 = q0;
    a.nq_tile = std::min(tile, nq - q0);
    cudaError_t e = cudaSuccess;
    const size_t smem = per_query * tile;
#define TQ_SCAN_LAUNCH(NQ)                                                                                  \
  {                                                                                                         \
    static std::atomic<unsigned long long> smem_devices{0};                                                 \
    e = allow_largest_smem(reinterpret_cast<const void*>(scan::scan_few_kernel<BITS, NQ, PROD>), smem_devices); \
    if (e == cudaSuccess) scan::scan_few_kernel<BITS, NQ, PROD><<<(unsigned)blocks, 256, smem, st>>>(a);    \
  }
    switch (tile) {
      case 8: TQ_SCAN_LAUNCH(8) break;
      case 4: TQ_SCAN_LAUNCH(4) break;
      case 2: TQ_SCAN_LAUNCH(2) break;
      default: TQ_SCAN_LAUNCH(1) break;
    }
#undef TQ_SCAN_LAUNCH
    if (e != cudaSuccess) return e;
    count_launches(1);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Scores of queries (already prepared in Qcat) against vectors [v0, v0 + cn).
cudaError_t score_block(const tq_plan* plan, const float* Qcat, int nq, int64_t v0, int64_t cn, const uint8_t* idx,
                        const uint8_t* qjl, const float* gamma, const float* norms, float* scores, int64_t lds,
                        cudaStream_t st) {
  const uint8_t* idx_b = idx ? idx + (size_t)v0 * plan->idx_row_bytes : nullptr;
  const uint8_t* qjl_b = qjl ? qjl + (size_t)v0 * plan->qjl_row_bytes : nullptr;
  const float* gamma_b = gamma ? gamma + v0 : nullptr;
  const float* norms_b = norms ? norms + v0 : nullptr;
  const int ncols = plan->ncat * plan->dpad;
  if (nq <= kFewQueries) {
    scan::ScanArgs a;
    a.idx = idx_b;
    a.idx_rb = plan->idx_row_bytes;
    a.qjl = (plan->mode == TQ_PROD) ? qjl_b : nullptr;
    a.qjl_rb = plan->qjl_row_bytes;
    a.gamma = gamma_b;
    a.norms = norms_b;
    a.cb = plan->cb;
    a.d = plan->d;
    a.groups = (plan->d + 31) / 32;
    a.coef = plan->coef;
    a.n = cn;
    a.Qcat = Qcat;
    a.ldq = ncols;
    a.dpad = plan->dpad;
    a.q0 = 0;
    a.nq_tile = 0;
    a.scores = scores;
    a.lds = lds;
    const bool prod = plan->mode == TQ_PROD;
    switch (plan->mse_bits) {
      case 0: return launch_scan_few<0, true>(a, nq, st);
      case 1: return prod ? launch_scan_few<1, true>(a, nq, st) : launch_scan_few<1, false>(a, nq, st);
      case 2: return prod ? launch_scan_few<2, true>(a, nq, st) : launch_scan_few<2, false>(a, nq, st);
      case 3: return prod ? launch_scan_few<3, true>(a, nq, st) : launch_scan_few<3, false>(a, nq, st);
      default: return prod ? launch_scan_few<4, true>(a, nq, st) : launch_scan_few<4, false>(a, nq, st);
    }
  }
  simt::RowsF32 A{Qcat, ncols, nq, ncols};
  simt::Codes B = make_codes(plan, cn, idx_b, qjl_b, gamma_b);
  simt::EpStore ep{scores, lds, nullptr, norms_b};
  return simt::launch_gemm(A, B, ep, (int64_t)nq, cn, ncols, st);
}

}  // namespace

// ======================================================================================
extern "C" int tq_plan_create(int d, int bits, int mode, const float* Pi, const float* S, const float* centroids,
                              tq_plan** out) {
  const char* who = "tq_plan_create";
  TQ_RANGE(who);
  TQ_REQUIRE(out != nullptr, TQ_ERR_INVALID_ARG, "%s: out is NULL", who);
  *out = nullptr;
  TQ_REQUIRE(mode == TQ_MSE || mode == TQ_PROD, TQ_ERR_INVALID_ARG, "%s: unknown mode %d", who, mode);
  TQ_REQUIRE(d >= 2 && d <= TQ_MAX_D, TQ_ERR_UNSUPPORTED, "%s: d=%d outside 2..%d", who, d, TQ_MAX_D);
  const int mse_bits = (mode == TQ_PROD) ? bits - 1 : bits;
  TQ_REQUIRE(bits >= 1 && mse_bits <= 4, TQ_ERR_UNSUPPORTED, "%s: bits=%d unsupported for this mode", who, bits);
  TQ_REQUIRE(Pi != nullptr && centroids != nullptr, TQ_ERR_INVALID_ARG, "%s: Pi / centroids is NULL", who);
  TQ_REQUIRE(mode == TQ_MSE || S != nullptr, TQ_ERR_INVALID_ARG, "%s: S is NULL for a TQ_PROD plan", who);
  const int levels = 1 << mse_bits;
  for (int i = 0; i < levels; ++i) {
    TQ_REQUIRE(std::isfinite(centroids[i]), TQ_ERR_INVALID_ARG, "%s: centroid %d is not finite", who, i);
    TQ_REQUIRE(i == 0 || centroids[i] > centroids[i - 1], TQ_ERR_INVALID_ARG, "%s: centroids must be strictly ascending", who);
  }

  tq_plan* p = new (std::nothrow) tq_plan();
  TQ_REQUIRE(p != nullptr, TQ_ERR_INVALID_ARG, "%s: out of host memory", who);
  std::memset(p, 0, sizeof(*p));
  p->d = d;
  p->dpad = round_up(d, 8);
  p->bits = bits;
  p->mode = mode;
  p->mse_bits = mse_bits;
  p->ncat = (mode == TQ_PROD) ? 2 : 1;
  p->coef = (float)(std::sqrt(M_PI / 2.0) / d);
  p->idx_row_bytes = tq_idx_row_bytes(d, mse_bits);
  p->qjl_row_bytes = tq_qjl_row_bytes(d);
  p->cb.bits = mse_bits;
  for (int i = 0; i < 16; ++i) p->cb.c[i] = (i < levels) ? centroids[i] : 0.f;
  for (int i = 0; i < 15; ++i) p->cb.t[i] = (i + 1 < levels) ? 0.5f * (centroids[i] + centroids[i + 1]) : INFINITY;

  const size_t dd = (size_t)d * d;
  const int ncols = p->ncat * p->dpad;
  auto fail = [&](int code) {
    tq_plan_destroy(p);
    return code;
  };
#define PLAN_CUDA(call, what)                                        \
  do {                                                               \
    cudaError_t e_ = (call);                                         \
    if (e_ != cudaSuccess) {                                         \
      set_error("%s: %s: %s", who, what, cudaGetErrorString(e_));    \
      return fail(TQ_ERR_CUDA);                                      \
    }                                                                \
  } while (0)
  PLAN_CUDA(cudaGetDevice(&p->device), "cudaGetDevice");
  PLAN_CUDA(cudaMalloc(&p->dPi, dd * sizeof(float)), "cudaMalloc Pi");
  PLAN_CUDA(cudaMemcpy(p->dPi, Pi, dd * sizeof(float), cudaMemcpyHostToDevice), "copy Pi");
  std::vector<float> rot((size_t)ncols * p->dpad, 0.f), back((size_t)d * ncols, 0.f);
  for (int i = 0; i < d; ++i) {
    std::memcpy(&rot[(size_t)i * p->dpad], Pi + (size_t)i * d, d * sizeof(float));
    for (int j = 0; j < d; ++j) back[(size_t)j * ncols + i] = Pi[(size_t)i * d + j];
  }
  float* dS = nullptr;
  if (mode == TQ_PROD) {
    for (int i = 0; i < d; ++i) {
      std::memcpy(&rot[(size_t)(p->dpad + i) * p->dpad], S + (size_t)i * d, d * sizeof(float));
      for (int j = 0; j < d; ++j) back[(size_t)j * ncols + p->dpad + i] = S[(size_t)i * d + j];
    }
    PLAN_CUDA(cudaMalloc(&dS, dd * sizeof(float)), "cudaMalloc S");
    cudaError_t e = cudaMemcpy(dS, S, dd * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMalloc(&p->dSp, dd * sizeof(float));
    if (e == cudaSuccess) {
      dim3 grid((d + 15) / 16, (d + 15) / 16), block(16, 16);
      sprime_kernel<<<grid, block>>>(dS, p->dPi, p->dSp, d);
      e = cudaGetLastError();
      if (e == cudaSuccess) e = cudaDeviceSynchronize();
    }
    cudaFree(dS);
    PLAN_CUDA(e, "S' = S Pi^T");
  }
  PLAN_CUDA(cudaMalloc(&p->dRotCat, rot.size() * sizeof(float)), "cudaMalloc RotCat");
  PLAN_CUDA(cudaMemcpy(p->dRotCat, rot.data(), rot.size() * sizeof(float), cudaMemcpyHostToDevice), "copy RotCat");
  PLAN_CUDA(cudaMalloc(&p->dBackT, back.size() * sizeof(float)), "cudaMalloc BackT");
  PLAN_CUDA(cudaMemcpy(p->dBackT, back.data(), back.size() * sizeof(float), cudaMemcpyHostToDevice), "copy BackT");
  PLAN_CUDA(cudaMalloc(&p->d_status, sizeof(int)), "cudaMalloc status");
  PLAN_CUDA(cudaMemset(p->d_status, 0, sizeof(int)), "clear status");
  if (tc::supported(d)) {
    PLAN_CUDA(tc::build_matrix_limbs(p->dPi, d, d, p->dpad, &p->pi_limbs), "bf16 limbs of Pi");
    if (mode == TQ_PROD)
      PLAN_CUDA(tc::build_matrix_limbs(p->dSp, d, d, p->dpad, &p->sp_limbs), "bf16 limbs of S'");
    p->tc_ok = 1;
  }
  PLAN_CUDA(sq::plan_init(p), "transpose of S'");
  PLAN_CUDA(dq::plan_init(p, Pi, mode == TQ_PROD ? S : nullptr), "fp16 limbs of Pi^T and S^T");
  mscan::plan_init(p);
  nscan::plan_init(p);
  PLAN_CUDA(cudaDeviceSynchronize(), "synchronize");
#undef PLAN_CUDA
  *out = p;
  return TQ_OK;
}

extern "C" int tq_plan_destroy(tq_plan* plan) {
  if (!plan) return TQ_OK;
  cudaFree(plan->dPi);
  cudaFree(plan->dSp);
  cudaFree(plan->dRotCat);
  cudaFree(plan->dBackT);
  cudaFree(plan->d_status);
  tc::free_matrix_limbs(&plan->pi_limbs);
  tc::free_matrix_limbs(&plan->sp_limbs);
  dq::plan_free(plan);
  sq::plan_free(plan);
  delete plan;
  return TQ_OK;
}

extern "C" int tq_plan_set_layout(tq_plan* plan, int layout) {
  const char* who = "tq_plan_set_layout";
  TQ_REQUIRE(plan != nullptr, TQ_ERR_INVALID_ARG, "%s: plan is NULL", who);
  TQ_REQUIRE(layout == TQ_LAYOUT_CANONICAL || layout == TQ_LAYOUT_NIBBLE, TQ_ERR_INVALID_ARG, "%s: unknown layout %d", who, layout);
  TQ_REQUIRE(layout == TQ_LAYOUT_CANONICAL || plan->nb.ok, TQ_ERR_UNSUPPORTED,
             "%s: the nibble layout needs a TQ_PROD plan with b = 4, d >= 128 (d=%d, b=%d, mode=%d)", who, plan->d, plan->bits,
             plan->mode);
  plan->layout = layout;
  return TQ_OK;
}

extern "C" int tq_plan_layout(const tq_plan* plan) { return plan ? plan->layout : -1; }

extern "C" int tq_convert_layout(const tq_plan* plan, int64_t n, uint8_t* idx, uint8_t* qjl, int from, int to, void* stream) {
  const char* who = "tq_convert_layout";
  TQ_RANGE(who);
  int rc = check_plan(plan, who);
  if (rc) return rc;
  TQ_REQUIRE(n >= 0, TQ_ERR_INVALID_ARG, "%s: n is negative", who);
  for (int l : {from, to})
    TQ_REQUIRE(l == TQ_LAYOUT_CANONICAL || l == TQ_LAYOUT_NIBBLE, TQ_ERR_INVALID_ARG, "%s: unknown layout %d", who, l);
  TQ_REQUIRE(plan->nb.ok, TQ_ERR_UNSUPPORTED, "%s: this plan has no nibble layout (TQ_PROD, b = 4, d >= 128 only)", who);
  if (n == 0 || from == to) return TQ_OK;
  TQ_REQUIRE(idx != nullptr && qjl != nullptr, TQ_ERR_INVALID_ARG, "%s: idx / qjl is NULL", who);
  TQ_REQUIRE(aligned(idx, 16) && aligned(qjl, 16), TQ_ERR_ALIGNMENT, "%s: idx / qjl is not 16-byte aligned", who);
  return nscan::convert(plan, n, idx, qjl, to, static_cast<cudaStream_t>(stream), who);
}

// A one-warp kernel whose barrier nobody arrives at: the bounded wait must give up after `limit` cycles, raise the
// CTA's abort flag and record TQ_ERR_TIMEOUT in the plan's status word.  Nothing traps, nothing spins past the limit.
__global__ void wait_timeout_selftest_kernel(int* status, long long limit) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    tc::mbar_init(&bar, 1);
    abort_flag = 0;
    tc::fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const bool ok = tc::mbar_wait_slow(&bar, 0u, &abort_flag, status, limit);
    if (ok || abort_flag != 1) atomicExch(status, TQ_ERR_CUDA);   // anything but "gave up and said so" is a different error
  }
}

extern "C" int tq_selftest_wait_timeout(tq_plan* plan, long long limit_cycles, void* stream) {
  const char* who = "tq_selftest_wait_timeout";
  TQ_RANGE(who);
  int rc = check_plan(plan, who);
  if (rc) return rc;
  TQ_REQUIRE(limit_cycles >= 1 && limit_cycles <= 100000000LL, TQ_ERR_INVALID_ARG, "%s: limit outside 1..1e8 cycles", who);
  wait_timeout_selftest_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(plan->d_status, limit_cycles);
  count_launches(1);
  TQ_CHECK_CUDA(cudaGetLastError(), who);
  return TQ_OK;
}

extern "C" int tq_plan_status(tq_plan* plan) {
  const char* who = "tq_plan_status";
  TQ_RANGE(who);
  TQ_REQUIRE(plan != nullptr, TQ_ERR_INVALID_ARG, "%s: plan is NULL", who);
  TQ_CHECK_CUDA(cudaDeviceSynchronize(), who);
  int st = 0;
  TQ_CHECK_CUDA(cudaMemcpy(&st, plan->d_status, sizeof(int), cudaMemcpyDeviceToHost), who);
  if (st != 0) {
    cudaMemset(plan->d_status, 0, sizeof(int));
    if (st == TQ_ERR_BOUNDS) {
      set_error("%s: a device-side index check of the TQ_DEBUG build failed (the access was skipped)", who);
      return TQ_ERR_BOUNDS;
    }
    if (st != TQ_ERR_TIMEOUT) {
      set_error("%s: a kernel recorded the unexpected status %d", who, st);
      return TQ_ERR_CUDA;
    }
    set_error("%s: a kernel gave up a bounded wait (pipeline stall); results of that call are invalid", who);
    return TQ_ERR_TIMEOUT;
  }
  return TQ_OK;
}

extern "C" size_t tq_workspace_bytes(const tq_plan* plan, int op, int64_t n, int nq, int k) {
  if (!plan || n < 0 || nq < 0) return 0;
  (void)k;
  switch (op) {
    case TQ_OP_QUANTIZE:
      if (n == 0) return 0;
      if (plan->tc_ok)
      {
        // rows per launch: 65,536 at d = 1536 and more for short rows (same scratch bytes), so that a launch of the
        // persistent GEMM stays long against its prologue and the launch sequence
        const int64_t chunk = std::min<int64_t>(kTensorChunk * std::max(1, 1536 / plan->dpad), 8 * kTensorChunk);
        // (half as many rows again when n exceeds the chunk: fewer, longer launches measured faster than 65,536-row
        // ones, also than 65,536-row ones whose operand split ran beside the previous block's GEMMs)
        return align_up((size_t)std::min<int64_t>(round_up64(n, 128), n > chunk ? chunk + chunk / 2 : chunk) *
                            tc::scratch_bytes_per_row(plan),
                        256);
      }
      if (plan->mode != TQ_PROD) return 0;
      return align_up((size_t)std::min<int64_t>(n, kResidualChunk) * plan->dpad * sizeof(float), 256);
    case TQ_OP_SCORE:
      return plan->ms.ok ? ms_score_fixed(plan, nq) : qcat_bytes(plan, nq);
    case TQ_OP_TOPK:
      if (plan->ms.ok)
        return std::max(screens(plan, nq, n, k) ? qcat_bytes(plan, nq) + screen_pref(plan, nq, n) : 0,
                        ms_topk_fixed(plan, nq) + align_up((size_t)pick_engine(plan, nq).qpp *
                                                               std::max<int64_t>(std::min<int64_t>(n, pick_engine(plan, nq).dense_rows_pref), kDenseRowsMin) *
                                                               sizeof(float),
                                                           256));
      return qcat_bytes(plan, nq) + align_up((size_t)nq * std::min<int64_t>(n, kTopkBlockPref) * sizeof(float), 256);
    case TQ_OP_WSUM: {
      const size_t ncols = (size_t)plan->ncat * plan->dpad;
      const size_t chunks = (size_t)((n + attend::WS_TOK - 1) / attend::WS_TOK);
      return align_up((size_t)nq * ncols * sizeof(float), 256) +
             align_up(chunks * std::min(nq, attend::WS_NW) * ncols * sizeof(float), 256);
    }
    default:
      return 0;
  }
}

extern "C" int tq_quantize_mse(const tq_plan* plan, const void* X, int x_dtype, int64_t n, int64_t ldx, uint8_t* idx,
                               float* norms, void* scratch, size_t scratch_bytes, void* stream) {
  const char* who = "tq_quantize_mse";
  TQ_RANGE(who);
  int rc = check_plan(plan, who);
  if (rc) return rc;
  TQ_REQUIRE(plan->mode == TQ_MSE, TQ_ERR_INVALID_ARG, "%s: plan was created for TQ_PROD", who);
  TQ_REQUIRE(n >= 0, TQ_ERR_INVALID_ARG, "%s: n is negative", who);
  if (n == 0) return TQ_OK;
  if ((rc = check_rows(who, "X", X, x_dtype, n, ldx, plan->d))) return rc;
  TQ_REQUIRE(idx != nullptr, TQ_ERR_INVALID_ARG, "%s: idx is NULL", who);
  TQ_REQUIRE(aligned(idx, 16) && aligned(norms, 4), TQ_ERR_ALIGNMENT, "%s: idx / norms is misaligned", who);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (plan->tc_ok) {
    const size_t need = tq_workspace_bytes(plan, TQ_OP_QUANTIZE, std::min<int64_t>(n, 128), 0, 0);
    TQ_REQUIRE(scratch != nullptr && scratch_bytes >= need, TQ_ERR_WORKSPACE, "%s: scratch of %zu bytes, at least %zu needed",
               who, scratch_bytes, need);
    TQ_REQUIRE(aligned(scratch, 256), TQ_ERR_ALIGNMENT, "%s: scratch is not 256-byte aligned", who);
    return tc::quantize(plan, X, x_dtype, n, ldx, idx, nullptr, nullptr, norms, scratch, scratch_bytes, st, who);
  }
  if (plan->sq.ok) return sq::quantize(plan, X, x_dtype, n, ldx, idx, nullptr, nullptr, norms, st, who);
  if (norms) TQ_CHECK_CUDA(compute_norms(X, x_dtype, n, ldx, plan->d, norms, st), who);
  if (has_pad_words(plan->d, plan->mse_bits, plan->idx_row_bytes))
    TQ_CHECK_CUDA(cudaMemsetAsync(idx, 0, (size_t)n * plan->idx_row_bytes, st), who);
  TQ_CHECK_CUDA(dispatch_rotate_quantize<0>(plan, X, x_dtype, n, ldx, norms, idx, nullptr, 0, st), who);
  return TQ_OK;
}

extern "C" int tq_quantize_prod(const tq_plan* plan, const void* X, int x_dtype, int64_t n, int64_t ldx, uint8_t* idx,
                                uint8_t* qjl, float* gamma, float* norms, void* scratch, size_t scratch_bytes,
                                void* stream) {
  const char* who = "tq_quantize_prod";
  TQ_RANGE(who);
  int rc = check_plan(plan, who);
  if (rc) return rc;
  TQ_REQUIRE(plan->mode == TQ_PROD, TQ_ERR_INVALID_ARG, "%s: plan was created for TQ_MSE", who);
  TQ_REQUIRE(n >= 0, TQ_ERR_INVALID_ARG, "%s: n is negative", who);
  if (n == 0) return TQ_OK;
  if ((rc = check_rows(who, "X", X, x_dtype, n, ldx, plan->d))) return rc;
  if ((rc = check_codes(plan, who, idx, qjl, gamma))) return rc;
  TQ_REQUIRE(aligned(norms, 4), TQ_ERR_ALIGNMENT, "%s: norms is misaligned", who);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (plan->tc_ok) {
    const size_t least = tq_workspace_bytes(plan, TQ_OP_QUANTIZE, std::min<int64_t>(n, 128), 0, 0);
    TQ_REQUIRE(scratch != nullptr && scratch_bytes >= least, TQ_ERR_WORKSPACE,
               "%s: scratch of %zu bytes, at least %zu needed", who, scratch_bytes, least);
    TQ_REQUIRE(aligned(scratch, 256), TQ_ERR_ALIGNMENT, "%s: scratch is not 256-byte aligned", who);
    // (the GEMM epilogues write whichever layout the plan has)
    return tc::quantize(plan, X, x_dtype, n, ldx, idx, qjl, gamma, norms, scratch, scratch_bytes, st, who);
  }
  const size_t need = tq_workspace_bytes(plan, TQ_OP_QUANTIZE, n, 0, 0);
  TQ_REQUIRE(scratch != nullptr && scratch_bytes >= need, TQ_ERR_WORKSPACE, "%s: scratch of %zu bytes, %zu needed", who,
             scratch_bytes, need);
  TQ_REQUIRE(aligned(scratch, 16), TQ_ERR_ALIGNMENT, "%s: scratch is not 16-byte aligned", who);
  if (plan->sq.ok) return sq::quantize(plan, X, x_dtype, n, ldx, idx, qjl, gamma, norms, st, who);
  const int d = plan->d;
  const int64_t ldE = plan->dpad;
  float* E = static_cast<float*>(scratch);
  int64_t chunk = (int64_t)(scratch_bytes / ((size_t)ldE * sizeof(float)));
  if (chunk < n) chunk = chunk / simt::BM * simt::BM;
  chunk = std::min(chunk, n);
  TQ_REQUIRE(chunk > 0, TQ_ERR_WORKSPACE, "%s: scratch too small for one block of rows", who);

  if (norms) TQ_CHECK_CUDA(compute_norms(X, x_dtype, n, ldx, d, norms, st), who);
  if (has_pad_words(d, plan->mse_bits, plan->idx_row_bytes))
    TQ_CHECK_CUDA(cudaMemsetAsync(idx, 0, (size_t)n * plan->idx_row_bytes, st), who);
  if (has_pad_words(d, 1, plan->qjl_row_bytes))
    TQ_CHECK_CUDA(cudaMemsetAsync(qjl, 0, (size_t)n * plan->qjl_row_bytes, st), who);
  const size_t xsz = (x_dtype == TQ_F32) ? 4 : 2;
  for (int64_t r0 = 0; r0 < n; r0 += chunk) {
    const int64_t rows = std::min(chunk, n - r0);
    const void* Xc = static_cast<const char*>(X) + (size_t)r0 * ldx * xsz;
    uint8_t* idx_c = idx ? idx + (size_t)r0 * plan->idx_row_bytes : nullptr;
    // Stage 1: y = Pi x, idx, rotated residual e = y/nu - c[idx]   (Algorithm 2, steps idx and r)
    TQ_CHECK_CUDA(dispatch_rotate_quantize<1>(plan, Xc, x_dtype, rows, ldx, norms ? norms + r0 : nullptr, idx_c, E, ldE, st), who);
    // gamma = ||r|| = ||e||
    TQ_CHECK_CUDA(launch_row_norm(E, ldE, rows, d, gamma + r0, st), who);
    // Stage 2: qjl = sign(S r) = sign(S' e)
    simt::EpQuantize<1, 2> ep;
    ep.cb = plan->cb;
    ep.nu = nullptr;
    ep.out = qjl + (size_t)r0 * plan->qjl_row_bytes;
    ep.out_rb = plan->qjl_row_bytes;
    ep.E = nullptr;
    ep.ldE = 0;
    ep.d = d;
    simt::RowsF32 A{E, ldE, rows, d};
    simt::RowsF32 B{plan->dSp, d, d, d};
    TQ_CHECK_CUDA(simt::launch_gemm(A, B, ep, rows, (int64_t)d, d, st), who);
  }
  return TQ_OK;
}

extern "C" int tq_dequantize(const tq_plan* plan, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma,
                             const float* norms, float* Xhat, int64_t ldxh, void* stream) {
  const char* who = "tq_dequantize";
  TQ_RANGE(who);
  int rc = check_plan(plan, who);
  if (rc) return rc;
  TQ_REQUIRE(n >= 0, TQ_ERR_INVALID_ARG, "%s: n is negative", who);
  if (n == 0) return TQ_OK;
  if ((rc = check_codes(plan, who, idx, qjl, gamma))) return rc;
  TQ_REQUIRE(Xhat != nullptr, TQ_ERR_INVALID_ARG, "%s: Xhat is NULL", who);
  TQ_REQUIRE(ldxh >= plan->d, TQ_ERR_INVALID_ARG, "%s: ldxh < d", who);
  TQ_REQUIRE(aligned(Xhat, 16), TQ_ERR_ALIGNMENT, "%s: Xhat is not 16-byte aligned", who);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (plan->dq.ok) return dq::dequantize(plan, n, idx, qjl, gamma, norms, Xhat, ldxh, st, who);
  const int ncols = plan->ncat * plan->dpad;
  simt::Codes A = make_codes(plan, n, idx, qjl, gamma);
  simt::RowsF32 B{plan->dBackT, ncols, plan->d, ncols};
  simt::EpStore ep{Xhat, ldxh, norms, nullptr};
  TQ_CHECK_CUDA(simt::launch_gemm(A, B, ep, n, (int64_t)plan->d, ncols, st), who);
  return TQ_OK;
}

// Engine for a score call whose workspace holds `avail` bytes behind the rotated queries: the preferred one, or,
// when the many-query engine's operand does not fit, the few-query engine (same estimates, more passes).
static bool engine_that_fits(const tq_plan* plan, int nq, size_t avail, ScanEngine* out) {
  *out = pick_engine(plan, nq);
  if (align_up(out->ws_bytes, 256) <= avail) return true;
  if (!out->tc) return false;
  *out = pick_engine(plan, std::min(nq, 4));
  return align_up(out->ws_bytes, 256) <= avail;
}

// tq_score on a workspace that is known to be large enough: rotated queries first, then the engine's operand.
static int score_on_workspace(const tq_plan* plan, const ScanEngine* eng, const void* Q, int q_dtype, int nq, int64_t ldq,
                              int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma, const float* norms,
                              float* scores, int64_t lds, void* workspace, cudaStream_t st, const char* who) {
  int rc;
  float* Qcat = static_cast<float*>(workspace);
  TQ_CHECK_CUDA(prepare_queries(plan, Q, q_dtype, nq, ldq, Qcat, st), who);
  if (plan->ms.ok) {
    void* msw = static_cast<char*>(workspace) + qcat_bytes(plan, nq);
    for (int q0 = 0; q0 < nq; q0 += eng->qpp) {
      const int nqp = std::min(eng->qpp, nq - q0);
      if ((rc = engine_prepare(*eng, Qcat, q0, nq, msw, st, who))) return rc;
      if ((rc = engine_run(*eng, q0, nqp, n, idx, qjl, gamma, norms, scores + (int64_t)q0 * lds, lds, nullptr, nullptr, msw, st, who)))
        return rc;
    }
    return TQ_OK;
  }
  TQ_CHECK_CUDA(score_block(plan, Qcat, nq, 0, n, idx, qjl, gamma, norms, scores, lds, st), who);
  return TQ_OK;
}

static int check_score_args(const tq_plan* plan, const char* who, const void* Q, int q_dtype, int nq, int64_t ldq, int64_t n,
                            const uint8_t* idx, const uint8_t* qjl, const float* gamma, const float* scores, int64_t lds) {
  int rc;
  if ((rc = check_rows(who, "Q", Q, q_dtype, nq, ldq, plan->d))) return rc;
  if ((rc = check_codes(plan, who, idx, qjl, gamma))) return rc;
  TQ_REQUIRE(scores != nullptr && lds >= n, TQ_ERR_INVALID_ARG, "%s: scores is NULL or lds < n", who);
  TQ_REQUIRE(aligned(scores, 16), TQ_ERR_ALIGNMENT, "%s: scores is not 16-byte aligned", who);
  return TQ_OK;
}

extern "C" int tq_score(const tq_plan* plan, const void* Q, int q_dtype, int nq, int64_t ldq, int64_t n,
                        const uint8_t* idx, const uint8_t* qjl, const float* gamma, const float* norms, float* scores,
                        int64_t lds, void* workspace, size_t workspace_bytes, void* stream) {
  const char* who = "tq_score";
  TQ_RANGE(who);
  int rc = check_plan(plan, who);
  if (rc) return rc;
  TQ_REQUIRE(n >= 0 && nq >= 0, TQ_ERR_INVALID_ARG, "%s: negative size", who);
  if (n == 0 || nq == 0) return TQ_OK;
  if ((rc = check_score_args(plan, who, Q, q_dtype, nq, ldq, n, idx, qjl, gamma, scores, lds))) return rc;
  const size_t need = tq_workspace_bytes(plan, TQ_OP_SCORE, n, nq, 0);
  TQ_REQUIRE(workspace != nullptr && workspace_bytes >= need, TQ_ERR_WORKSPACE, "%s: workspace of %zu bytes, %zu needed",
             who, workspace_bytes, need);
  TQ_REQUIRE(aligned(workspace, 16), TQ_ERR_ALIGNMENT, "%s: workspace is not 16-byte aligned", who);
  ScanEngine eng{};
  if (plan->ms.ok) eng = pick_engine(plan, nq);
  return score_on_workspace(plan, &eng, Q, q_dtype, nq, ldq, n, idx, qjl, gamma, norms, scores, lds, workspace,
                            static_cast<cudaStream_t>(stream), who);
}

// ---- prepared queries: rotation and operand set-up once, any number of scans afterwards
// Buffer: rotated queries, then one engine workspace per pass (per group of 256 queries on the tcgen05 engine).
static size_t prepared_slots(const ScanEngine& e, int nq) {
  const int per = e.tc ? kGroupQueries : e.qpp;
  return (size_t)((nq + per - 1) / per);
}

extern "C" size_t tq_query_bytes(const tq_plan* plan, int nq) {
  if (!plan || nq <= 0) return 0;
  size_t b = qcat_bytes(plan, nq);
  if (plan->ms.ok) {
    const ScanEngine e = pick_engine(plan, nq);
    b += prepared_slots(e, nq) * align_up(e.ws_bytes, 256);
  }
  return b;
}

extern "C" int tq_query_prepare(const tq_plan* plan, const void* Q, int q_dtype, int nq, int64_t ldq, void* prepared,
                                size_t prepared_bytes, void* stream) {
  const char* who = "tq_query_prepare";
  TQ_RANGE(who);
  int rc = check_plan(plan, who);
  if (rc) return rc;
  TQ_REQUIRE(nq >= 0, TQ_ERR_INVALID_ARG, "%s: negative size", who);
  if (nq == 0) return TQ_OK;
  if ((rc = check_rows(who, "Q", Q, q_dtype, nq, ldq, plan->d))) return rc;
  const size_t need = tq_query_bytes(plan, nq);
  TQ_REQUIRE(prepared != nullptr && prepared_bytes >= need, TQ_ERR_WORKSPACE, "%s: buffer of %zu bytes, %zu needed", who,
             prepared_bytes, need);
  TQ_REQUIRE(aligned(prepared, 256), TQ_ERR_ALIGNMENT, "%s: buffer is not 256-byte aligned", who);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  float* Qcat = static_cast<float*>(prepared);
  TQ_CHECK_CUDA(prepare_queries(plan, Q, q_dtype, nq, ldq, Qcat, st), who);
  if (!plan->ms.ok) return TQ_OK;
  const ScanEngine eng = pick_engine(plan, nq);
  const size_t slot = align_up(eng.ws_bytes, 256);
  char* base = static_cast<char*>(prepared) + qcat_bytes(plan, nq);
  const int per = eng.tc ? kGroupQueries : eng.qpp;
  for (int q0 = 0; q0 < nq; q0 += per)
    if ((rc = engine_prepare(eng, Qcat, q0, nq, base + (size_t)(q0 / per) * slot, st, who))) return rc;
  return TQ_OK;
}

extern "C" int tq_score_prepared(const tq_plan* plan, const void* prepared, int nq, int64_t n, const uint8_t* idx,
                                 const uint8_t* qjl, const float* gamma, const float* norms, float* scores, int64_t lds,
                                 void* stream) {
  const char* who = "tq_score_prepared";
  TQ_RANGE(who);
  int rc = check_plan(plan, who);
  if (rc) return rc;
  TQ_REQUIRE(n >= 0 && nq >= 0, TQ_ERR_INVALID_ARG, "%s: negative size", who);
  if (n == 0 || nq == 0) return TQ_OK;
  TQ_REQUIRE(prepared != nullptr && aligned(prepared, 256), TQ_ERR_INVALID_ARG, "%s: prepared buffer is NULL or misaligned", who);
  if ((rc = check_codes(plan, who, idx, qjl, gamma))) return rc;
  TQ_REQUIRE(scores != nullptr && lds >= n, TQ_ERR_INVALID_ARG, "%s: scores is NULL or lds < n", who);
  TQ_REQUIRE(aligned(scores, 16), TQ_ERR_ALIGNMENT, "%s: scores is not 16-byte aligned", who);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const float* Qcat = static_cast<const float*>(prepared);
  if (!plan->ms.ok) {
    TQ_CHECK_CUDA(score_block(plan, Qcat, nq, 0, n, idx, qjl, gamma, norms, scores, lds, st), who);
    return TQ_OK;
  }
  const ScanEngine eng = pick_engine(plan, nq);
  const size_t slot = align_up(eng.ws_bytes, 256);
  const char* base = static_cast<const char*>(prepared) + qcat_bytes(plan, nq);
  const int per = eng.tc ? kGroupQueries : eng.qpp;
  for (int q0 = 0; q0 < nq; q0 += eng.qpp) {
    const int nqp = std::min(eng.qpp, nq - q0);
    const void* ws = base + (size_t)(q0 / per) * slot;
    // the codes may have been written by the kernel just ahead in the stream: no early start of the scan here
    if (eng.nib) rc = nscan::run(plan, nqp, n, idx, qjl, gamma, norms, scores + (int64_t)q0 * lds, lds, nullptr, nullptr, ws, false, st, who);
    else rc = engine_run(eng, q0, nqp, n, idx, qjl, gamma, norms, scores + (int64_t)q0 * lds, lds, nullptr, nullptr, ws, st, who);
    if (rc) return rc;
  }
  return TQ_OK;
}

// Pilot rows m of a search for the k best of n: the pass over all rows then has n / m times as many candidates as the pilot has
// scores down to the threshold, which are k where it meets the k-th best exactly.  That number varies like a sum of k
// exponentials, so that at k = 1 the count is four times the expected one in one query of 55, and one overflow of a list of 32,768
// has all rows scored again for the whole pass (k = 1, 64 queries, 34 * 10^6 rows, 8,192 expected: 28.3 ms instead of 5.5).
// m = n (k + 8) / 8192 expects 910 at k = 1 and 7,585 at k = 100; a larger pilot costs a longer pilot scan and selection.
static int64_t pilot_rows(int64_t n, int k, int64_t most) {
  const int64_t m = std::max<int64_t>(round_up64((int64_t)((double)n * (k + 8) / 8192.0), 256), 4096);
  return std::min<int64_t>(m, std::min<int64_t>(most / 256 * 256, n));
}

// Dense block flow over the queries of one pass: the whole job for small n, the guarded last resort of a filtered search otherwise.
static int topk_dense(const ScanEngine& eng, int q0, int nqp, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma,
                      const float* norms, int k, float* ts, int32_t* ti, float* dense, int64_t dense_floats, const int* guard, void* msw,
                      cudaStream_t st, const char* who) {
  int rc;
  const size_t xrb = eng.plan->idx_row_bytes, qrb = eng.plan->qjl_row_bytes;
  int64_t block = std::min<int64_t>(dense_floats / eng.qpp, n);
  if (block < n) block = block / 256 * 256;
  for (int64_t v0 = 0; v0 < n; v0 += block) {
    const int64_t cn = std::min(block, n - v0);
    if ((rc = engine_run(eng, q0, nqp, cn, idx ? idx + (size_t)v0 * xrb : nullptr, qjl ? qjl + (size_t)v0 * qrb : nullptr,
                         gamma ? gamma + v0 : nullptr, norms ? norms + v0 : nullptr, dense, block, nullptr, guard, msw, st, who)))
      return rc;
    TQ_CHECK_CUDA(mscan::select_topk(dense, nullptr, nullptr, (int)block, (int)cn, (int)v0, nqp, k, v0 > 0 ? 1 : 0, ts, ti,
                                     nullptr, nullptr, guard, nullptr, nullptr, st), who);
  }
  return TQ_OK;
}

// Top-k of many queries by screening: lower bounds of samples' estimates give a threshold that k rows reach, the rows whose upper
// bounds reach it are listed, and those whose upper bounds reach the list's k-th lower bound are scored exactly.
// A pass of the exact engine among whose queries one has more rows to score than that pays for (rows all alike at the top, rows that
// the bounds do not cover) is run, with the k-th lower bounds as its thresholds.  Only where its lists overflow too the rows are
// scored densely, whose selection out of all scores takes longer than the scan (12,000 equal rows at the top for 256 queries, d = 200,
// k = 10, 10^6 rows: 12.6 ms without the filtered passes between, 4.7 with them; they cost 5 us per 256 queries where they are off).
static int topk_screened(const ScanEngine& eng, const float* Qcat, int nq, int64_t n, const uint8_t* idx, const uint8_t* qjl,
                         const float* gamma, const float* norms, int k, float* top_scores, int32_t* top_ids, char* ws, size_t ws_bytes,
                         cudaStream_t st, const char* who) {
  int rc;
  const tq_plan* plan = eng.plan;
  const ScreenSpace sp = screen_space(plan);
  void* msw = ws;
  char* p = ws + align_up(eng.ws_bytes, 256);
  auto at = [&](size_t offset) { return static_cast<void*>(p + offset); };
  float *tau = (float*)at(sp.tau), *kth = (float*)at(sp.kth), *cand_s = (float*)at(sp.cand_s), *left_s = (float*)at(sp.left_s);
  int *count = (int*)at(sp.count), *count1 = (int*)at(sp.count1), *left = (int*)at(sp.left), *flag = (int*)at(sp.flag),
      *cand_i = (int*)at(sp.cand_i), *left_i = (int*)at(sp.left_i);
  void* operand = at(sp.operand);
  float* dense = (float*)at(sp.total);
  const int64_t dense_floats = (int64_t)((ws + ws_bytes - reinterpret_cast<char*>(dense)) / sizeof(float));
  const ScreenSamples sm = screen_samples(n, k, dense_floats / screen::kQueries);
  static_assert(screen::kQueries == kGroupQueries, "one exact operand per screened pass");
  constexpr int kFlags = screen::kQueries / kScreenPass;
  int *flag2 = flag + kFlags, *unused = flag2 + kFlags;
  // lists of the filtered exact passes: in the dense buffer where it has room for longer ones than the screening lists
  const int64_t room = dense_floats / (2 * screen::kQueries);
  const int xcap = (int)std::min<int64_t>(std::max<int64_t>(room, kScreenCap), kCandCap);
  float* x_s = room > kScreenCap ? dense : cand_s;
  int* x_i = room > kScreenCap ? reinterpret_cast<int*>(dense + (int64_t)screen::kQueries * xcap) : cand_i;
  const screen::QueryTerms* terms = screen::query_terms(plan, operand);
  for (int q0 = 0; q0 < nq; q0 += screen::kQueries) {
    const int nqp = std::min(screen::kQueries, nq - q0);
    float* ts = top_scores + (size_t)q0 * k;
    int32_t* ti = top_ids + (size_t)q0 * k;
    if ((rc = engine_prepare(eng, Qcat, q0, nq, msw, st, who))) return rc;
    if ((rc = screen::prepare(plan, Qcat + (size_t)q0 * plan->ncat * plan->dpad, nqp, operand, st, who))) return rc;
    auto filter = [&](int64_t rows, int64_t step, int* counts) {
      return screen::run(plan, nqp, rows, idx, qjl, gamma, norms, nullptr, 0, tau, counts, cand_s, cand_i, kScreenCap, operand, st, who, step);
    };
    if ((rc = screen::run(plan, nqp, sm.dense, idx, qjl, gamma, norms, dense, sm.dense, nullptr, nullptr, nullptr, nullptr, 0, operand, st, who,
                          sm.dense_step)))
      return rc;
    TQ_CHECK_CUDA(mscan::select_topk(dense, nullptr, nullptr, (int)sm.dense, (int)sm.dense, 0, nqp, k, 0, nullptr, nullptr, tau, nullptr, nullptr,
                                     sm.first > 0 ? count1 : count, sm.first > 0 ? unused : flag, st, eng.qpp), who);
    if (sm.first > 0) {   // (a list that is too short here still gives a threshold that k rows reach)
      if ((rc = filter(sm.first, sm.first_step, count1))) return rc;
      TQ_CHECK_CUDA(mscan::select_topk(cand_s, cand_i, count1, kScreenCap, 0, 0, nqp, k, 0, nullptr, nullptr, tau, nullptr, nullptr, count, flag, st,
                                       eng.qpp), who);
    }
    if ((rc = filter(n, 1, count))) return rc;
    TQ_CHECK_CUDA(mscan::select_topk(cand_s, cand_i, count, kScreenCap, 0, 0, nqp, k, 0, nullptr, nullptr, kth, nullptr, nullptr, left, unused, st,
                                     eng.qpp), who);
    if ((rc = tscan::rescore(plan, nqp, n, idx, qjl, gamma, norms, msw, terms, tau, kth, count, cand_s, cand_i, kScreenCap,
                             k, left_s, left_i, left, flag, eng.qpp, st, who)))
      return rc;
    TQ_CHECK_CUDA(mscan::select_topk(left_s, left_i, left, screen::kSurvivors, 0, 0, nqp, k, 0, ts, ti, nullptr, nullptr, nullptr, count1, flag2, st,
                                     eng.qpp), who);
    mscan::Filter f{kth, count1, x_s, x_i, xcap};
    if ((rc = engine_run(eng, q0, nqp, n, idx, qjl, gamma, norms, nullptr, 0, &f, flag, msw, st, who))) return rc;
    TQ_CHECK_CUDA(mscan::select_topk(x_s, x_i, count1, xcap, 0, 0, nqp, k, 0, ts, ti, nullptr, flag2, flag, nullptr, nullptr, st, eng.qpp), who);
    for (int s = 0; s < nqp; s += eng.qpp)   // (the buffer holds the scores of one pass)
      if ((rc = topk_dense(eng, q0 + s, std::min(eng.qpp, nqp - s), n, idx, qjl, gamma, norms, k, ts + (size_t)s * k, ti + (size_t)s * k, dense,
                           dense_floats, flag2 + s / eng.qpp, msw, st, who)))
        return rc;
  }
  return TQ_OK;
}

// Top-k through the tensor-path scan.  Large n: a pilot pass over a sample of the rows gives, per query,
// the k-th best score among them -- a lower bound on the final k-th score -- and the full pass
// keeps only (score, id) pairs at or above it; a final selection sorts the survivors.  Should a
// candidate list overflow (massive ties, adversarial order) a device-side flag switches on a
// dense block-by-block rescue pass that is otherwise launched as a no-op.
static int topk_ms(const tq_plan* plan, const float* Qcat, int nq, int64_t n, const uint8_t* idx, const uint8_t* qjl,
                   const float* gamma, const float* norms, int k, float* top_scores, int32_t* top_ids, char* ws,
                   size_t ws_bytes, cudaStream_t st, const char* who) {
  int rc;
  // (a workspace of the documented minimum has no room for the lists)
  if (screens(plan, nq, n, k) && ws_bytes >= screen_least(plan))
    return topk_screened(pick_engine(plan, nq), Qcat, nq, n, idx, qjl, gamma, norms, k, top_scores, top_ids, ws, ws_bytes, st, who);
  const ScanEngine eng = pick_engine(plan, nq);
  void* msw = ws;
  char* p = ws + align_up(eng.ws_bytes, 256);
  float* tau = reinterpret_cast<float*>(p);          // [qpp] (qpp <= 64: 256 bytes)
  int* count = reinterpret_cast<int*>(p + 256);      // [qpp], then the overflow flag
  int* overflow = count + eng.qpp;
  p += 1024;
  float* cand_s = reinterpret_cast<float*>(p);
  int* cand_i = reinterpret_cast<int*>(p + (size_t)eng.qpp * kCandCap * 4);
  p += (size_t)eng.qpp * kCandCap * 8;
  float* dense = reinterpret_cast<float*>(p);
  const int64_t dense_floats = (int64_t)((ws + ws_bytes - p) / sizeof(float));
  const int qpp = eng.qpp;
  for (int q0 = 0; q0 < nq; q0 += qpp) {
    const int nqp = std::min(qpp, nq - q0);
    float* ts = top_scores + (size_t)q0 * k;
    int32_t* ti = top_ids + (size_t)q0 * k;
    if ((rc = engine_prepare(eng, Qcat, q0, nq, msw, st, who))) return rc;
    const int64_t dense_rows = dense_floats / qpp;
    const bool use_filter = n >= kFilterMinN && dense_rows >= std::min<int64_t>(n, eng.dense_rows_pref);
    const int* guard = nullptr;
    if (use_filter) {
      // The rows are spread over the whole index: the first ones say nothing about the others where an index is stored by topic
      // or time (1,000 clusters in turn, 8 queries, k = 10, 10^6 rows: 607 us from the first 4,096 rows, 84 when shuffled).
      const int64_t m = pilot_rows(n, k, dense_rows);
      if ((rc = engine_run(eng, q0, nqp, m, idx, qjl, gamma, norms, dense, m, nullptr, nullptr, msw, st, who, n / m))) return rc;
      TQ_CHECK_CUDA(mscan::select_topk(dense, nullptr, nullptr, (int)m, (int)m, 0, nqp, k, 0, nullptr, nullptr, tau, nullptr, nullptr, count, overflow, st), who);
      mscan::Filter f{tau, count, cand_s, cand_i, kCandCap};
      if ((rc = engine_run(eng, q0, nqp, n, idx, qjl, gamma, norms, nullptr, 0, &f, nullptr, msw, st, who))) return rc;
      TQ_CHECK_CUDA(mscan::select_topk(cand_s, cand_i, count, kCandCap, 0, 0, nqp, k, 0, ts, ti, nullptr, overflow, nullptr, nullptr, nullptr, st), who);
      guard = overflow;
    }
    if ((rc = topk_dense(eng, q0, nqp, n, idx, qjl, gamma, norms, k, ts, ti, dense, dense_floats, guard, msw, st, who))) return rc;
  }
  return TQ_OK;
}

extern "C" int tq_topk(const tq_plan* plan, const void* Q, int q_dtype, int nq, int64_t ldq, int64_t n,
                       const uint8_t* idx, const uint8_t* qjl, const float* gamma, const float* norms, int k,
                       float* top_scores, int32_t* top_ids, void* workspace, size_t workspace_bytes, void* stream) {
  const char* who = "tq_topk";
  TQ_RANGE(who);
  int rc = check_plan(plan, who);
  if (rc) return rc;
  TQ_REQUIRE(n >= 0 && nq >= 0, TQ_ERR_INVALID_ARG, "%s: negative size", who);
  if (nq == 0) return TQ_OK;
  TQ_REQUIRE(n <= 0x7fffffffLL, TQ_ERR_UNSUPPORTED, "%s: ids are int32, n too large", who);
  TQ_REQUIRE(k >= 1 && k <= TQ_MAX_K && k <= n, TQ_ERR_UNSUPPORTED, "%s: k=%d outside 1..min(n, %d)", who, k, TQ_MAX_K);
  if ((rc = check_rows(who, "Q", Q, q_dtype, nq, ldq, plan->d))) return rc;
  if ((rc = check_codes(plan, who, idx, qjl, gamma))) return rc;
  TQ_REQUIRE(top_scores != nullptr && top_ids != nullptr, TQ_ERR_INVALID_ARG, "%s: output is NULL", who);
  const size_t qb = qcat_bytes(plan, nq);
  const size_t need = plan->ms.ok ? ms_topk_fixed(plan, nq) + (size_t)pick_engine(plan, nq).qpp * kDenseRowsMin * sizeof(float)
                                  : qb + align_up((size_t)nq * std::min<int64_t>(n, kTopkBlockMin) * sizeof(float), 256);
  TQ_REQUIRE(workspace != nullptr && workspace_bytes >= need, TQ_ERR_WORKSPACE, "%s: workspace of %zu bytes, %zu needed",
             who, workspace_bytes, need);
  TQ_REQUIRE(aligned(workspace, 256), TQ_ERR_ALIGNMENT, "%s: workspace is not 256-byte aligned", who);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  float* Qcat = static_cast<float*>(workspace);
  if (plan->ms.ok) {
    TQ_CHECK_CUDA(prepare_queries(plan, Q, q_dtype, nq, ldq, Qcat, st), who);
    return topk_ms(plan, Qcat, nq, n, idx, qjl, gamma, norms, k, top_scores, top_ids, static_cast<char*>(workspace) + qb,
                   workspace_bytes - qb, st, who);
  }
  float* blockbuf = reinterpret_cast<float*>(static_cast<char*>(workspace) + qb);
  int64_t block = (int64_t)((workspace_bytes - qb) / ((size_t)nq * sizeof(float)));
  block = std::min(block, n);
  if (block < n) block = block / 256 * 256;
  TQ_CHECK_CUDA(prepare_queries(plan, Q, q_dtype, nq, ldq, Qcat, st), who);
  for (int64_t v0 = 0; v0 < n; v0 += block) {
    const int64_t cn = std::min(block, n - v0);
    TQ_CHECK_CUDA(score_block(plan, Qcat, nq, v0, cn, idx, qjl, gamma, norms, blockbuf, block, st), who);
    scan::topk_merge_kernel<<<nq, 256, 0, st>>>(blockbuf, block, v0, cn, k, v0 == 0 ? 1 : 0, top_scores, top_ids);
    count_launches(1);
    TQ_CHECK_CUDA(cudaGetLastError(), who);
  }
  return TQ_OK;
}

#ifdef TQ_DEBUG
// Hook for the tests of the debug build: the screening pass's lower bound of every pair's estimate into low [nq, n], and per query the
// error constant and the scale (screen::QueryTerms) into terms [nq, 2].  Queries fp32, rows of d; nq <= 256.
extern "C" int tq_debug_screen_bounds(const tq_plan* plan, const float* Q, int nq, int64_t n, const uint8_t* idx, const uint8_t* qjl,
                                      const float* gamma, const float* norms, float* low, float* terms, void* workspace,
                                      size_t workspace_bytes, void* stream) {
  const char* who = "tq_debug_screen_bounds";
  int rc = check_plan(plan, who);
  if (rc) return rc;
  TQ_REQUIRE(nq > 0 && nq <= screen::kQueries && n > 0 && plan->ms.ok && tscan::available(plan), TQ_ERR_INVALID_ARG, "%s: sizes", who);
  const size_t qb = qcat_bytes(plan, nq);
  TQ_REQUIRE(workspace != nullptr && aligned(workspace, 256) && workspace_bytes >= qb + screen::workspace_bytes(plan), TQ_ERR_WORKSPACE,
             "%s: workspace", who);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  float* Qcat = static_cast<float*>(workspace);
  void* operand = static_cast<char*>(workspace) + qb;
  TQ_CHECK_CUDA(prepare_queries(plan, Q, TQ_F32, nq, plan->d, Qcat, st), who);
  if ((rc = screen::prepare(plan, Qcat, nq, operand, st, who))) return rc;
  if ((rc = screen::run(plan, nq, n, idx, qjl, gamma, norms, low, n, nullptr, nullptr, nullptr, nullptr, 0, operand, st, who, 1))) return rc;
  TQ_CHECK_CUDA(cudaMemcpyAsync(terms, screen::query_terms(plan, operand), (size_t)nq * sizeof(screen::QueryTerms), cudaMemcpyDeviceToDevice, st), who);
  return TQ_OK;
}
#endif

template <int BITS>
static cudaError_t launch_wsum_partial(const tq_plan* plan, const attend::WsumArgs& a, dim3 grid, cudaStream_t st) {
  if (plan->mode == TQ_PROD) attend::wsum_partial_kernel<BITS, true><<<grid, 128, 0, st>>>(a);
  else attend::wsum_partial_kernel<BITS, false><<<grid, 128, 0, st>>>(a);
  count_launches(1);
  return cudaGetLastError();
}

extern "C" int tq_wsum(const tq_plan* plan, const float* W, int nw, int64_t ldw, int64_t n, const uint8_t* idx,
                       const uint8_t* qjl, const float* gamma, const float* norms, float* out, int64_t ldo,
                       void* workspace, size_t workspace_bytes, void* stream) {
  const char* who = "tq_wsum";
  TQ_RANGE(who);
  int rc = check_plan(plan, who);
  if (rc) return rc;
  TQ_REQUIRE(n >= 0 && nw >= 0, TQ_ERR_INVALID_ARG, "%s: negative size", who);
  if (nw == 0) return TQ_OK;
  TQ_REQUIRE(out != nullptr && ldo >= plan->d, TQ_ERR_INVALID_ARG, "%s: out is NULL or ldo < d", who);
  TQ_REQUIRE(aligned(out, 16), TQ_ERR_ALIGNMENT, "%s: out is not 16-byte aligned", who);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (n == 0) {
    TQ_CHECK_CUDA(cudaMemset2DAsync(out, (size_t)ldo * sizeof(float), 0, (size_t)plan->d * sizeof(float), nw, st), who);
    return TQ_OK;
  }
  TQ_REQUIRE(W != nullptr && ldw >= n, TQ_ERR_INVALID_ARG, "%s: W is NULL or ldw < n", who);
  if ((rc = check_codes(plan, who, idx, qjl, gamma))) return rc;
  const size_t need = tq_workspace_bytes(plan, TQ_OP_WSUM, n, nw, 0);
  TQ_REQUIRE(workspace != nullptr && workspace_bytes >= need, TQ_ERR_WORKSPACE, "%s: workspace of %zu bytes, %zu needed",
             who, workspace_bytes, need);
  TQ_REQUIRE(aligned(workspace, 16), TQ_ERR_ALIGNMENT, "%s: workspace is not 16-byte aligned", who);
  const int ncols = plan->ncat * plan->dpad;
  float* oprime = static_cast<float*>(workspace);
  float* partial = reinterpret_cast<float*>(static_cast<char*>(workspace) + align_up((size_t)nw * ncols * sizeof(float), 256));
  const int nchunks = (int)((n + attend::WS_TOK - 1) / attend::WS_TOK);
  for (int w0 = 0; w0 < nw; w0 += attend::WS_NW) {
    attend::WsumArgs a;
    a.W = W + (int64_t)w0 * ldw;
    a.ldw = ldw;
    a.nw = std::min(attend::WS_NW, nw - w0);
    a.n = n;
    a.idx = idx;
    a.idx_rb = plan->idx_row_bytes;
    a.qjl = qjl;
    a.qjl_rb = plan->qjl_row_bytes;
    a.gamma = gamma;
    a.norms = norms;
    a.cb = plan->cb;
    a.d = plan->d;
    a.dpad = plan->dpad;
    a.ncols = ncols;
    a.coef = plan->coef;
    a.nibble = plan->layout == TQ_LAYOUT_NIBBLE;
    a.partial = partial;
    const dim3 grid((unsigned)nchunks, (unsigned)((plan->d + 127) / 128));
    // columns the partial kernel never writes (pad coordinates) must read as zero
    TQ_CHECK_CUDA(cudaMemsetAsync(partial, 0, (size_t)nchunks * a.nw * ncols * sizeof(float), st), who);
    cudaError_t e;
    switch (plan->mse_bits) {
      case 0: e = launch_wsum_partial<0>(plan, a, grid, st); break;
      case 1: e = launch_wsum_partial<1>(plan, a, grid, st); break;
      case 2: e = launch_wsum_partial<2>(plan, a, grid, st); break;
      case 3: e = launch_wsum_partial<3>(plan, a, grid, st); break;
      default: e = launch_wsum_partial<4>(plan, a, grid, st); break;
    }
    TQ_CHECK_CUDA(e, who);
    attend::wsum_reduce_kernel<<<(unsigned)((a.nw * ncols + 255) / 256), 256, 0, st>>>(partial, nchunks, a.nw, ncols,
                                                                                        oprime + (size_t)w0 * ncols);
    count_launches(1);
    TQ_CHECK_CUDA(cudaGetLastError(), who);
  }
  // out = o' [Pi ; S]
  simt::RowsF32 A{oprime, ncols, nw, ncols};
  simt::RowsF32 B{plan->dBackT, ncols, plan->d, ncols};
  simt::EpStore ep{out, ldo, nullptr, nullptr};
  TQ_CHECK_CUDA(simt::launch_gemm(A, B, ep, (int64_t)nw, (int64_t)plan->d, ncols, st), who);
  return TQ_OK;
}

extern "C" int tq_select_topk(const float* cand_scores, const int32_t* cand_ids, int nq, int64_t m, int64_t ld, int k,
                              float* top_scores, int32_t* top_ids, void* stream) {
  const char* who = "tq_select_topk";
  TQ_RANGE(who);
  TQ_REQUIRE(nq >= 0 && m >= 0, TQ_ERR_INVALID_ARG, "%s: negative size", who);
  TQ_REQUIRE(k >= 1 && k <= TQ_MAX_K, TQ_ERR_UNSUPPORTED, "%s: k=%d outside 1..%d", who, k, TQ_MAX_K);
  TQ_REQUIRE(m <= 0x7fffffffLL && ld <= 0x7fffffffLL, TQ_ERR_UNSUPPORTED, "%s: m / ld too large", who);
  if (nq == 0) return TQ_OK;
  TQ_REQUIRE(top_scores != nullptr && top_ids != nullptr, TQ_ERR_INVALID_ARG, "%s: output is NULL", who);
  TQ_REQUIRE(m == 0 || (cand_scores != nullptr && cand_ids != nullptr && ld >= m), TQ_ERR_INVALID_ARG,
             "%s: candidates are NULL or ld < m", who);
  TQ_CHECK_CUDA(mscan::select_pairs(cand_scores, cand_ids, (int)ld, (int)m, nq, k, top_scores, top_ids,
                                    static_cast<cudaStream_t>(stream)), who);
  return TQ_OK;
}

extern "C" int tq_softmax(const float* s1, const float* s2, int nw, int64_t n, int64_t lds, float scale, float* W,
                          int64_t ldw, void* stream) {
  const char* who = "tq_softmax";
  TQ_RANGE(who);
  TQ_REQUIRE(nw >= 0 && n >= 0, TQ_ERR_INVALID_ARG, "%s: negative size", who);
  if (nw == 0 || n == 0) return TQ_OK;
  TQ_REQUIRE(s1 != nullptr && W != nullptr, TQ_ERR_INVALID_ARG, "%s: s1 / W is NULL", who);
  TQ_REQUIRE(lds >= n && ldw >= n, TQ_ERR_INVALID_ARG, "%s: row stride smaller than n", who);
  attend::softmax_rows_kernel<<<nw, 1024, 0, static_cast<cudaStream_t>(stream)>>>(s1, s2, lds, n, scale, W, ldw);
  count_launches(1);
  TQ_CHECK_CUDA(cudaGetLastError(), who);
  return TQ_OK;
}

// ======================================================================================
// tq_score_static: tq_score for callers that cannot allocate.  The rotated-query workspace is
// this file-scope device array instead of a caller buffer.  In host code the array's name is
// only a handle for the runtime, not a device address, so the address is looked up once per
// device with cudaGetSymbolAddress and that pointer is what the kernels get.
namespace {

static __device__ __align__(256) unsigned char g_static_scratch[TQ_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
void* g_static_ptr[kMaxDevices] = {};   // device address of g_static_scratch, per device ordinal

// Device address of the static scratch on the current device (looked up on first use).
int static_scratch(const char* who, int device, void** out) {
  TQ_REQUIRE(device >= 0 && device < kMaxDevices, TQ_ERR_UNSUPPORTED, "%s: device ordinal %d not supported", who, device);
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (g_static_ptr[device] == nullptr) {
    void* p = nullptr;
    TQ_CHECK_CUDA(cudaGetSymbolAddress(&p, g_static_scratch), who);
    TQ_REQUIRE(p != nullptr && aligned(p, 256), TQ_ERR_CUDA, "%s: static scratch has no usable device address", who);
    g_static_ptr[device] = p;
  }
  *out = g_static_ptr[device];
  return TQ_OK;
}

}  // namespace

// Largest nq tq_score_static accepts for this plan (0 if even one query does not fit).
extern "C" int tq_score_static_max_queries(const tq_plan* plan) {
  if (!plan) return 0;
  int lo = 0, hi = 1 << 16;
  while (lo < hi) {   // the need grows with nq
    const int mid = lo + (hi - lo + 1) / 2;
    const size_t qb = qcat_bytes(plan, mid);
    ScanEngine e{};
    const bool ok = qb <= (size_t)TQ_STATIC_SCRATCH_BYTES &&
                    (!plan->ms.ok || engine_that_fits(plan, mid, (size_t)TQ_STATIC_SCRATCH_BYTES - qb, &e));
    if (ok) lo = mid; else hi = mid - 1;
  }
  return lo;
}

extern "C" int tq_score_static(const tq_plan* plan, const void* Q, int q_dtype, int nq, int64_t ldq, int64_t n,
                               const uint8_t* idx, const uint8_t* qjl, const float* gamma, const float* norms,
                               float* scores, int64_t lds, void* stream) {
  const char* who = "tq_score_static";
  TQ_RANGE(who);
  int rc = check_plan(plan, who);   // also makes sure the plan's device is the current one
  if (rc) return rc;
  TQ_REQUIRE(n >= 0 && nq >= 0, TQ_ERR_INVALID_ARG, "%s: negative size", who);
  if (n == 0 || nq == 0) return TQ_OK;
  if ((rc = check_score_args(plan, who, Q, q_dtype, nq, ldq, n, idx, qjl, gamma, scores, lds))) return rc;
  const size_t qb = qcat_bytes(plan, nq);
  ScanEngine eng{};
  const bool fits = qb <= (size_t)TQ_STATIC_SCRATCH_BYTES &&
                    (!plan->ms.ok || engine_that_fits(plan, nq, (size_t)TQ_STATIC_SCRATCH_BYTES - qb, &eng));
  TQ_REQUIRE(fits, TQ_ERR_WORKSPACE,
             "%s: %d queries at d=%d need more scratch than the built-in array holds (%u bytes; at most %d queries "
             "for this plan); use tq_score with a caller workspace or fewer queries per call",
             who, nq, plan->d, (unsigned)TQ_STATIC_SCRATCH_BYTES, tq_score_static_max_queries(plan));
  void* ws = nullptr;
  if ((rc = static_scratch(who, plan->device, &ws))) return rc;
  // Every byte the kernels read from the array (rotated queries, then the scan engine's constants and operand)
  // is written by this call before it is read, so the previous call's leftovers never show.
  return score_on_workspace(plan, &eng, Q, q_dtype, nq, ldq, n, idx, qjl, gamma, norms, scores, lds, ws,
                            static_cast<cudaStream_t>(stream), who);
}
