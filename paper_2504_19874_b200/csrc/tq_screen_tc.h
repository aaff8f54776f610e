// Interface of the screening scan (tq_screen_tc.cu) towards the API layer.
#pragma once

#include "tq_internal.h"

namespace tq {
namespace screen {

constexpr int kQueries = 256;          // queries per pass over the codes
// Rows of a query that are scored again at most.  One costs 1.0 ns at d = 200 prod b = 3 and 1.4 at d = 1536 prod b = 4 (256 queries with
// as many each, 10^6 rows), so that 8,192 cost about what the exact passes do that stand in for them (6,000 equal rows at the top, a
// limit of 4,096: 3.4 and 5.1 ms; scored one by one 2.0 and 3.6).
constexpr int kSurvivors = 8192;
// Lower bounds of listed rows are formed by four operations whose results are no larger than |tau| and the row's own terms: half a
// place each, 2^-22 |tau| in all (the row's own terms are covered by its error constant).  Twice that is taken off.
constexpr float kThresholdSlack = 4.76837158e-7f;   // 2^-21

// K-blocks of 64 coordinates that a row takes.
int k_blocks(const tq_plan* plan);

// Bytes of workspace for one pass: the fp16 query operand and the per-query constants.
size_t workspace_bytes(const tq_plan* plan);

// Builds operand and constants of queries [0, nqp) (nqp <= kQueries) from the rotated queries Qcat.
int prepare(const tq_plan* plan, const float* Qcat, int nqp, void* workspace, cudaStream_t st, const char* who);

// Bounds of the estimates of vectors [0, n) (vector i is row i step of the arrays).
//   dense != nullptr: dense[q lds + i] = a lower bound of the estimate that the exact engines return for (query q, vector i)
//   else: the vectors whose upper bound reaches tau[q] are appended to query q's list as (lower bound, row); the upper bound is at most
//         the lower one + 2 rho E + 2 kThresholdSlack |tau[q]|
int run(const tq_plan* plan, int nqp, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma, const float* norms,
        float* dense, int64_t lds, const float* tau, int* count, float* cand_s, int* cand_i, int cap, const void* workspace,
        cudaStream_t st, const char* who, int64_t step);

// What the estimate of row (nu, gamma) may differ from its screened value by, per unit of the query's error constant; the row's
// values as the screening uses them.  A row that the bounds do not hold for (negative or non-finite norm or gamma, a norm near the
// ends of the range of fp32) has nu 0 and an infinite bound: it passes every threshold, unless a scalar of it is NaN.
struct RowTerms {
  float nu, rho, gamma;
};
#ifdef __CUDACC__
__device__ __forceinline__ RowTerms row_terms(float nu, float gamma) {
  const bool odd = !(nu >= 0.f && nu < 1e25f && (nu == 0.f || nu > 1e-20f) && gamma >= 0.f && gamma < 60000.f);
  RowTerms t;
  t.nu = odd ? 0.f : nu;
  t.gamma = odd ? 0.f : gamma;
  t.rho = odd ? __int_as_float(0x7f800000) : __fmaf_rn(nu, gamma, nu);
  return t;
}
#endif

// Per-query constants (device array in the workspace): error constant (scaled like the screened values) and the power of two
// that scales them back.  Two queries have no bounds and list no row: one of zeros, whose estimates all are zero, so that its result
// is the first k rows (of the first k + kZeroSpare, some of whose estimates may be NaN), and one with a NaN, whose estimates all are.
struct QueryTerms {
  float err, unscale;
};
constexpr float kZeroQuery = -1.f, kNanQuery = -2.f;   // their error constants
constexpr int kZeroSpare = 128;
const QueryTerms* query_terms(const tq_plan* plan, const void* workspace);

}  // namespace screen
}  // namespace tq
