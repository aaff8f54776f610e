// Interface of the many-query packed-code scan on tcgen05 (tq_scan_tc.cu) towards the API layer.
#pragma once

#include "tq_internal.h"
#include "tq_scan_mma.h"
#include "tq_screen_tc.h"

namespace tq {
namespace tscan {

constexpr int kQueriesPerPass = 32;    // 96 MMA columns = 32 queries x 3 radix-256 digits
constexpr int kPassesPerGroup = 8;     // B operands are built for up to 8 passes (256 queries) at a time

// Queries one pass over the codes serves when a call has nq of them: 32, or 64 (the wide kernel) beyond 32 queries.
int queries_per_pass(int nq);

// Whether the plan can use this path (same conditions as the bit-plane scan, plus shared-memory room).
bool available(const tq_plan* plan);

// Bytes of workspace for one group of passes: per-query constants + both B matrices.
size_t workspace_bytes(const tq_plan* plan);

// Builds constants and B matrices for queries [0, nqg) of a group (nqg <= 256), rotated queries in Qcat.
int prepare_group(const tq_plan* plan, const float* Qcat, int nqg, void* workspace, cudaStream_t st, const char* who);

// One pass of up to 32 queries (pass index `pass` inside the prepared group), or of 33 to 64 queries (the queries of
// passes `pass` and `pass + 1`, `pass` even), over vectors [0, n): dense estimates into scores[nqp, lds] or the pairs
// admitted by the filter.  run_if and step as in mscan::run.  More queries, up to the end of the group: several passes of 64 in one
// launch, run_if[i] the switch of the i-th.
int run_pass(const tq_plan* plan, int pass, int nqp, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma,
             const float* norms, float* scores, int64_t lds, const mscan::Filter* filter, const int* run_if,
             const void* workspace, cudaStream_t st, const char* who, int64_t step = 1);

// The candidates (lower bound, row of n; listed with thresholds tau) of nqp queries of a prepared group whose upper bound reaches kth[q],
// scored exactly -- the bits of run_pass -- into out_s / out_i [nqp, screen::kSurvivors] (NaN estimates as empty slots), their numbers added to
// out_count (zero before).
// overflow[q / per_flag] is set to 1 where more are left than fit, or where the list is longer than cap or has fewer than k entries.
int rescore(const tq_plan* plan, int nqp, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma, const float* norms,
            const void* workspace, const screen::QueryTerms* terms, const float* tau, const float* kth, const int* count,
            const float* cand_s, const int* cand_i, int cap, int k, float* out_s, int* out_i, int* out_count, int* overflow, int per_flag,
            cudaStream_t st, const char* who);

}  // namespace tscan
}  // namespace tq
