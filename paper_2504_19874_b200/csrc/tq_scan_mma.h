// Interface of the tensor-path packed-code scan (tq_scan_mma.cu) towards the API layer.
#pragma once

#include "tq_internal.h"

namespace tq {
namespace mscan {

// Decides whether the plan's codebook / dimension admit the bit-plane scan and fills plan->ms.
void plan_init(tq_plan* plan);

// Queries served by one pass over the codes when nq queries remain (2, 4 or 8).
int queries_per_pass(const tq_plan* plan, int nq);

// Bytes of workspace a pass of a call of nq queries needs: per-query constants + the B operand (query-side matrix).
size_t workspace_bytes(const tq_plan* plan, int nq);

struct Filter {          // top-k candidate collection for the queries of one pass
  const float* tau;      // [nqp] admission threshold per query (score >= tau is kept)
  int* count;            // [nqp] candidates appended so far (may exceed cap: the excess was dropped)
  float* cand_s;         // [nqp, cap]
  int* cand_i;           // [nqp, cap]  ids = row numbers
  int cap;
};

// Builds the per-query constants and the B operand of one pass (nqp <= queries_per_pass) from the
// rotated queries Qcat[nqp, ncat*dpad] into `workspace`.
int prepare(const tq_plan* plan, const float* Qcat, int nqp, void* workspace, cudaStream_t st, const char* who);

// One pass over vectors [0, n) with the operand prepared in `workspace`: dense estimates into
// scores[nqp, lds], or, with a filter, only the (score, row) pairs it admits.  When run_if is not null
// the kernel returns at once if *run_if == 0 (device-side switch, read at launch).  step > 1: vector i of the pass is row i step
// of the arrays (a sample of the database).
int run(const tq_plan* plan, int nqp, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma,
        const float* norms, float* scores, int64_t lds, const Filter* filter, const int* run_if, const void* workspace,
        cudaStream_t st, const char* who, int64_t step = 1);

// The k best (score desc, id asc) per query out of `count[q]` (clamped to cap) candidate pairs, or, when
// cand_i is nullptr, out of the dense row cand_s[q*cap .. +m) with ids id0 + position.  Optionally merges
// the previous best list (top_s/top_i, when merge != 0) and writes the k-th score to kth[q].
// With top_s == nullptr only kth[q] is written: a lower bound of the k-th score that at least k entries reach.
// overflow[q / per_flag] is set to 1 if the count of query q exceeded cap; run_if[q / per_flag] as above.  clear_count[0 .. nq) and the
// flags clear_flag[q / per_flag] are set to 0 (the counters of the filter pass that follows a pilot's selection).
cudaError_t select_topk(const float* cand_s, const int* cand_i, const int* count, int cap, int m, int id0, int nq, int k,
                        int merge, float* top_s, int* top_i, float* kth, int* overflow, const int* run_if, int* clear_count,
                        int* clear_flag, cudaStream_t st, int per_flag = 1 << 30);

// The k best of m candidate pairs per query (row stride ld); pairs with id < 0 are skipped.
cudaError_t select_pairs(const float* cand_s, const int* cand_i, int ld, int m, int nq, int k, float* top_s, int* top_i,
                         cudaStream_t st);

}  // namespace mscan
}  // namespace tq
