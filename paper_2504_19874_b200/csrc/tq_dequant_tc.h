// Interface of the tensor-core reconstruction path (tq_dequant_tc.cu) towards the API layer.
#pragma once

#include "tq_internal.h"

namespace tq {
namespace dq {

// Builds the fp16 limbs of Pi^T and S^T and their TMA descriptors (d >= 128; Pi and S host matrices, S NULL for TQ_MSE).
cudaError_t plan_init(tq_plan* plan, const float* Pi, const float* S);
void plan_free(tq_plan* plan);

// DeQuant_mse / DeQuant_prod of n rows (plan->dq.ok).
int dequantize(const tq_plan* plan, int64_t n, const uint8_t* idx, const uint8_t* qjl, const float* gamma, const float* norms,
               float* Xhat, int64_t ldxh, cudaStream_t st, const char* who);

}  // namespace dq
}  // namespace tq
