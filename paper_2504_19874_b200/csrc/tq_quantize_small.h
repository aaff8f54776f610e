// Interface of the one-launch quantiser for short vectors (tq_quantize_small.cu) towards the API layer.
#pragma once

#include "tq_internal.h"

namespace tq {
namespace sq {

// The transpose of S' for d = 32, 64, 96 (plan->dSp already on the device).
cudaError_t plan_init(tq_plan* plan);
void plan_free(tq_plan* plan);

// Quant_mse / Quant_prod of n rows in one launch (plan->sq.ok; qjl, gamma unused for TQ_MSE).
int quantize(const tq_plan* plan, const void* X, int x_dtype, int64_t n, int64_t ldx, uint8_t* idx, uint8_t* qjl, float* gamma,
             float* norms, cudaStream_t st, const char* who);

}  // namespace sq
}  // namespace tq
