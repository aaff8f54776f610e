// Interface of the one-launch quantiser for short vectors (tq_quantize_small.cu) towards the API layer.
#pragma once

#include "tq_internal.h"

namespace tq {
namespace sq {

// Limb images of Pi and S' for d = 32, 64, 96, 128 (plan->dPi, plan->dSp already on the device).
cudaError_t plan_init(tq_plan* plan);
void plan_free(tq_plan* plan);

// Whether a plan that both this and the tcgen05 path can serve (d = 128) goes through this one for n rows.
bool preferred(const tq_plan* plan, int x_dtype, int64_t n);

// Quant_mse / Quant_prod of n rows in one launch (plan->sq.ok; canonical layout; qjl, gamma unused for TQ_MSE).
int quantize(const tq_plan* plan, const void* X, int x_dtype, int64_t n, int64_t ldx, uint8_t* idx, uint8_t* qjl, float* gamma,
             float* norms, cudaStream_t st, const char* who);

}  // namespace sq
}  // namespace tq
