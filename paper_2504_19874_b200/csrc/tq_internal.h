// Internal declarations shared by the translation units of libtq (not part of the ABI).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <nvtx3/nvToolsExt.h>

#include <atomic>
#include <cstdarg>
#include <cstdint>
#include <cstdio>

#include "tq.h"

namespace tq {

void set_error(const char* fmt, ...);
void count_launches(int k);   // kernels enqueued by this library (diagnostic counter)
int lloyd_max(int d, int bits, double* c_out);

// Every API call that enqueues device work opens an NVTX range with its own name (visible in Nsight Systems /
// Compute timelines; a no-op without a profiler attached) and, when the environment variable TQ_LOG is set to a
// non-empty value other than 0, writes one line to stderr.
bool log_enabled();
struct CallRange {
  explicit CallRange(const char* name) {
    nvtxRangePushA(name);
    if (log_enabled()) std::fprintf(stderr, "[tq] %s\n", name);
  }
  ~CallRange() { nvtxRangePop(); }
  CallRange(const CallRange&) = delete;
  CallRange& operator=(const CallRange&) = delete;
};
#define TQ_RANGE(name) tq::CallRange tq_call_range_(name)

inline int round_up(int v, int m) { return (v + m - 1) / m * m; }
inline int64_t round_up64(int64_t v, int64_t m) { return (v + m - 1) / m * m; }

// Codebook and thresholds by value, so kernels get them through the parameter space.
struct Codebook {
  float c[16];   // centroids, ascending
  float t[15];   // boundaries fl32(0.5f * (c_i + c_{i+1}))
  int bits;      // b_m
};

// A d x d fp32 matrix split into two bf16 limbs (M = hi + lo + O(2^-17)), rows padded to dpad,
// with the TMA descriptors the tensor-core GEMM uses for it as the B operand.
// Device-side index checks of the TQ_DEBUG build: `if (TQ_DEVICE_CHECK(row < n, status)) out[row] = v;`.  In a release
// build the condition is not evaluated.  A failed check records TQ_ERR_BOUNDS in the plan's status word (reported by
// tq_plan_status) and the access is skipped.
#ifdef __CUDACC__
#ifdef TQ_DEBUG
__device__ __forceinline__ bool device_check_failed(int* status) {
  if (status != nullptr) atomicExch(status, TQ_ERR_BOUNDS);
  return false;
}
#define TQ_DEVICE_CHECK(cond, status) ((cond) ? true : ::tq::device_check_failed(status))
#else
#define TQ_DEVICE_CHECK(cond, status) (true)
#endif
#endif

#ifdef __CUDACC__
// Programmatic dependent launch: the grid may be scheduled while the kernel ahead of it in the stream drains.  Such a kernel
// calls wait_for_predecessor() in every thread before it touches global memory that another kernel writes or reads (constants
// of a plan may be read before); the call returns once the kernel ahead -- and with it, by the same rule, everything before --
// has completed.  allow_successor() lets the next such kernel be scheduled.
__device__ __forceinline__ void allow_successor() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... KArgs, typename... LArgs>
cudaError_t launch_dependent(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, LArgs... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
  return e != cudaSuccess ? e : cudaGetLastError();
}
#endif

// Lets a kernel be launched with as much dynamic shared memory as a block of the current device may have.  Once per device
// (`devices`: one word of bits per kernel), and always to the same value: the attribute is the kernel's, and a thread that set it
// to the size of its own call would make another thread's larger launch fail.
inline cudaError_t allow_largest_smem(const void* kern, std::atomic<unsigned long long>& devices) {
  int dev = 0, most = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 64 && ((devices.load(std::memory_order_relaxed) >> dev) & 1ull)) return cudaSuccess;
  cudaFuncAttributes own;
  if ((e = cudaFuncGetAttributes(&own, kern)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)own.sharedSizeBytes);
  if (e == cudaSuccess && dev < 64) devices.fetch_or(1ull << dev, std::memory_order_relaxed);
  return e;
}

constexpr int kBoxes = 4;
struct MatrixLimbs {
  __nv_bfloat16* hi;
  __nv_bfloat16* lo;
  alignas(64) CUtensorMap map_hi[kBoxes];   // box i: 32 (i + 1) rows, what one CTA of a tile loads
  alignas(64) CUtensorMap map_lo[kBoxes];
};

}  // namespace tq

// Per-(d, b, mode) device state: the "global parameters" of Algorithms 1 and 2.
struct tq_plan {
  int d;          // dimension
  int dpad;       // d rounded up to a multiple of 8 (virtual K extent of one code half)
  int bits;       // total bits b
  int mode;       // TQ_MSE / TQ_PROD
  int mse_bits;   // b_m
  int device;
  float coef;     // sqrt(pi/2) / d
  size_t idx_row_bytes, qjl_row_bytes;
  tq::Codebook cb;
  float* dPi;      // [d, d]            y = Pi x            (rows of Pi)
  float* dSp;      // [d, d]            S' = S Pi^T         (TQ_PROD)
  float* dRotCat;  // [ncat*dpad, dpad] rows: Pi (padded to dpad rows) then S, zeros in the padding (query preparation)
  float* dBackT;   // [d, ncat*dpad]    row j: [ Pi[:, j] | S[:, j] ]             (dequantisation)
  int ncat;        // 1 (mse) or 2 (prod): halves of the virtual K axis [ c[idx] | coef*gamma*z ]
  // tensor-core quantisation path (d >= 128)
  int tc_ok;       // 1 when the limbs / TMA descriptors below are built
  tq::MatrixLimbs pi_limbs;   // Pi
  tq::MatrixLimbs sp_limbs;   // S' (TQ_PROD)
  // bit-plane scan on the integer tensor path (d >= 128, antisymmetric codebook)
  struct {
    int ok;            // 1 when this plan can use it
    int R;             // ranges of 512 coordinates per row
    double alpha[8];   // odd Walsh coefficients of the codebook: index bits 0..3, then the 3-bit parities
    double amax;       // max |alpha|
    double csum;       // mean term minus the sum of alpha: constant part of sum_j q'_j c[idx_j]
  } ms;
  // nibble layout of the codes and the table-lookup scan (TQ_PROD with a 3-bit MSE stage)
  int layout;      // TQ_LAYOUT_*: arrangement of the idx / qjl rows this plan writes and reads
  struct {
    int ok;                            // 1 when this plan may be switched to TQ_LAYOUT_NIBBLE
    int nbi, nbq;                      // 64-byte blocks of an idx row / a qjl row
    uint32_t hi_a, hi_b, lo_a, lo_b;   // 16-bit centroid table t_i = 256 h_i + l_i as bytes: h of entries 0..3, 4..7, l alike
    double delta;                      // c_i ~ delta * t_i
  } nb;
  // tensor-core reconstruction (d >= 128)
  struct {
    int ok;
    int pitch;                         // row pitch of the limb matrices, elements
    __half *p_hi, *p_lo, *s_hi, *s_lo; // fp16 limbs of Pi^T and S^T, scaled by powers of two
    alignas(64) CUtensorMap map_p_hi, map_p_lo, map_s_hi, map_s_lo;
    uint32_t tab[4][4];                // bytes of the codebook's limbs: hi low / high byte, lo low / high byte, 16 entries each
    float gscale, oscale;              // weights of the accumulated sign term (per unit of gamma) and centroid term
  } dq;
  // one-launch quantiser for short vectors (d = 32, 64, 96)
  struct {
    int ok;
    float* spt;                        // [d, d] transpose of S' (TQ_PROD)
  } sq;
  int* d_status;   // device word: set to TQ_ERR_TIMEOUT by a kernel whose bounded wait ran out
};

#define TQ_CHECK_CUDA(call, what)                                                        \
  do {                                                                                   \
    cudaError_t e_ = (call);                                                             \
    if (e_ != cudaSuccess) {                                                             \
      tq::set_error("%s: %s", what, cudaGetErrorString(e_));                             \
      return TQ_ERR_CUDA;                                                                \
    }                                                                                    \
  } while (0)

#define TQ_REQUIRE(cond, code, ...)                                                      \
  do {                                                                                   \
    if (!(cond)) {                                                                       \
      tq::set_error(__VA_ARGS__);                                                        \
      return code;                                                                       \
    }                                                                                    \
  } while (0)
