// Internal declarations shared by the translation units of the DDTS library (not part of the ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "rodimus_ddts.h"

namespace ddts {

// Device-visible words at the start of the caller's workspace.
struct WorkspaceHeader {
  int32_t status;        // rodimus_status recorded by kernels (0 = ok); only ever raised
  int32_t pad[63];
};
static_assert(sizeof(WorkspaceHeader) == 256, "workspace header is 256 bytes");

constexpr int kMaxSortedSeqs = 4096;  // varlen: sequences beyond this keep their given order

// The current device and its SM count (the count is asked for once per device).
cudaError_t current_device(int* dev, int* sms);

// Opt-in to more than 48 KiB of dynamic shared memory, once per kernel and device: `done` is a
// per-kernel bit mask over device ordinals (devices beyond 63 simply ask every time).
template <typename Kernel>
inline cudaError_t opt_in_shared_memory(Kernel kernel, int bytes, int dev, std::atomic<unsigned long long>& done) {
  const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
  if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_release);
  return e;
}

// Launch of a kernel that may start while the one before it on the stream still runs: it sets up, then
// calls wait_for_previous_kernel() before it touches what that one wrote.  The one before says with
// let_next_kernel_start() from when on that is allowed (once every CTA of it has said so or ended).
template <typename... P, typename... A>
inline cudaError_t launch_overlapped(void (*kernel)(P...), unsigned grid, int threads, int smem, cudaStream_t st, const A&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}
__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_kernel_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Limit, in clock cycles, that the tensor-core prefill kernels give each of their main-loop
// waits (see rodimus_ddts_test_set_wait_limit).
long long main_loop_wait_cycles();

// Launchers: all arguments validated by the caller; they return a cudaError_t.
cudaError_t launch_step(const rodimus_ddts_step_params& p, int* n_launches);
cudaError_t launch_plan(const rodimus_ddts_fwd_params& p, int* n_launches);
cudaError_t launch_fwd_simt(const rodimus_ddts_fwd_params& p, int* n_launches);
size_t fwd_simt_chunks_workspace_bytes(const rodimus_ddts_fwd_params& p);   // 0: not the parallel form
cudaError_t launch_fwd_tc(const rodimus_ddts_fwd_params& p, int* n_launches);
cudaError_t launch_fwd_pair(const rodimus_ddts_fwd_params& p, int* n_launches);
cudaError_t launch_bwd(const rodimus_ddts_bwd_params& p, size_t scratch_offset, int* n_launches);
bool bwd_supported(const rodimus_ddts_bwd_params& p);
size_t bwd_scratch_bytes(const rodimus_ddts_bwd_params& p);   // beyond the header and the order
cudaError_t launch_bwd_tc(const rodimus_ddts_bwd_params& p, size_t scratch_offset, int* n_launches);   // bf16
size_t bwd_tc_scratch_bytes(const rodimus_ddts_bwd_params& p);
cudaError_t launch_swska(const rodimus_swska_fwd_params& p, int* n_launches);
cudaError_t launch_swska_tc(const rodimus_swska_fwd_params& p, int* n_launches);   // bf16, tcgen05
bool swska_supported(const rodimus_swska_fwd_params& p);
cudaError_t launch_fwd_scan(const rodimus_ddts_fwd_params& p, int* n_launches);
// Workspace with which the prefill that forms operands first takes this request, in two launches or split along
// time in four; 0: it does not.
size_t fwd_scan_workspace_bytes(const rodimus_ddts_fwd_params& p);
size_t fwd_scan_split_workspace_bytes(const rodimus_ddts_fwd_params& p);
bool fwd_tc_supported(const rodimus_ddts_fwd_params& p);
bool fwd_pair_supported(const rodimus_ddts_fwd_params& p);
// Workspace a dense call needs if its sequences are to be split along time (0: no split).
size_t fwd_pair_split_workspace_bytes(const rodimus_ddts_fwd_params& p);

// The largest n in [0, count) with holds(n), -1 if there is none, where holds() is true up to some n and false
// from there on (otherwise some n of that range).  Block-wide.  Every round asks as many n as the block has
// threads, evenly spread, and counts the answers: one round for up to THREADS of them.  (Every n asked, and the
// largest taken by an atomic: fp32 prefill of 20000 sequences of 1 to 8 tokens 4.10 ms, 2.79 this way; of 64
// sequences 207 and 201 us.)
template <int THREADS, typename Holds>
__device__ __forceinline__ int last_that_holds(int count, Holds holds) {
  if (count > THREADS) {
    int first = 0, end = count, stride;
    do {
      stride = (end - first + THREADS - 1) / THREADS;
      const int at = first + (int)threadIdx.x * stride;
      const int yes = __syncthreads_count(at < end && holds(at));
      if (yes == 0) return -1;
      first += (yes - 1) * stride;
      end = min(end, first + stride);
    } while (stride > 1);
    return first;
  }
  return __syncthreads_count((int)threadIdx.x < count && holds((int)threadIdx.x)) - 1;
}

// ---------------------------------------------------------------------------------------------
// Element access for the two token dtypes.
// ---------------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ float to_f32(T v);
template <>
__device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename T>
__device__ __forceinline__ T from_f32(float v);
template <>
__device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// ---------------------------------------------------------------------------------------------
// Gate math in full fp32 precision (Eq. "alpha_def"): natural-log decay and natural-log input
// weight for one key channel.  Used where accuracy matters more than issue slots (decode, fp32
// prefill).  log_alpha = -softplus(x) * sigmoid(y) <= 0;  log_ahat = sigmoid(y) * log(g) for
// the paper's form, sigmoid(y) * log(1 - exp(-g)) = -sigmoid(y) * softplus(-x) for the other.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float softplus_f32(float x) {
  return x > 0.f ? x + log1pf(expf(-x)) : log1pf(expf(x));
}

__device__ __forceinline__ void gate_logs_f32(float x, float y, int ingate, float& log_alpha,
                                              float& log_ahat) {
  const float g = softplus_f32(x);
  const float tau = y >= 0.f ? 1.f / (1.f + expf(-y)) : expf(y) / (1.f + expf(y));
  log_alpha = -g * tau;
  if (ingate == RODIMUS_INGATE_POW_G) {
    // g > 0 for every finite x >= -87; log(g) -> x as x -> -inf
    log_ahat = tau * logf(g);
  } else {
    log_ahat = -tau * softplus_f32(-x);
  }
}

}  // namespace ddts
