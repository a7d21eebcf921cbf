// Shared declarations of the pepsvmc CUDA library (kernels + host engine).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <string>

namespace pv {

// Batched contraction written as C[b] (scattered) = alpha * A[b] x B[b].
//   A(m,k) = A + b*bsA + m*sAm + k*sAk
//   B(k,n) = B + slot(b)*ssB + b*bsB + k*sBk + n*sBn,
//            slot(b) = (sel[b*sel_stride] < 0) ^ sel_xor when sel != nullptr, else 0
//   C index of (m,n): m = ((m1*cm2)+m2)*cm3+m3 -> m1*sCm1 + m2*sCm2 + m3*sCm3,
//                     n likewise with (cn2, cn3, sCn*).
//   alpha * (inv_scale ? 1/inv_scale[b] : 1).  accumulate: C += instead of C =.
struct GemmDesc {
  int M = 0, N = 0, K = 0, batch = 0;
  const float* A = nullptr;
  long long sAm = 0, sAk = 0, bsA = 0;
  const float* B = nullptr;
  long long sBk = 0, sBn = 0, bsB = 0, ssB = 0;
  const int8_t* sel = nullptr;
  long long sel_stride = 0;
  int sel_xor = 0;
  float* C = nullptr;
  long long bsC = 0;
  int cm2 = 1, cm3 = 1;
  long long sCm1 = 0, sCm2 = 0, sCm3 = 0;
  int cn2 = 1, cn3 = 1;
  long long sCn1 = 0, sCn2 = 0, sCn3 = 0;
  float alpha = 1.f;
  const double* inv_scale = nullptr;
  int accumulate = 0;
  long long wait_cycles = 0;  // clock budget of each device-side wait (0 = kDefaultWaitCycles)
};

// Default clock budget of a device-side wait (~2 s at 2 GHz).
constexpr long long kDefaultWaitCycles = 4000000000LL;

// Tile configurations of the FP32 contraction kernel (index into a fixed table).
int gemm_f32_num_configs();
const char* gemm_f32_config_name(int cfg);
cudaError_t gemm_f32(const GemmDesc& d, int cfg, cudaStream_t st);
int gemm_f32_pick(const GemmDesc& d);

// Same contraction on the tcgen05 tensor cores with FP32 accumulation in tensor memory.
// mode 2: operands rounded to BF16 (kind::f16); 3: split BF16, x = hi + lo, three MMAs
// per step; 4: operands rounded to TF32 (kind::tf32); 6: mode 3 with two shared-memory
// stages (bn 32 or 64).  Device waits are bounded; on
// expiry ST_TIMEOUT is set in *status.  bn: N tile (32, 64, 128, 256; 0 = smallest >= N).
cudaError_t gemm_tc(const GemmDesc& d, int mode, int bn, unsigned* status, cudaStream_t st);

// Batched Householder QR with diag(R) >= 0; writes the thin Q.
//   Y(i,j) = Y + b*bsY + i*yrs + j*ycs,   i < rows, j < cols, rows >= cols
//   Q(i,j) = Q + b*bsQ + i*qrs + j*qcs
cudaError_t qr_pos_batched(const float* Y, long long bsY, long long yrs, long long ycs,
                           float* Q, long long bsQ, long long qrs, long long qcs,
                           int rows, int cols, int batch, cudaStream_t st);

// Dry-run mode: every kernel wrapper returns at once without touching the device.
// The engine then runs its whole host-side orchestration (with bounds validation
// of every launch) on a machine without a GPU.
extern bool g_dry_run;

// Status word bits set by device code (checked by the host after a sync).
enum : unsigned {
  ST_ZEROPSI = 1u,
  ST_NONFINITE = 2u,
  ST_TIMEOUT = 4u,
};

// e, a runtime call's result, to be returned to the caller: as the runtime's last error it would be
// reported a second time, by the next check in this library or of the caller's.  An error that was
// pending before stays.
inline cudaError_t reported(cudaError_t e) {
  if (e != cudaSuccess && cudaPeekAtLastError() == e) cudaGetLastError();
  return e;
}

// The SMs of the current device (0.03 us of host time, so it is asked for at every launch that needs it).
inline cudaError_t sm_count(int* sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  return reported(e);
}

// Launch that may begin when the blocks of the kernel ahead of it on the stream have ended, before
// its end is complete (programmatic dependent launch).  A call is hundreds to thousands of
// dependent launches of a few us: launched one by one, a 4x4 measurement took 1.86 ms with
// plain launches and 1.18 ms with these, an 8x8 sweep of 16 chains 25.2 and 17.8 ms.  Every kernel launched
// this way calls after_previous() in all threads before it touches memory that another kernel may
// write or read, and before any return, so that its own end still implies the end of
// everything ahead of it, and reads such memory by plain, volatile or asynchronous loads: one that promises
// that the memory does not change during the kernel (__ldg, const __restrict__) may be moved ahead of
// the wait.  No kernel lets the next one start earlier: blocks of the next one
// then gathered on the few SMs that were free and took longer (a step of 128 chains of 8x8, D 8:
// 91 against 81 ms).  In a graph, whose launches follow each other without the host, the
// plain form is as fast or faster (80.1 against 80.8 ms), so a capture gets that.
inline bool plain_launches(cudaStream_t st) {
  cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
  // a capture elsewhere bars the legacy stream: the launch itself reports that
  return reported(cudaStreamIsCapturing(st, &s)) != cudaSuccess || s != cudaStreamCaptureStatusNone;
}
template <typename... Par, typename... Arg>
cudaError_t launch(bool plain, void (*kernel)(Par...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const Arg&... arg) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = plain ? 0 : 1;
  return reported(cudaLaunchKernelEx(&cfg, kernel, static_cast<Par>(arg)...));
}
template <typename... Par, typename... Arg>
cudaError_t launch_early(void (*kernel)(Par...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const Arg&... arg) {
  return launch(plain_launches(st), kernel, grid, block, smem, st, arg...);
}

// The same for a kernel with more than 48 KB of shared memory, its static variables included: it may be
// launched once its limit of dynamic shared memory is raised, which holds for the device that is
// current and until that device is reset.  The limit is set on the first launch on a device, and
// again when a launch is refused (a device that was reset); inside a capture, which a refused launch
// might spoil, always.  (Set at every launch it cost the smallest steps 7 %: 0.2 us, twice where
// `all` is, of 6.6.)  A refusal is reported and not kept.
constexpr size_t kCtaSmem = 227 * 1024;  // what a CTA of sm_103a may have, static and dynamic
struct SmemLimit {
  size_t bytes;  // the most that any launch of the kernel asks for: threads do not lower each other's limit
  bool all;      // the SM's whole shared memory rather than first-level cache, so that two CTAs fit an SM
  std::atomic<uint64_t> devices{0};  // bit of each device (modulo 64) it was set on
  template <typename... Par>
  cudaError_t set(void (*kernel)(Par...), uint64_t bit) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && all) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e == cudaSuccess) devices.fetch_or(bit, std::memory_order_relaxed);
    return reported(e);
  }
};
// early: whether the kernel calls after_previous().
template <typename... Par, typename... Arg>
cudaError_t launch_large(SmemLimit& limit, bool early, void (*kernel)(Par...), dim3 grid, dim3 block, size_t smem,
                         cudaStream_t st, const Arg&... arg) {
  int dev = 0;
  cudaError_t e = reported(cudaGetDevice(&dev));
  if (e != cudaSuccess) return e;
  const uint64_t bit = (uint64_t)1 << (dev & 63);
  const bool capture = plain_launches(st), plain = capture || !early;
  if (capture || !(limit.devices.load(std::memory_order_relaxed) & bit)) {
    e = limit.set(kernel, bit);
    return e == cudaSuccess ? launch(plain, kernel, grid, block, smem, st, arg...) : e;
  }
  e = launch(plain, kernel, grid, block, smem, st, arg...);
  if (e != cudaErrorInvalidValue) return e;
  e = limit.set(kernel, bit);
  return e == cudaSuccess ? launch(plain, kernel, grid, block, smem, st, arg...) : e;
}
#ifdef __CUDACC__
__device__ __forceinline__ void after_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
#endif

}  // namespace pv

#define PV_CUDA(x)                                                        \
  do {                                                                    \
    cudaError_t e_ = (x);                                                 \
    if (e_ != cudaSuccess) return e_;                                     \
  } while (0)
