// A CUDA runtime of the host alone, for tests of the launching code on a machine without a GPU:
// linked with the library's objects in the place of libcudart.  Kernels do not run; every launch
// is recorded under its kernel's name.  A launch with more than 48 KB of shared memory is refused
// unless that kernel's limit was raised on the current device since that device was last reset,
// and errors stay pending until cudaGetLastError, as the runtime documents.
#include <cuda_runtime_api.h>
#include <stdint.h>
#include <string.h>

#include <map>
#include <string>
#include <utility>
#include <vector>

#include "fused.cuh"
#include "fused_f32.cuh"
#include "kernels.cuh"
#include "stages.cuh"

namespace {

struct Launch {
  std::string name;
  dim3 grid, block;
  size_t smem;
  bool early;
};
std::map<const void*, std::string> names;
std::map<std::pair<int, const void*>, size_t> limits;  // dynamic shared memory, by device and kernel
std::vector<Launch> launches;
cudaError_t pending = cudaSuccess;
int device = 0, refuse_limits = 0, limits_set = 0;
bool capture_elsewhere = false;

cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) pending = e;
  return e;
}
cudaError_t launch(const void* f, dim3 g, dim3 b, size_t smem, bool early) {
  if (capture_elsewhere) return set(cudaErrorStreamCaptureImplicit);
  // static shared memory of the kernels that have both kinds (at least)
  size_t fixed = 0;
  for (const auto& k : {std::make_pair("13qr_pos_kernel", 544), std::make_pair("gemm_tc_kernel", 272)})
    if (names[f].find(k.first) != std::string::npos) fixed = k.second;
  const auto l = limits.find({device, f});
  if (l == limits.end() ? smem + fixed > 48 * 1024 : smem > l->second) return set(cudaErrorInvalidValue);
  if (!g.x || g.x > 0x7fffffffu || g.y > 65535u || g.z > 65535u) return set(cudaErrorInvalidConfiguration);
  launches.push_back(Launch{names[f], g, b, smem, early});
  return cudaSuccess;
}
struct {
  dim3 g, b;
  size_t smem;
  void* st;
} config;

}  // namespace

extern "C" {

void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names[f] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* st) {
  config = {g, b, smem, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  *g = config.g;
  *b = config.b;
  *smem = config.smem;
  memcpy(st, &config.st, sizeof(void*));
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t smem, cudaStream_t) {
  return launch((const void*)k, g, b, smem, false);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  bool early = false;
  for (unsigned i = 0; i < c->numAttrs; ++i) early |= c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization;
  return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, early);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  ++limits_set;
  if (refuse_limits > 0) {
    --refuse_limits;
    return set(cudaErrorNotReady);
  }
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    if (v < 0 || v > 227 * 1024) return set(cudaErrorInvalidValue);
    limits[{device, f}] = (size_t)v;
  }
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  if (capture_elsewhere) return set(cudaErrorStreamCaptureImplicit);
  *s = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = pending;
  pending = cudaSuccess;
  return e;
}
cudaError_t cudaPeekAtLastError() { return pending; }
cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int d) {
  *v = a == cudaDevAttrMultiProcessorCount ? (d ? 76 : 152) : 0;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
  *p = const_cast<void*>(s);
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "error of the fake runtime"; }

// What the tests here do not reach.
#define UNUSED(name, ...) \
  cudaError_t name(__VA_ARGS__) { return set(cudaErrorNotSupported); }
UNUSED(cudaDeviceSynchronize)
UNUSED(cudaEventCreate, cudaEvent_t*)
UNUSED(cudaEventCreateWithFlags, cudaEvent_t*, unsigned)
UNUSED(cudaEventDestroy, cudaEvent_t)
UNUSED(cudaEventElapsedTime, float*, cudaEvent_t, cudaEvent_t)
UNUSED(cudaEventRecord, cudaEvent_t, cudaStream_t)
UNUSED(cudaEventSynchronize, cudaEvent_t)
UNUSED(cudaFree, void*)
UNUSED(cudaGraphDestroy, cudaGraph_t)
UNUSED(cudaGraphExecDestroy, cudaGraphExec_t)
UNUSED(cudaGraphInstantiate, cudaGraphExec_t*, cudaGraph_t, unsigned long long)
UNUSED(cudaGraphLaunch, cudaGraphExec_t, cudaStream_t)
UNUSED(cudaMalloc, void**, size_t)
UNUSED(cudaMemcpyAsync, void*, const void*, size_t, cudaMemcpyKind, cudaStream_t)
UNUSED(cudaMemsetAsync, void*, int, size_t, cudaStream_t)
UNUSED(cudaStreamBeginCapture, cudaStream_t, cudaStreamCaptureMode)
UNUSED(cudaStreamCreateWithFlags, cudaStream_t*, unsigned)
UNUSED(cudaStreamDestroy, cudaStream_t)
UNUSED(cudaStreamEndCapture, cudaStream_t, cudaGraph_t*)
UNUSED(cudaStreamSynchronize, cudaStream_t)
UNUSED(cudaStreamWaitEvent, cudaStream_t, cudaEvent_t, unsigned)

// ---- what the tests set and read
void fake_device(int d) { device = d; }
void fake_reset_device() {
  for (auto it = limits.begin(); it != limits.end();) it = it->first.first == device ? limits.erase(it) : ++it;
}
void fake_refuse_limits(int n) { refuse_limits = n; }
void fake_capture_elsewhere(int on) { capture_elsewhere = on; }
void fake_pending(int e) { pending = (cudaError_t)e; }
int fake_limits_set() { return limits_set; }
int fake_launches() { return (int)launches.size(); }
void fake_clear() { launches.clear(); }
const char* fake_name(int i) { return launches[i].name.c_str(); }
long long fake_grid(int i) { return (long long)launches[i].grid.x * launches[i].grid.y * launches[i].grid.z; }
int fake_threads(int i) { return (int)(launches[i].block.x * launches[i].block.y * launches[i].block.z); }
long long fake_smem(int i) { return (long long)launches[i].smem; }

// ---- the library's launchers by plain arguments; d: bonds and legs in the order of the C ABI
int host_env3_f32_fits(int n, const int* d) {
  pv::Env3Fused f;
  f.batch = n;
  f.cT = d[0]; f.cB = d[1]; f.cT2 = d[2]; f.cB2 = d[3]; f.Dl = d[4]; f.Dr = d[5]; f.Du = d[6]; f.Dd = d[7];
  f.sTa = (long long)f.Du * f.cT2; f.sTu = f.cT2; f.sTa2 = 1;
  return pv::env3_f32_fits(f);
}
static int env4_f32_question(int n, const int* d, int variants, bool takes) {
  pv::Env4Fused f;
  f.batch = n;
  f.cT = d[0]; f.cB = d[1]; f.cT2 = d[2]; f.cB2 = d[3];
  f.D1l = d[4]; f.D1r = d[5]; f.Du1 = d[6]; f.Dd1 = d[7]; f.D2l = d[8]; f.D2r = d[9]; f.Dd2 = d[10];
  f.sEl2 = f.cB; f.sEl1 = (long long)f.D2l * f.cB;
  f.sTa = (long long)f.Du1 * f.cT2; f.sTu = f.cT2; f.sTa2 = 1;
  pv::Env4Outs o;
  for (int i = 0; i < variants; ++i) o.p[i] = (float*)16;
  return takes ? pv::env4_f32_takes(f, o, n) : pv::env4_f32_fits(f, o);
}
int host_env4_f32_fits(int n, const int* d, int variants) { return env4_f32_question(n, d, variants, false); }
int host_env4_f32_takes(int n, const int* d, int variants) { return env4_f32_question(n, d, variants, true); }

static float* at(int k) { return (float*)((uintptr_t)k << 44); }  // far apart and aligned
static pv::Env3Fused env3(int n, int chi, int D) {
  pv::Env3Fused f;
  f.batch = n;
  f.cT = f.cB = f.cT2 = f.cB2 = chi;
  f.Dl = f.Dr = f.Du = f.Dd = D;
  f.E = at(1); f.T = at(2); f.A = at(3); f.B = at(5); f.out = at(6);
  f.bsE = f.bsT = f.bsB = f.bsO = (long long)chi * D * chi;
  f.sEa = f.sTa = f.sBb = f.sOa2 = (long long)D * chi;
  f.sEl = f.sTu = f.sBd = f.sOr = chi;
  f.sEb = f.sTa2 = f.sBb2 = f.sOb2 = 1;
  f.ssA = (long long)D * D * D * D;
  f.sAl = (long long)D * D * D; f.sAu = (long long)D * D; f.sAr = D; f.sAd = 1;
  return f;
}
static pv::Env4Fused env4(int n, int chi, int D, bool bmajor) {
  pv::Env4Fused f;
  f.batch = n;
  f.cT = f.cB = f.cT2 = f.cB2 = chi;
  f.D1l = f.D1r = f.Du1 = f.Dd1 = f.D2l = f.D2r = f.Dd2 = D;
  f.E = at(1); f.T = at(2); f.A1 = at(3); f.A2 = at(4); f.B = at(5); f.out = at(6);
  f.bsE = f.bsO = (long long)chi * D * D * chi;
  f.bsT = f.bsB = (long long)chi * D * chi;
  const long long chi_stride = (long long)D * D * (bmajor ? 1 : chi);
  f.sEa = f.sOa2 = chi_stride;
  f.sEb = f.sOb2 = bmajor ? (long long)chi * D * D : 1;
  f.sEl2 = f.sOr2 = bmajor ? 1 : chi;
  f.sEl1 = f.sOr1 = D * f.sEl2;
  f.sTa = f.sBb = (long long)D * chi; f.sTu = f.sBd = chi; f.sTa2 = f.sBb2 = 1;
  f.ss1 = f.ss2 = (long long)D * D * D * D;
  f.s1l = f.s2l = (long long)D * D * D; f.s1u = f.s2u = (long long)D * D; f.s1r = f.s2r = D; f.s1d = f.s2d = 1;
  return f;
}
static unsigned status;
int host_env3(int n, int chi, int D, int mode) { return pv::env3_fused(env3(n, chi, D), mode == 3, &status, nullptr); }
int host_proj3(int n, int chi, int cV, int D, int mode) {
  pv::Proj3Fused f;
  f.batch = n;
  f.cT = f.cT2 = f.cV2 = chi;
  f.cV = cV;
  f.Dl = f.Dr = f.Du = f.Dd = D;
  f.L = at(1); f.T = at(2); f.A = at(3); f.R = at(5); f.out = at(6);
  f.bsL = f.bsT = f.bsR = f.bsO = (long long)chi * D * chi;
  f.sLa = f.sTa = f.sRa = f.sOv = (long long)D * chi;
  f.sLl = f.sTu = f.sRr = f.sOd = chi;
  f.sLv = f.sTa2 = f.sRv = f.sOv2 = 1;
  f.ssA = (long long)D * D * D * D;
  f.sAl = (long long)D * D * D; f.sAu = (long long)D * D; f.sAr = D; f.sAd = 1;
  return pv::proj3_fused(f, mode == 3, &status, nullptr);
}
int host_env4(int n, int chi, int D, int mode) { return pv::env4_fused(env4(n, chi, D, true), mode == 3, &status, nullptr); }
int host_env4_f32(int n) {
  pv::Env4Outs o;
  o.p[0] = at(6);
  return pv::env4_f32(env4(n, 16, 4, false), o, false, nullptr);
}
int host_proj_f32(int n) {
  pv::Mid3 mid;
  mid.p = at(7);
  return pv::env3_f32(env3(n, 24, 6), nullptr, true, false, mid, nullptr);
}
int host_dot(int n, int chains) { return pv::k_dot(at(1), n, at(2), n, n, (double*)at(3), chains, &status, nullptr); }
int host_normalize(int n, int arrays, int chains) {
  return pv::k_normalize_pow2(at(1), n, n, arrays > 1 ? at(2) : nullptr, n, arrays > 1 ? n : 0, arrays > 2 ? at(3) : nullptr, n,
                              arrays > 2 ? n : 0, (int*)at(4), chains, &status, nullptr);
}
int host_env3_f32(int n, int chi, int D) { return pv::env3_f32(env3(n, chi, D), nullptr, false, false, pv::Mid3(), nullptr); }
int host_gemm_tc(int mode, int bn) {
  pv::GemmDesc g;
  g.M = g.N = g.K = 128;
  g.batch = 2;
  g.A = at(1); g.B = at(2); g.C = at(3);
  g.sAm = g.sBn = g.sCn1 = 1;
  g.sAk = g.sBk = g.sCm1 = 128;
  return pv::gemm_tc(g, mode, bn, &status, nullptr);
}

}  // extern "C"
