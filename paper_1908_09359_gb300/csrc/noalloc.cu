// The three-line environment step for callers that cannot allocate device memory.
//
// Some callers of this library cannot call cudaMalloc at the point where they need
// an environment step: a service that reserved all of its device memory at start-up
// and must not allocate afterwards (cudaMalloc can synchronise the device and
// fragments a pre-planned pool), or host code that runs under a latency budget or
// holds a lock that an allocation could stall.  pepsvmc_env3_left needs a context,
// whose creation allocates; this entry point needs none.  Its two intermediates stay in
// shared memory where they fit; the separate products of larger steps (and of results that
// lie over an input) keep them in one fixed array of device memory that the library itself
// defines below.
//
// Host code cannot use the array's name as a device address (in host code it names
// a host-side stand-in), so every call that uses it looks the device address up with
// cudaGetSymbolAddress for the current device and context and passes it to the
// kernels.  The lookup allocates nothing and is cheap (0.13 us) once the library's device code is
// loaded; doing it per call (rather than caching it per device ordinal) keeps the
// address right after a device reset or when another context is current on the device.

#include "common.cuh"
#include "fused_f32.cuh"
#include "pepsvmc.h"
#include "stages.cuh"

using namespace pv;

namespace {

static __device__ __align__(256) float noalloc_scratch[PEPSVMC_NOALLOC_SCRATCH_FLOATS];

// Device address of noalloc_scratch in the current context.
int scratch_on_current_device(float** out) {
  void* p = nullptr;
  if (reported(cudaGetSymbolAddress(&p, noalloc_scratch)) != cudaSuccess || !p) return PEPSVMC_ECUDA;
  *out = static_cast<float*>(p);
  return PEPSVMC_OK;
}

}  // namespace

extern "C" int pepsvmc_env3_left_noalloc(const float* E, const float* T, const float* A, const int8_t* spins,
                                         const float* B, float* out, int32_t n_chains, int32_t cT, int32_t cB,
                                         int32_t cT2, int32_t cB2, int32_t Dl, int32_t Dr, int32_t Du, int32_t Dd,
                                         void* stream) {
  const Env3Dims d{cT, cB, cT2, cB2, Dl, Dr, Du, Dd};
  if (!E || !T || !A || !B || !out || n_chains < 1 || !env3_dims_ok(d)) return PEPSVMC_EINVAL;
  const long long per_chain = env3_scratch(d);
  if (per_chain > PEPSVMC_NOALLOC_SCRATCH_FLOATS / 2 / n_chains) return PEPSVMC_EINVAL;  // does not fit
  Env3Fused f;  // all intermediates in shared memory where they fit
  f.cT = cT; f.cB = cB; f.cT2 = cT2; f.cB2 = cB2; f.Dl = Dl; f.Dr = Dr; f.Du = Du; f.Dd = Dd;
  f.batch = n_chains;
  f.E = E; f.bsE = (long long)cT * Dl * cB; f.sEa = (long long)Dl * cB; f.sEl = cB; f.sEb = 1;
  f.T = T; f.bsT = (long long)cT * Du * cT2; f.sTa = (long long)Du * cT2; f.sTu = cT2; f.sTa2 = 1;
  f.A = A; f.ssA = (long long)Dl * Dr * Du * Dd;
  f.sAl = (long long)Du * Dr * Dd; f.sAu = (long long)Dr * Dd; f.sAr = Dd; f.sAd = 1;
  f.sel = spins; f.sel_stride = 1;
  f.B = B; f.bsB = (long long)cB * Dd * cB2; f.sBb = (long long)Dd * cB2; f.sBd = cB2; f.sBb2 = 1;
  f.out = out; f.bsO = (long long)cT2 * Dr * cB2; f.sOa2 = (long long)Dr * cB2; f.sOr = cB2; f.sOb2 = 1;
  const long long no = n_chains * f.bsO;
  if (env3_f32_fits(f) && !overlaps(out, no, E, n_chains * f.bsE) && !overlaps(out, no, T, n_chains * f.bsT) &&
      !overlaps(out, no, A, 2 * f.ssA) && !overlaps(out, no, B, n_chains * f.bsB) && !overlaps(out, no, spins, n_chains))
    return env3_f32(f, nullptr, false, false, Mid3(), (cudaStream_t)stream) == cudaSuccess ? PEPSVMC_OK : PEPSVMC_ECUDA;
  float* scratch = nullptr;
  const int rc = scratch_on_current_device(&scratch);
  if (rc != PEPSVMC_OK) return rc;
  float* t1 = scratch;
  float* t2 = scratch + (long long)n_chains * per_chain;
  GemmDesc g[3];
  env3_left_descs(g, d, E, (long long)cT * Dl * cB, T, (long long)cT * Du * cT2, A, (long long)Dl * Dr * Du * Dd,
                  spins, 1, 0, B, (long long)cB * Dd * cB2, out, (long long)cT2 * Dr * cB2, t1, t2, per_chain);
  for (int i = 0; i < 3; ++i) {
    g[i].batch = n_chains;
    if (gemm_f32(g[i], gemm_f32_pick(g[i]), (cudaStream_t)stream) != cudaSuccess) return PEPSVMC_ECUDA;
  }
  return PEPSVMC_OK;
}
