// Column steps in FP32 on the CUDA cores, all products of a step in one kernel.
#pragma once
#include "fused.cuh"

namespace pv {

// Three-line step of every chain as Env3Fused describes it (any strides); out1 (nullable):
// the result with the other slot of the site tensor, sharing E . T.  rev2, rev3: the sums over
// (l, u), over (b, d) run u, d slowest (both in the separate products of a right step) instead
// of l, b.  mid.p (nullable): Y(b,d,r,a') is also stored at p[c*bs + b*sb + d*sd + r*sr + a'*sj].
// Sums ascend in k with one fused multiply-add per term, as gemm_f32's do.
struct Mid3 {
  float* p = nullptr;
  long long bs = 0;
  int sb = 0, sd = 0, sr = 0, sj = 0;
};
bool env3_f32_fits(const Env3Fused& a);
cudaError_t env3_f32(const Env3Fused& a, float* out1, bool rev2, bool rev3, const Mid3& mid, cudaStream_t st);

// Four-line step; p[2 f1 + f2] (nullable): the result with the slots of the two sites flipped by
// f1 and f2, sharing E . T and, between the two f2, the product with a1.  rev: the sums over
// (l1, u1), (l2, d1) and (b, d2) run the second index slowest.
struct Env4Outs {
  float* p[4] = {};
};
bool env4_f32_fits(const Env4Fused& a, const Env4Outs& outs);
// Whether it fits and is faster than the separate products at this number of chains.
bool env4_f32_takes(const Env4Fused& a, const Env4Outs& outs, int chains);
cudaError_t env4_f32(const Env4Fused& a, const Env4Outs& outs, bool rev, cudaStream_t st);

}  // namespace pv
