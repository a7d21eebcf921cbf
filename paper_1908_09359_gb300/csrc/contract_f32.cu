// FP32 batched tensor-contraction kernel (CUDA cores).
//
// Every contraction of the boundary-MPS method (App. B of arXiv:1908.09359:
// MPO x MPS fit steps, three-line and four-line environments of App. C, the
// defect network Delta of Eq. (7)) is written by the engine as a chain of
// batched matrix products over the Markov chains.  The kernel reads A and B
// through arbitrary (m,k)/(k,n) strides, selects the site tensor A_k^{s_k} per
// chain from the spin array (slot = sigma < 0), and scatters C into the layout
// the next stage wants (up to three nested indices on each of m and n), so no
// separate transpose kernels are needed.
//
// The products are small (K of a few tens, one or two tiles per chain), so a CTA's time is
// its load latency, not its arithmetic: the next BK values of k are fetched into registers
// while the present ones are multiplied.  Measured (1024 chains, with ~6 us of event time):
// M 64, N 16, K 64 29.9 -> 20.7 us; M 144, N 24, K 144 with 40 chains 20.9 -> 11.7 us.
#include "common.cuh"

namespace pv {
namespace {

template <int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__(256) gemm_f32_kernel(const GemmDesc d) {
  constexpr int TX = BN / TN;
  constexpr int TY = BM / TM;
  static_assert(TX * TY == 256, "256 threads per tile");
  __shared__ __align__(16) float As[BK][BM + 4];
  __shared__ __align__(16) float Bs[BK][BN + 4];
  __shared__ long long s_on[BN];  // C offset of each tile column (the same for every row)

  after_previous();
  const int b = blockIdx.y + blockIdx.z * gridDim.y;
  if (b >= d.batch) return;
  const int tiles_n = (d.N + BN - 1) / BN;
  const int m0 = (blockIdx.x / tiles_n) * BM;
  const int n0 = (blockIdx.x % tiles_n) * BN;

  const float* A = d.A + (long long)b * d.bsA;
  long long boff = (long long)b * d.bsB;
  if (d.sel) boff += (long long)(((d.sel[(long long)b * d.sel_stride] < 0) ? 1 : 0) ^ d.sel_xor) * d.ssB;
  const float* B = d.B + boff;

  const int t = threadIdx.x;
  const int tx = t % TX, ty = t / TX;
  for (int c = t; c < BN; c += 256) {
    const int n = n0 + c, cn23 = d.cn2 * d.cn3;
    s_on[c] = n < d.N ? (long long)(n / cn23) * d.sCn1 + (long long)((n / d.cn3) % d.cn2) * d.sCn2 +
                            (long long)(n % d.cn3) * d.sCn3
                      : 0;
  }
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;

  // this thread's elements of a tile of A: LA of them, dm rows and dk values of k apart
  const bool a_m_fast = (d.sAm == 1);
  const bool b_n_fast = (d.sBn == 1);
  static_assert(256 % BM == 0 && 256 % BN == 0 && 256 % BK == 0);
  constexpr int LA = BM * BK / 256, LB = BN * BK / 256;
  const int am = a_m_fast ? t % BM : t / BK, ak = a_m_fast ? t / BM : t % BK;
  const int adm = a_m_fast ? 0 : 256 / BK, adk = a_m_fast ? 256 / BM : 0;
  const int bn = b_n_fast ? t % BN : t / BK, bk = b_n_fast ? t / BN : t % BK;
  const int bdn = b_n_fast ? 0 : 256 / BK, bdk = b_n_fast ? 256 / BN : 0;
  const float* pa = A + (long long)(m0 + am) * d.sAm + (long long)ak * d.sAk;
  const float* pb = B + (long long)bk * d.sBk + (long long)(n0 + bn) * d.sBn;
  const long long ia = adm * d.sAm + adk * d.sAk, ib = bdk * d.sBk + bdn * d.sBn;
  float ra[LA], rb[LB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < LA; ++q)
      ra[q] = (m0 + am + q * adm < d.M && k0 + ak + q * adk < d.K) ? pa[k0 * d.sAk + q * ia] : 0.f;
#pragma unroll
    for (int q = 0; q < LB; ++q)
      rb[q] = (n0 + bn + q * bdn < d.N && k0 + bk + q * bdk < d.K) ? pb[k0 * d.sBk + q * ib] : 0.f;
  };
  fetch(0);
  for (int k0 = 0; k0 < d.K; k0 += BK) {
#pragma unroll
    for (int q = 0; q < LA; ++q) As[ak + q * adk][am + q * adm] = ra[q];
#pragma unroll
    for (int q = 0; q < LB; ++q) Bs[bk + q * bdk][bn + q * bdn] = rb[q];
    __syncthreads();
    if (k0 + BK < d.K) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[TM], bb[TN];
      if constexpr (TM % 4 == 0) {
#pragma unroll
        for (int i = 0; i < TM; i += 4) {
          const float4 v = *reinterpret_cast<const float4*>(&As[kk][ty * TM + i]);
          a[i] = v.x; a[i + 1] = v.y; a[i + 2] = v.z; a[i + 3] = v.w;
        }
      } else {
#pragma unroll
        for (int i = 0; i < TM; ++i) a[i] = As[kk][ty * TM + i];
      }
      if constexpr (TN % 4 == 0) {
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
          const float4 v = *reinterpret_cast<const float4*>(&Bs[kk][tx * TN + j]);
          bb[j] = v.x; bb[j + 1] = v.y; bb[j + 2] = v.z; bb[j + 3] = v.w;
        }
      } else if constexpr (TN % 2 == 0) {
#pragma unroll
        for (int j = 0; j < TN; j += 2) {
          const float2 v = *reinterpret_cast<const float2*>(&Bs[kk][tx * TN + j]);
          bb[j] = v.x; bb[j + 1] = v.y;
        }
      } else {
#pragma unroll
        for (int j = 0; j < TN; ++j) bb[j] = Bs[kk][tx * TN + j];
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], bb[j], acc[i][j]);
    }
    __syncthreads();
  }

  float alpha = d.alpha;
  if (d.inv_scale) alpha = (float)((double)alpha / d.inv_scale[b]);
  float* __restrict__ C = d.C + (long long)b * d.bsC;
  const int cm23 = d.cm2 * d.cm3;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty * TM + i;
    if (m >= d.M) continue;
    const long long om = (long long)(m / cm23) * d.sCm1 + (long long)((m / d.cm3) % d.cm2) * d.sCm2 +
                         (long long)(m % d.cm3) * d.sCm3;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int n = n0 + tx * TN + j;
      if (n >= d.N) continue;
      const long long on = s_on[tx * TN + j];
      const float v = alpha * acc[i][j];
      if (d.accumulate) C[om + on] += v; else C[om + on] = v;
    }
  }
}

struct Cfg {
  int BM, BN;
  const char* name;
};
const Cfg kCfgs[] = {{64, 64, "f32_64x64"},  {128, 64, "f32_128x64"}, {64, 32, "f32_64x32"},
                     {32, 32, "f32_32x32"},  {128, 32, "f32_128x32"}, {128, 128, "f32_128x128"}};

template <int BM, int BN, int TM, int TN>
cudaError_t launch(const GemmDesc& d, cudaStream_t st) {
  const int tiles = ((d.M + BM - 1) / BM) * ((d.N + BN - 1) / BN);
  dim3 grid(tiles, d.batch < 65535 ? d.batch : 65535, (d.batch + 65534) / 65535);
  return launch_early(gemm_f32_kernel<BM, BN, 16, TM, TN>, grid, 256, 0, st, d);
}

}  // namespace

int gemm_f32_num_configs() { return (int)(sizeof(kCfgs) / sizeof(kCfgs[0])); }
const char* gemm_f32_config_name(int cfg) { return kCfgs[cfg].name; }

int gemm_f32_pick(const GemmDesc& d) {
  if (d.N <= 32) return d.M >= 128 ? 4 : (d.M >= 64 ? 2 : 3);
  if (d.N <= 64) return d.M >= 128 ? 1 : 0;
  return d.M >= 128 ? 5 : 0;
}

cudaError_t gemm_f32(const GemmDesc& d, int cfg, cudaStream_t st) {
  if (g_dry_run || d.M <= 0 || d.N <= 0 || d.batch <= 0) return cudaSuccess;
  switch (cfg) {
    case 0: return launch<64, 64, 4, 4>(d, st);
    case 1: return launch<128, 64, 8, 4>(d, st);
    case 2: return launch<64, 32, 4, 2>(d, st);
    case 3: return launch<32, 32, 2, 2>(d, st);
    case 4: return launch<128, 32, 8, 2>(d, st);
    case 5: return launch<128, 128, 8, 8>(d, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pv
