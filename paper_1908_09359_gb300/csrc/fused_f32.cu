// Column steps in FP32 on the CUDA cores with every intermediate in shared memory (the
// three- and four-line steps of App. C in the default precision).
//
// One CTA takes one chain and one tile of 8 values of the outgoing top bond a', and runs the
// step's products one after the other.  All of them have one form: for every k in ascending
// order, one fused multiply-add per output, rows (i, a') by columns c,
//   S1  X(l,u | b,a')     = sum_a     T(a,u,a') E(a,l,b)          i = u,  c = (l,b)
//   S2  Y(b,d | r,a')     = sum_(l,u) X A_s(l,u,r,d)              i = b,  c = (r,d)
//   S3  O(a',r,b')        = sum_(b,d) Y B(b,d,b')                 i = r,  c = b'
// (four lines: one more product between S2 and S3), which is the sum, in the same order, that
// the separate products (contract_f32.cu) form, so results have the same bits.  a' stays the
// fastest index of every intermediate: a thread holds 8 (or 4) values of a' by 4 (or 2)
// columns and reads both operands as 16-byte words.
//
// The optimal site of the boundary-MPS fit is the same chain of products with a boundary bond
// in the place of a'; its middle product goes to memory as well, where the product that
// makes the next environment reads it (fit of Dc 16, D 4, 1024 chains: 92 us in three products,
// 32 us in one kernel, with ~6 us of event time per launch).
//
// Bound: FP32 arithmetic.  The separate products wrote and read every intermediate through
// global memory, 4 bytes per 32-byte sector where the next product wanted another order, and
// waited for their loads.  Here all operands of a step are in flight at once, by asynchronous
// copies (through registers, in turn, a third of the time went to loading: Dc 24, D 6 350 us,
// and odd bonds, one CTA per SM, were slower than the separate products: Dc 25, D 7, 40 chains
// 65 us against 40).  Measured in a graph, separate products (each with its fastest tile) -> this:
// three-line step Dc 24, D 6, 2048 chains 900 -> 238 us (30 TFLOP/s), Dc 16, D 4, 1024 chains 71.5 ->
// 18.7 us, 64 chains 15.7 -> 5.2 us, Dc 32, D 8, 512 chains 568 -> 254 us, Dc 23, D 7, 1624 chains 880 ->
// 484 us, Dc 25, D 7, 40 chains 49.6 -> 35.0 us; four-line step Dc 16, D 4, 1024 chains 376 -> 83 us,
// Dc 17, D 5, 104 chains 106 -> 82 us.  Over 1,900 drawn steps (bonds to 64 and 12, 1-2048 chains) about
// ten are slower, by up to 21 %, all of them ragged or four-line steps of a few chains.  Steps whose
// intermediates exceed a CTA's shared memory keep the separate products.
#include <limits.h>
#include <math.h>

#include "fused_f32.cuh"

namespace pv {
namespace {

constexpr int kTA = 8;        // a' per CTA
constexpr int kMaxSmem = kCtaSmem - 1024;

// One product of the chain.  Operand P (rows): element (k, i, j) at p + k*ldp + i*8 + j; operand
// Q (columns): element (k, c) at q + k*ldq + c (ldq and c padded to 4).  Output (i, c, j) at
// o + (i / ni2)*si1 + (i % ni2)*si2 + (c / nc2)*sc1 + (c % nc2)*sc2 + j*sj.
struct Product {
  int K, ni, nc;
  int ldp, ldq;
  int ni2, si1, si2, nc2, sc1, sc2;
};

// TJ values of a' by TC columns per thread; tasks run c fastest, then (TJ = 4) the half of a'.
struct Copy {  // of a product's output in global memory: (i, c, j) at p + i*si + (c / nc2)*sc1 + (c % nc2)*sc2 + j*sj
  float* p = nullptr;
  int si = 0, sc1 = 0, sc2 = 0, sj = 0;
  int nc2 = 1;
};
template <int TJ, int TC, bool GLOBAL, bool COPY>
__device__ __forceinline__ void product(const Product& g, const float* __restrict__ p, const float* __restrict__ q,
                                        float* o, int sj, int nj, const Copy& cp) {
  constexpr int H = kTA / TJ;
  const int ncg = (g.nc + TC - 1) / TC, tasks = g.ni * H * ncg;
  for (int t = threadIdx.x; t < tasks; t += blockDim.x) {
    const int cg = t % ncg, ih = t / ncg, i = ih / H, j0 = (ih % H) * TJ, c0 = cg * TC;
    const float* pp = p + i * kTA + j0;
    const float* qq = q + c0;
    float2 acc[TC][TJ / 2];
#pragma unroll
    for (int c = 0; c < TC; ++c)
#pragma unroll
      for (int j = 0; j < TJ / 2; ++j) acc[c][j] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int k = 0; k < g.K; ++k) {
      float2 a[TJ / 2];
      float b[TC];
#pragma unroll
      for (int j = 0; j < TJ; j += 4) {
        const float4 v = *reinterpret_cast<const float4*>(pp + j);
        a[j / 2] = make_float2(v.x, v.y);
        a[j / 2 + 1] = make_float2(v.z, v.w);
      }
      if constexpr (TC == 4) {
        const float4 v = *reinterpret_cast<const float4*>(qq);
        b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
      } else {
        const float2 v = *reinterpret_cast<const float2*>(qq);
        b[0] = v.x; b[1] = v.y;
      }
#pragma unroll
      for (int c = 0; c < TC; ++c)
#pragma unroll
        for (int j = 0; j < TJ / 2; ++j) acc[c][j] = __ffma2_rn(a[j], make_float2(b[c], b[c]), acc[c][j]);
      pp += g.ldp;
      qq += g.ldq;
    }
    const int oi = (i / g.ni2) * g.si1 + (i % g.ni2) * g.si2;
#pragma unroll
    for (int c = 0; c < TC; ++c) {
      if (c0 + c >= g.nc) break;
      float* d = o + oi + ((c0 + c) / g.nc2) * g.sc1 + ((c0 + c) % g.nc2) * g.sc2 + j0 * sj;
      if constexpr (!GLOBAL) {
#pragma unroll
        for (int j = 0; j < TJ; j += 4)
          *reinterpret_cast<float4*>(d + j) =
              make_float4(acc[c][j / 2].x, acc[c][j / 2].y, acc[c][j / 2 + 1].x, acc[c][j / 2 + 1].y);
      } else {
#pragma unroll
        for (int j = 0; j < TJ; ++j)
          if (j0 + j < nj) d[j * sj] = (j & 1) ? acc[c][j / 2].y : acc[c][j / 2].x;
      }
    }
    if constexpr (COPY) {
      {
        float* d = cp.p + i * cp.si + j0 * cp.sj;
        const int e = c0 % cp.nc2;
        if (TC == 4 && cp.sc2 == 1 && c0 + 3 < g.nc && e + 3 < cp.nc2 &&
            ((reinterpret_cast<uintptr_t>(cp.p) | ((cp.si | cp.sc1 | cp.sj | e) * 4)) & 15) == 0) {
          d += (c0 / cp.nc2) * cp.sc1 + e;
#pragma unroll
          for (int j = 0; j < TJ; ++j)
            if (j0 + j < nj)
              *reinterpret_cast<float4*>(d + j * cp.sj) =
                  (j & 1) ? make_float4(acc[0][j / 2].y, acc[1][j / 2].y, acc[TC - 2][j / 2].y, acc[TC - 1][j / 2].y)
                          : make_float4(acc[0][j / 2].x, acc[1][j / 2].x, acc[TC - 2][j / 2].x, acc[TC - 1][j / 2].x);
        } else {
#pragma unroll
          for (int c = 0; c < TC; ++c) {
            if (c0 + c >= g.nc) break;
            float* f = d + ((c0 + c) / cp.nc2) * cp.sc1 + ((c0 + c) % cp.nc2) * cp.sc2;
#pragma unroll
            for (int j = 0; j < TJ; ++j)
              if (j0 + j < nj) f[j * cp.sj] = (j & 1) ? acc[c][j / 2].y : acc[c][j / 2].x;
          }
        }
      }
    }
  }
}
// The widest tile that still gives every thread something to do.
template <bool GLOBAL, bool COPY = false>
__device__ __forceinline__ void run(const Product& g, const float* p, const float* q, float* o, int sj = 1, int nj = kTA,
                                    const Copy& cp = Copy()) {
  const int cols4 = (g.nc + 3) / 4;
  if (2 * g.ni * cols4 > (int)blockDim.x) product<8, 4, GLOBAL, COPY>(g, p, q, o, sj, nj, cp);
  else product<4, 2, GLOBAL, COPY>(g, p, q, o, sj, nj, cp);
}

// Operands come in by asynchronous copies, all of a step's in flight at once; loads_done waits
// for this thread's (before the barrier that precedes their use).
template <int BYTES>
__device__ __forceinline__ void copy_async(float* dst, const float* src, bool valid = true) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void loads_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The threads as rows of 1 to 32 lanes (a power of two that covers n, if 32 do).
struct Rows {
  int lanes, lane, row, rows;
  __device__ __forceinline__ explicit Rows(int n) {
    const int lg = n >= 32 ? 5 : 32 - __clz(n - 1);
    lanes = 1 << lg;
    lane = threadIdx.x & (lanes - 1);
    row = threadIdx.x >> lg;
    rows = blockDim.x >> lg;
  }
};

// dst[k*ld + c] for k < n0 * n1 (n0 outer), c < nc, c = (c / nc2, c % nc2), zero up to ld.
__device__ __forceinline__ void load_cols(float* dst, int ld, const float* src, int n0, int s0, int n1, int s1, int nc,
                                          int nc2, int sc1, int sc2) {
  const bool row = sc2 == 1 && (nc == nc2 || sc1 == nc2);  // rows contiguous
  // a dense block in the same order: 16-byte copies
  if (ld == nc && row && (n1 == 1 || s1 == nc) && s0 == n1 * nc && (reinterpret_cast<uintptr_t>(src) & 15) == 0) {
    const int n = n0 * n1 * nc / 4;
    for (int e = threadIdx.x; e < n; e += blockDim.x) copy_async<16>(dst + 4 * e, src + 4 * e);
  } else if (n1 == 1 && s0 == 1 && sc2 != 1) {  // k contiguous (a mirrored view): lanes along k
    const Rows t(n0);
    for (int c = t.row; c < ld; c += t.rows) {
      const float* p = src + (c < nc ? (c / nc2) * sc1 + (c % nc2) * sc2 : 0);
      for (int k = t.lane; k < n0; k += t.lanes) copy_async<4>(dst + k * ld + c, p + k, c < nc);
    }
  } else {
    const Rows t(ld);
    for (int k = t.row; k < n0 * n1; k += t.rows) {
      const float* p = src + (n1 == 1 ? k * s0 : (k / n1) * s0 + (k % n1) * s1);
      for (int c = t.lane; c < ld; c += t.lanes)
        copy_async<4>(dst + k * ld + c, c < nc ? p + (row ? c : (c / nc2) * sc1 + (c % nc2) * sc2) : src, c < nc);
    }
  }
}
// T tile: dst[(a*Du + u)*8 + j], zero beyond the bond.
__device__ __forceinline__ void load_top(float* dst, const float* T, int cT, int Du, int sTa, int sTu, int sTa2, int nj) {
  const int n = cT * Du * kTA;
  if (sTa2 == 1 && nj == kTA && ((reinterpret_cast<uintptr_t>(T) | (sTa | sTu) * 4) & 15) == 0) {
    for (int e = threadIdx.x; e < n / 4; e += blockDim.x) {
      const int au = e >> 1, a = au / Du;
      copy_async<16>(dst + 4 * e, T + a * sTa + (au - a * Du) * sTu + (e & 1) * 4);
    }
  } else if (sTa2 == 1 || sTa != 1) {
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
      const int j = e % kTA, au = e / kTA, a = au / Du;
      copy_async<4>(dst + e, j < nj ? T + a * sTa + (au - a * Du) * sTu + j * sTa2 : T, j < nj);
    }
  } else {  // a contiguous (mirrored view): lanes along a
    const Rows t(cT);
    for (int ju = t.row; ju < kTA * Du; ju += t.rows) {
      const int j = ju / Du, u = ju - j * Du;
      for (int a = t.lane; a < cT; a += t.lanes)
        copy_async<4>(dst + (a * Du + u) * kTA + j, j < nj ? T + a + u * sTu + j * sTa2 : T, j < nj);
    }
  }
}
__host__ __device__ inline int pad4(int n) { return (n + 3) & ~3; }
inline double pad4(double n) { return 4 * ceil(n / 4); }

__device__ __forceinline__ int slot_of(const int8_t* sel, long long stride, int flip, int c) {
  return sel ? ((sel[c * stride] < 0) ? 1 : 0) ^ flip : 0;
}

// Floats of shared memory: E, T, A, B, X; Y takes the place of E and T, which only the first
// product reads.  N: int for a step that fits; double (whatever the bonds, no product of them wraps
// around) where that is still to be decided.
template <typename N>
__host__ __device__ inline N layout3(const Env3Fused& a, N off[5]) {
  const N cT = a.cT, cB = a.cB, cB2 = a.cB2, Dl = a.Dl, Dr = a.Dr, Du = a.Du, Dd = a.Dd;
  const N t = cT * pad4(Dl * cB), et = t + cT * Du * kTA, y = cB * Dd * Dr * kTA;
  off[0] = 0;
  off[1] = t;
  off[2] = et > y ? et : y;
  off[3] = off[2] + Dl * Du * pad4(Dr * Dd);
  off[4] = off[3] + cB * Dd * pad4(cB2);
  return off[4] + Dl * Du * cB * kTA;
}

template <bool MID>
__global__ void __maxnreg__(80) env3_f32_kernel(const Env3Fused a, float* out1, bool rev2, bool rev3, const Mid3 mid) {
  extern __shared__ __align__(16) float sf[];
  int off[5];
  layout3(a, off);
  float *E = sf + off[0], *T = sf + off[1], *A = sf + off[2], *B = sf + off[3], *X = sf + off[4], *Y = sf;
  const int n_at = (a.cT2 + kTA - 1) / kTA, c = blockIdx.x / n_at, a0 = (blockIdx.x % n_at) * kTA;
  const int nj = min(kTA, a.cT2 - a0);
  after_previous();
  const int slot = slot_of(a.sel, a.sel_stride, a.sel_xor, c);
  const int ldE = pad4(a.Dl * a.cB), ldA = pad4(a.Dr * a.Dd), ldB = pad4(a.cB2);
  const int sAl = (int)a.sAl, sAu = (int)a.sAu, sAr = (int)a.sAr, sAd = (int)a.sAd;
  auto load_site = [&](int s) {
    const float* src = a.A + s * a.ssA;
    if (rev2) load_cols(A, ldA, src, a.Du, sAu, a.Dl, sAl, a.Dr * a.Dd, a.Dd, sAr, sAd);
    else load_cols(A, ldA, src, a.Dl, sAl, a.Du, sAu, a.Dr * a.Dd, a.Dd, sAr, sAd);
  };
  load_cols(E, ldE, a.E + c * a.bsE, a.cT, (int)a.sEa, 1, 0, a.Dl * a.cB, a.cB, (int)a.sEl, (int)a.sEb);
  load_top(T, a.T + c * a.bsT + a0 * a.sTa2, a.cT, a.Du, (int)a.sTa, (int)a.sTu, (int)a.sTa2, nj);
  load_site(slot);
  if (rev3) load_cols(B, ldB, a.B + c * a.bsB, a.Dd, (int)a.sBd, a.cB, (int)a.sBb, a.cB2, a.cB2, 0, (int)a.sBb2);
  else load_cols(B, ldB, a.B + c * a.bsB, a.cB, (int)a.sBb, a.Dd, (int)a.sBd, a.cB2, a.cB2, 0, (int)a.sBb2);
  loads_done();
  __syncthreads();
  const int ldX = a.cB * kTA, ldY = a.Dr * kTA;
  const int xl = rev2 ? ldX : a.Du * ldX, xu = rev2 ? a.Dl * ldX : ldX;
  const int yb = rev3 ? ldY : a.Dd * ldY, yd = rev3 ? a.cB * ldY : ldY;
  run<false>(Product{a.cT, a.Du, a.Dl * a.cB, a.Du * kTA, ldE, a.Du, 0, xu, a.cB, xl, kTA}, T, E, X);
  __syncthreads();
  const Product s2{a.Dl * a.Du, a.cB, a.Dr * a.Dd, ldX, ldA, a.cB, 0, yb, a.Dd, kTA, yd};
  const Product s3{a.cB * a.Dd, a.Dr, a.cB2, ldY, ldB, a.Dr, 0, (int)a.sOr, a.cB2, 0, (int)a.sOb2};
  for (int v = 0; v < 2; ++v) {
    float* O = v ? out1 : a.out;
    if (!O) break;
    if (v) {  // the other slot of the site, X shared
      load_site(slot ^ 1);
      loads_done();
      __syncthreads();
    }
    Copy cp;
    if constexpr (MID) {
      cp.p = mid.p + c * mid.bs + a0 * mid.sj;
      cp.si = mid.sb; cp.sc1 = mid.sr; cp.sc2 = mid.sd; cp.sj = mid.sj; cp.nc2 = a.Dd;
    }
    run<false, MID>(s2, X, A, Y, 1, nj, cp);
    __syncthreads();
    run<true>(s3, Y, B, O + c * a.bsO + a0 * a.sOa2, (int)a.sOa2, nj);
    if (v == 0 && out1) __syncthreads();
  }
}

// Floats of shared memory: E, T, A1, A2, B, X, Z; Y in the place of E and T, and with one
// variant Z in X's.  N as in layout3.
template <typename N>
__host__ __device__ inline N layout4(const Env4Fused& a, bool several, N off[7]) {
  const N cT = a.cT, cB = a.cB, cB2 = a.cB2, D1l = a.D1l, D1r = a.D1r, Du1 = a.Du1, Dd1 = a.Dd1, D2l = a.D2l, D2r = a.D2r,
          Dd2 = a.Dd2;
  const N x = D1l * Du1 * D2l * cB * kTA, z = cB * Dd2 * D1r * D2r * kTA;
  const N t = cT * pad4(D1l * D2l * cB), et = t + cT * Du1 * kTA, y = D2l * Dd1 * cB * D1r * kTA;
  off[0] = 0;
  off[1] = t;
  off[2] = et > y ? et : y;
  off[3] = off[2] + D1l * Du1 * pad4(D1r * Dd1);
  off[4] = off[3] + D2l * Dd1 * pad4(D2r * Dd2);
  off[5] = off[4] + cB * Dd2 * pad4(cB2);
  off[6] = off[5] + (several || x > z ? x : z);
  return off[6] + (several ? z : 0);
}

__global__ void __maxnreg__(80) env4_f32_kernel(const Env4Fused a, const Env4Outs outs, bool several, bool rev) {
  extern __shared__ __align__(16) float sf[];
  int off[7];
  layout4(a, several, off);
  float *E = sf + off[0], *T = sf + off[1], *A1 = sf + off[2], *A2 = sf + off[3], *B = sf + off[4], *X = sf + off[5], *Y = sf,
        *Z = several ? sf + off[6] : X;
  const int n_at = (a.cT2 + kTA - 1) / kTA, c = blockIdx.x / n_at, a0 = (blockIdx.x % n_at) * kTA;
  const int nj = min(kTA, a.cT2 - a0);
  const int nE = a.D1l * a.D2l * a.cB, ldE = pad4(nE), ld1 = pad4(a.D1r * a.Dd1), ld2 = pad4(a.D2r * a.Dd2),
            ldB = pad4(a.cB2);
  after_previous();
  const int slot1 = slot_of(a.sel1, a.sel_stride, a.xor1, c), slot2 = slot_of(a.sel2, a.sel_stride, a.xor2, c);
  auto load1 = [&](int s) {
    const float* src = a.A1 + s * a.ss1;
    if (rev) load_cols(A1, ld1, src, a.Du1, (int)a.s1u, a.D1l, (int)a.s1l, a.D1r * a.Dd1, a.Dd1, (int)a.s1r, (int)a.s1d);
    else load_cols(A1, ld1, src, a.D1l, (int)a.s1l, a.Du1, (int)a.s1u, a.D1r * a.Dd1, a.Dd1, (int)a.s1r, (int)a.s1d);
  };
  auto load2 = [&](int s) {
    const float* src = a.A2 + s * a.ss2;
    if (rev) load_cols(A2, ld2, src, a.Dd1, (int)a.s2u, a.D2l, (int)a.s2l, a.D2r * a.Dd2, a.Dd2, (int)a.s2r, (int)a.s2d);
    else load_cols(A2, ld2, src, a.D2l, (int)a.s2l, a.Dd1, (int)a.s2u, a.D2r * a.Dd2, a.Dd2, (int)a.s2r, (int)a.s2d);
  };
  // E's columns (l1, l2, b): l1 and l2 are one index of stride sEl2 (dense storage)
  load_cols(E, ldE, a.E + c * a.bsE, a.cT, (int)a.sEa, 1, 0, nE, a.cB, (int)a.sEl2, (int)a.sEb);
  load_top(T, a.T + c * a.bsT + a0 * a.sTa2, a.cT, a.Du1, (int)a.sTa, (int)a.sTu, (int)a.sTa2, nj);
  if (rev) load_cols(B, ldB, a.B + c * a.bsB, a.Dd2, (int)a.sBd, a.cB, (int)a.sBb, a.cB2, a.cB2, 0, (int)a.sBb2);
  else load_cols(B, ldB, a.B + c * a.bsB, a.cB, (int)a.sBb, a.Dd2, (int)a.sBd, a.cB2, a.cB2, 0, (int)a.sBb2);
  const int n2b = a.D2l * a.cB, ldX = n2b * kTA, ldY = a.cB * a.D1r * kTA, ldZ = a.D1r * a.D2r * kTA;
  const int xl = rev ? ldX : a.Du1 * ldX, xu = rev ? a.D1l * ldX : ldX;
  const int yl = rev ? ldY : a.Dd1 * ldY, yd = rev ? a.D2l * ldY : ldY;
  const int zb = rev ? ldZ : a.Dd2 * ldZ, zd = rev ? a.cB * ldZ : ldZ;
  bool fresh = true;
  for (int f1 = 0; f1 < 2; ++f1) {
    if (!outs.p[2 * f1] && !outs.p[2 * f1 + 1]) continue;
    load1(slot1 ^ f1);
    loads_done();
    __syncthreads();
    // X(l1,u1 | l2,b): columns (l1, (l2,b)), rows u1
    if (fresh) {
      run<false>(Product{a.cT, a.Du1, nE, a.Du1 * kTA, ldE, a.Du1, 0, xu, n2b, xl, kTA}, T, E, X);
      __syncthreads();
      fresh = false;
    }
    // Y(l2,d1 | b,r1): rows (l2, b), columns (r1, d1)
    run<false>(Product{a.D1l * a.Du1, n2b, a.D1r * a.Dd1, ldX, ld1, a.cB, yl, a.D1r * kTA, a.Dd1, kTA, yd}, X, A1, Y);
    for (int f2 = 0; f2 < 2; ++f2) {
      float* O = outs.p[2 * f1 + f2];
      if (!O) continue;
      load2(slot2 ^ f2);
      loads_done();
      __syncthreads();
      // Z(b,d2 | r1,r2): rows (b, r1), columns (r2, d2)
      run<false>(Product{a.D2l * a.Dd1, a.cB * a.D1r, a.D2r * a.Dd2, ldY, ld2, a.D1r, zb, a.D2r * kTA, a.Dd2, kTA, zd}, Y, A2, Z);
      __syncthreads();
      // O(a',r1,r2,b'): rows (r1, r2), columns b'
      run<true>(Product{a.cB * a.Dd2, a.D1r * a.D2r, a.cB2, ldZ, ldB, a.D2r, (int)a.sOr1, (int)a.sOr2, a.cB2, 0, (int)a.sOb2},
                Z, B, O + c * a.bsO + a0 * a.sOa2, (int)a.sOa2, nj);
    }
  }
}

// Threads of a CTA.  Where CTAs share an SM: enough for the first products' tasks of 8 x 4, at most 256,
// or 512 where the shared memory lets an SM hold one CTA only.  A CTA that has an SM to itself is
// bound by the latency of its products, and takes as many threads as have work in the narrow tiles
// (run: 4 x 2, four times the tasks).  Measured over 580 steps of up to 152 CTAs, these / as where
// CTAs share: 0.89-0.96 of the time up to 16 tasks, 0.67-0.73 from 17 to 64, 0.82-0.86 to 128, 0.92-0.95
// above 256 (128 tasks fill 128 threads at once: 384 take 1.18 of the time); over 66 of up to 304 CTAs
// 0.72-0.84 from 17 to 64 tasks.  With 64 threads, few
// chains were slower than in separate products (a ragged step of Dc 19, 4 chains 14.8 us against
// 11.0; now 7.5).
int threads_for(int tasks, int smem, long long blocks, int sms) {
  if (blocks <= sms) {
    if (tasks < 128) return tasks > 64 ? 384 : tasks > 4 ? 256 : 64;
    if (tasks == 128) return 128;
    return tasks > 256 ? 512 : 256;
  }
  if (blocks <= 2LL * sms && tasks > 16 && tasks <= 64) return 256;
  return tasks > 256 && 2 * (smem + 1024) > 228 * 1024 ? 512 : tasks > 128 ? 256 : tasks > 64 ? 128 : 64;
}

}  // namespace

// The kernels address an operand's tile by 32-bit offsets.  What lies in shared memory as a whole
// bounds them; of T only a tile does, so its extent is looked at by itself.
static bool tile_in_32_bits(int cT, long long sTa, int Du, long long sTu, long long sTa2) {
  return (double)(cT - 1) * sTa + (double)(Du - 1) * sTu + (double)(kTA - 1) * sTa2 <= INT_MAX;
}

bool env3_f32_fits(const Env3Fused& a) {
  double off[5];
  return layout3(a, off) * 4 <= kMaxSmem && tile_in_32_bits(a.cT, a.sTa, a.Du, a.sTu, a.sTa2);
}

cudaError_t env3_f32(const Env3Fused& a, float* out1, bool rev2, bool rev3, const Mid3& mid, cudaStream_t st) {
  if (g_dry_run || a.batch <= 0) return cudaSuccess;
  int off[5];
  const int smem = layout3(a, off) * 4;
  const long long blocks = (long long)a.batch * ((a.cT2 + kTA - 1) / kTA);
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  const int tasks = a.Du * ((a.Dl * a.cB + 3) / 4), tasks2 = a.cB * ((a.Dr * a.Dd + 3) / 4);
  int sms = 0;
  PV_CUDA(sm_count(&sms));
  auto* kernel = mid.p ? env3_f32_kernel<true> : env3_f32_kernel<false>;
  const int threads = threads_for(tasks > tasks2 ? tasks : tasks2, smem, blocks, sms);
  if (smem <= 48 * 1024) return launch_early(kernel, (unsigned)blocks, threads, smem, st, a, out1, rev2, rev3, mid);
  static SmemLimit limit[2] = {{kMaxSmem, false}, {kMaxSmem, false}};
  return launch_large(limit[mid.p != nullptr], true, kernel, (unsigned)blocks, threads, smem, st, a, out1, rev2, rev3, mid);
}

static bool several(const Env4Outs& o) { return (o.p[0] != nullptr) + (o.p[1] != nullptr) + (o.p[2] != nullptr) + (o.p[3] != nullptr) > 1; }

bool env4_f32_fits(const Env4Fused& a, const Env4Outs& outs) {
  double off[7];
  return a.sEl1 == (long long)a.D2l * a.sEl2 && layout4(a, several(outs), off) * 4 <= kMaxSmem &&
         tile_in_32_bits(a.cT, a.sTa, a.Du1, a.sTu, a.sTa2);
}

// Passes over k of one product, in passes of the wide tile (run).
static double passes(double ni, double nc, double K, int threads) {
  const double wide = ni * ceil(nc / 4);
  return 2 * wide > threads ? ceil(wide / threads) * K : 0.5 * ceil(ni * 2 * ceil(nc / 2) / threads) * K;
}

// A CTA alone on its SM takes about 0.14 us per pass, however few others there are; the separate
// products spread a chain over many CTAs: 5.5 us a launch, and 3.9e6 multiply-adds per us once the
// chip is full.  Measured, separate / this: one chain of Dc 15, D 6 23.9 / 33.0 us, 3 of Dc 17, D 5 22.9 /
// 28.0, 2 of Dc 12, D 6 22.3 / 26.1, one of Dc 16, D 4 20.3 / 9.9.
bool env4_f32_takes(const Env4Fused& a, const Env4Outs& outs, int chains) {
  if (!env4_f32_fits(a, outs)) return false;
  const long long blocks = (long long)chains * ((a.cT2 + kTA - 1) / kTA);
  int sms = 0, off[7];
  if (sm_count(&sms) != cudaSuccess || blocks > sms) return true;
  const int n0 = (outs.p[0] != nullptr) + (outs.p[1] != nullptr), n1 = (outs.p[2] != nullptr) + (outs.p[3] != nullptr);
  const int flips = (n0 > 0) + (n1 > 0), n = n0 + n1;
  const int t = threads_for(a.D2l * a.cB * ((a.D1r * a.Dd1 + 3) / 4), layout4(a, several(outs), off) * 4, blocks, sms);
  const double E = (double)a.D1l * a.D2l * a.cB, Y = (double)a.D2l * a.cB, r1d1 = (double)a.D1r * a.Dd1, l1u1 = (double)a.D1l * a.Du1,
               Z = (double)a.cB * a.D1r, r2d2 = (double)a.D2r * a.Dd2, l2d1 = (double)a.D2l * a.Dd1, O = (double)a.D1r * a.D2r,
               bd2 = (double)a.cB * a.Dd2;
  const double here = 0.14 * (passes(a.Du1, E, a.cT, t) + flips * passes(Y, r1d1, l1u1, t) +
                              n * (passes(Z, r2d2, l2d1, t) + passes(O, a.cB2, bd2, t)));
  const double adds = chains * (double)a.cT2 * (a.Du1 * E * a.cT + flips * Y * r1d1 * l1u1 + n * (Z * r2d2 * l2d1 + O * a.cB2 * bd2));
  return here <= 5.5 * (1 + flips + 2 * n) + adds / 3.9e6;
}

cudaError_t env4_f32(const Env4Fused& a, const Env4Outs& outs, bool rev, cudaStream_t st) {
  if (g_dry_run || a.batch <= 0) return cudaSuccess;
  int off[7];
  const int smem = layout4(a, several(outs), off) * 4;
  const long long blocks = (long long)a.batch * ((a.cT2 + kTA - 1) / kTA);
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  const int tasks = a.D2l * a.cB * ((a.D1r * a.Dd1 + 3) / 4);
  int sms = 0;
  PV_CUDA(sm_count(&sms));
  const int threads = threads_for(tasks, smem, blocks, sms);
  if (smem <= 48 * 1024) return launch_early(env4_f32_kernel, (unsigned)blocks, threads, smem, st, a, outs, several(outs), rev);
  static SmemLimit limit{kMaxSmem, false};
  return launch_large(limit, true, env4_f32_kernel, (unsigned)blocks, threads, smem, st, a, outs, several(outs), rev);
}

}  // namespace pv
