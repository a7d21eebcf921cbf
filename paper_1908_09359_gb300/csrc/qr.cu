// Batched Householder QR with a non-negative diagonal of R (thin Q only).
//
// The variational fit of App. B (arXiv:1908.09359) moves the orthogonality
// centre of the truncated MPS with a QR of every optimal site tensor; the
// random starting guess is made right-orthonormal the same way.  Choosing the
// sign of each column so that diag(R) >= 0 makes Q unique for full-rank input,
// so the truncated MPS does not depend on the QR routine used.
//
// One CTA per matrix.  General form: the matrix and the growing Q live in shared
// memory in column-major order; for rows <= 256, cols <= 32 a register-resident form
// (below) is used instead.  Reflector j: v = x + sign(x0)|x| e1, beta = 2/(v.v);
// a zero column gets no reflector and a zero diagonal.
#include "common.cuh"
#include "pepsvmc.h"

namespace pv {
namespace {

constexpr int kQrThreads = 256;
constexpr int kQrMaxCols = 64;
constexpr int kQrRegCols = 32;  // the register-resident form's maximum

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__global__ void __launch_bounds__(kQrThreads) qr_pos_kernel(const float* __restrict__ Y, long long bsY,
                                                            long long yrs, long long ycs, float* __restrict__ Q,
                                                            long long bsQ, long long qrs, long long qcs, int R,
                                                            int C) {
  extern __shared__ float sm[];
  float* A = sm;           // A[j*R + i]
  float* Qs = sm + R * C;  // Qs[j*R + i]
  __shared__ float beta[kQrMaxCols];
  __shared__ int flip[kQrMaxCols];
  __shared__ float red[kQrThreads / 32];

  const int b = blockIdx.x;
  const float* Yb = Y + (long long)b * bsY;
  for (int idx = threadIdx.x; idx < R * C; idx += blockDim.x) {
    const int i = idx % R, j = idx / R;
    A[idx] = Yb[(long long)i * yrs + (long long)j * ycs];
    Qs[idx] = (i == j) ? 1.f : 0.f;
  }
  __syncthreads();

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int j = 0; j < C; ++j) {
    float* a = A + j * R;
    float s = 0.f;
    for (int i = j + threadIdx.x; i < R; i += blockDim.x) s = fmaf(a[i], a[i], s);
    s = warp_sum(s);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      float tot = 0.f;
      for (int w = 0; w < nw; ++w) tot += red[w];
      const float alpha = sqrtf(tot);
      const float x0 = a[j];
      if (alpha == 0.f) {
        beta[j] = 0.f;
        flip[j] = 0;
      } else {
        const float sg = (x0 >= 0.f) ? 1.f : -1.f;
        a[j] = x0 + sg * alpha;
        beta[j] = 1.f / (alpha * (alpha + fabsf(x0)));
        flip[j] = (sg > 0.f) ? 1 : 0;  // R_jj = -sign(x0)|x| < 0 -> negate column j of Q
      }
    }
    __syncthreads();
    const float bj = beta[j];
    if (bj != 0.f) {
      for (int jj = j + 1 + warp; jj < C; jj += nw) {
        float* c = A + jj * R;
        float w = 0.f;
        for (int i = j + lane; i < R; i += 32) w = fmaf(a[i], c[i], w);
        w = warp_sum(w) * bj;
        for (int i = j + lane; i < R; i += 32) c[i] = fmaf(-w, a[i], c[i]);
      }
    }
    __syncthreads();
  }
  for (int j = C - 1; j >= 0; --j) {
    const float bj = beta[j];
    if (bj == 0.f) continue;
    const float* a = A + j * R;
    for (int jj = j + warp; jj < C; jj += nw) {
      float* q = Qs + jj * R;
      float w = 0.f;
      for (int i = j + lane; i < R; i += 32) w = fmaf(a[i], q[i], w);
      w = warp_sum(w) * bj;
      for (int i = j + lane; i < R; i += 32) q[i] = fmaf(-w, a[i], q[i]);
    }
    __syncthreads();
  }
  float* Qb = Q + (long long)b * bsQ;
  for (int idx = threadIdx.x; idx < R * C; idx += blockDim.x) {
    const int i = idx % R, j = idx / R;
    const float v = Qs[idx];
    Qb[(long long)i * qrs + (long long)j * qcs] = flip[j] ? -v : v;
  }
}

// Register-resident form for rows <= 256, cols <= 32 (every bulk shape of D <= 8,
// Dc <= 32).  A warp-wide reduction per column is what bounds a Householder QR of this
// size, so as much of every column sum as possible is done inside a thread: thread
// (group g, lane l) of 32-row group g holds the RPT rows of that group whose low bits
// are l, for all columns, and adds its own RPT products before any shuffle; the
// 32 / RPT lanes of a group finish the sum with a transposing butterfly over the live
// columns only (7/8 of a shuffle per column at RPT = 4), the group sums are added in
// group order from shared memory.  Every column sum is the same balanced tree over each
// group's 32 rows (row bits 4, 3, 2, 1, 0 in that order) followed by the groups in
// order, whatever RPT and W are.
//
// Bound: instruction issue when an SM holds several matrices, the dependent chain of one
// reflector (two reductions, ~0.5 us) when it holds one; RPT = 4 halves the instructions per
// matrix, RPT = 2 the chain.  Measured on 256 x 32, row-major / column-major, against the form
// with one row per thread and a 32-wide warp butterfly per reduction: 512 matrices 55.8 /
// 54.7 us (RPT 4; RPT 2: 61.6 / 59.5) from 112.2 / 84.9, 128 matrices 32.8 / 32.9 us (RPT 2;
// RPT 4: 39.0 / 43.1) from 53.3 / 45.2; 2048 of 144 x 24 125 / 133 us from 252 / 250.
//
// The column loop is rolled, eight columns to a block of fixed width: after the update
// column j + 1 + i moves to register i, so the current column is always register 0 and
// every index is static, and the code stays small enough for the instruction cache (fully
// unrolled it is 64 reflectors of ~270 instructions, each executed once per warp).  The
// reflectors are kept in shared memory, each thread's own entries as one vector.
template <int RPT>
struct VecOf;
template <>
struct VecOf<2> {
  using T = float2;
};
template <>
struct VecOf<4> {
  using T = float4;
};

// Columns each lane is left with after fold<N, MASK>.
template <int N, int MASK>
constexpr int fold_left() {
  if constexpr (MASK == 0) return N;
  else if constexpr (N % 2 == 0) return fold_left<N / 2, MASK / 2>();
  else return fold_left<N, MASK / 2>();
}
// Butterfly over the lanes of a group, largest mask first: sums of N columns; each level
// with an even count halves the columns a lane carries on.  start: the lane's first column.
template <int N, int MASK>
__device__ __forceinline__ void fold(float* p, int lane, int& start) {
  if constexpr (MASK > 0) {
    if constexpr (N % 2 == 0) {
      const bool up = (lane & MASK) != 0;
#pragma unroll
      for (int i = 0; i < N / 2; ++i) {
        const float send = up ? p[i] : p[i + N / 2];
        const float keep = up ? p[i + N / 2] : p[i];
        p[i] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, MASK));
      }
      if (up) start += N / 2;
      fold<N / 2, MASK / 2>(p, lane, start);
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) p[i] = __fadd_rn(p[i], __shfl_xor_sync(0xffffffffu, p[i], MASK));
      fold<N, MASK / 2>(p, lane, start);
    }
  }
}

// Sum of the RPT products of one column in this thread: row bit 4 first, then bit 3.
template <int RPT>
__device__ __forceinline__ float own_sum(const float (&x)[RPT]) {
  if constexpr (RPT == 2) return __fadd_rn(x[0], x[1]);
  else return __fadd_rn(__fadd_rn(x[0], x[1]), __fadd_rn(x[2], x[3]));
}

template <int RPT, int W, int NB>
struct QrTree {
  static constexpr int NT = 32 * W, NC = 8 * NB, LPG = 32 / RPT, NG = W * RPT;
  using Vec = typename VecOf<RPT>::T;
  struct Smem {
    Vec v[NC][NT];              // reflector j, this thread's rows
    float red[2][NG][NC + 4];   // group sums of the live columns
    float cs[W][NC];            // -beta w of the live columns, one copy per warp
    float redn[2][NG];          // group sums of the norm, by parity of j
    float x0s[2];
    float beta[NC];
    int flip[NC];
  };
  static __device__ __forceinline__ void sync() {
    if constexpr (W > 1) __syncthreads();
    else __syncwarp();
  }
  // row of slot s: slots differ in row bit 4, then bit 3
  static __device__ __forceinline__ int row_of(int tid, int s) {
    const int lane = tid & 31, g = (tid >> 5) * RPT + lane / LPG, l = lane % LPG;
    return g * 32 + l + ((s & 1) << 4) + ((s >> 1) << 3);
  }
  static __device__ __forceinline__ float norm_part(const float (&c)[RPT], int tid, int j) {
    float x[RPT];
#pragma unroll
    for (int s = 0; s < RPT; ++s) x[s] = row_of(tid, s) >= j ? __fmul_rn(c[s], c[s]) : 0.f;
    float t = own_sum<RPT>(x);
#pragma unroll
    for (int m = LPG / 2; m > 0; m >>= 1) t = __fadd_rn(t, __shfl_xor_sync(0xffffffffu, t, m));
    return t;
  }
  // group sums of N columns (already summed over this thread's rows) to c[0..N-1]
  // (-beta times the total) of every thread
  template <int N>
  static __device__ __forceinline__ void totals(Smem& sm, int buf, float (&p)[N], float bj, int tid, float (&c)[N]) {
    const int lane = tid & 31, warp = tid >> 5;
    int start = 0;
    fold<N, LPG / 2>(p, lane, start);
    constexpr int L = fold_left<N, LPG / 2>();
    float* r = sm.red[buf][warp * RPT + lane / LPG] + start;
#pragma unroll
    for (int i = 0; i < L; ++i) r[i] = p[i];
    sync();
    if (lane < N) {
      float t = sm.red[buf][0][lane];
#pragma unroll
      for (int g = 1; g < NG; ++g) t = __fadd_rn(t, sm.red[buf][g][lane]);
      sm.cs[warp][lane] = -bj * t;
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      const float4 f = *reinterpret_cast<const float4*>(&sm.cs[warp][i]);
      c[i] = f.x; c[i + 1] = f.y; c[i + 2] = f.z; c[i + 3] = f.w;
    }
  }

  // Columns 8b .. 8b+7 of the factorisation; a[s][i] is column j + i.
  template <int B>
  static __device__ __forceinline__ void factor(Smem& sm, float (&a)[RPT][NC], int tid, int C) {
    constexpr int N = 8 * (NB - B);
#pragma unroll 1
    for (int j = 8 * B; j < 8 * B + 8; ++j) {
      if (j >= C) break;
      const int par = j & 1;
      sync();
      float n2 = sm.redn[par][0];
#pragma unroll
      for (int g = 1; g < NG; ++g) n2 = __fadd_rn(n2, sm.redn[par][g]);
      const float alpha = sqrtf(n2), x0 = sm.x0s[par];
      const float sg = (x0 >= 0.f) ? 1.f : -1.f;
      const float bj = alpha == 0.f ? 0.f : 1.f / (alpha * (alpha + fabsf(x0)));
      if (tid == 0) {
        sm.beta[j] = bj;
        sm.flip[j] = (alpha != 0.f && sg > 0.f) ? 1 : 0;  // R_jj = -sign(x0)|x| < 0 -> negate column j of Q
      }
      float next[RPT];
      if (bj == 0.f) {  // uniform over the block: zero column, no reflector
#pragma unroll
        for (int s = 0; s < RPT; ++s) {
#pragma unroll
          for (int i = 0; i + 1 < N; ++i) a[s][i] = a[s][i + 1];
          next[s] = a[s][0];
        }
      } else {
        float v[RPT];
#pragma unroll
        for (int s = 0; s < RPT; ++s) {
          const int row = row_of(tid, s);
          v[s] = row > j ? a[s][0] : (row == j ? x0 + sg * alpha : 0.f);
        }
        *reinterpret_cast<Vec*>(&sm.v[j][tid]) = *reinterpret_cast<Vec*>(v);
        if (j + 1 == C) break;
        float p[N], c[N];
#pragma unroll
        for (int i = 0; i + 1 < N; ++i) {
          float x[RPT];
#pragma unroll
          for (int s = 0; s < RPT; ++s) x[s] = __fmul_rn(v[s], a[s][i + 1]);
          p[i] = own_sum<RPT>(x);
        }
        p[N - 1] = 0.f;
        totals<N>(sm, 0, p, bj, tid, c);
#pragma unroll
        for (int s = 0; s < RPT; ++s) next[s] = a[s][0] = fmaf(c[0], v[s], a[s][1]);
#pragma unroll
        for (int i = 1; i + 1 < N; ++i)
#pragma unroll
          for (int s = 0; s < RPT; ++s) a[s][i] = fmaf(c[i], v[s], a[s][i + 1]);
      }
      put_norm(sm, next, tid, j + 1);
    }
    if constexpr (B + 1 < NB) factor<B + 1>(sm, a, tid, C);
  }
  static __device__ __forceinline__ void put_norm(Smem& sm, const float (&c)[RPT], int tid, int j) {
    const float t = norm_part(c, tid, j);
    if (((tid & 31) % LPG) == 0) sm.redn[j & 1][(tid >> 5) * RPT + (tid & 31) / LPG] = t;
#pragma unroll
    for (int s = 0; s < RPT; ++s)
      if (row_of(tid, s) == j) sm.x0s[j & 1] = c[s];
  }

  // Thin Q = H_0 ... H_{C-1} [I; 0], accumulated backwards; H_j touches rows >= j and, at
  // that point, only columns >= j; q[s][i] is column j + i once reflector j is applied.
  template <int B>
  static __device__ __forceinline__ void accumulate(Smem& sm, float (&q)[RPT][NC], int tid, int C, int& par) {
    constexpr int N = 8 * (NB - B);
#pragma unroll 1
    for (int j = min(8 * B + 7, C - 1); j >= 8 * B; --j) {
      const float bj = sm.beta[j];
      float e[RPT];
#pragma unroll
      for (int s = 0; s < RPT; ++s) e[s] = row_of(tid, s) == j ? 1.f : 0.f;
      if (bj == 0.f) {
#pragma unroll
        for (int s = 0; s < RPT; ++s) {
#pragma unroll
          for (int i = N - 1; i > 0; --i) q[s][i] = q[s][i - 1];
          q[s][0] = e[s];
        }
        continue;
      }
      float v[RPT];
      *reinterpret_cast<Vec*>(v) = sm.v[j][tid];
      float p[N], c[N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        float x[RPT];
#pragma unroll
        for (int s = 0; s < RPT; ++s) x[s] = __fmul_rn(v[s], i == 0 ? e[s] : q[s][i > 0 ? i - 1 : 0]);
        p[i] = own_sum<RPT>(x);
      }
      totals<N>(sm, par, p, bj, tid, c);
      par ^= 1;
#pragma unroll
      for (int i = N - 1; i > 0; --i)
#pragma unroll
        for (int s = 0; s < RPT; ++s) q[s][i] = fmaf(c[i], v[s], q[s][i - 1]);
#pragma unroll
      for (int s = 0; s < RPT; ++s) q[s][0] = fmaf(c[0], v[s], e[s]);
    }
    if constexpr (B > 0) accumulate<B - 1>(sm, q, tid, C, par);
  }
};

// Y and Q may be the same array (in-place QR): a thread reads and writes only its own
// rows.  Barriers: in the factorisation one before the norm is read and one before the
// column sums are, so one buffer of column sums is enough; the Q accumulation has one
// barrier per reflector and alternates two buffers.
template <int RPT, int W, int NB>
__global__ void __launch_bounds__(32 * W, (RPT == 4 ? 8 : 16) / W) qr_pos_tree_kernel(const float* Y, long long bsY, long long yrs,
                                                             long long ycs, float* Q, long long bsQ, long long qrs,
                                                             long long qcs, int R, int C) {
  using T = QrTree<RPT, W, NB>;
  __shared__ __align__(16) typename T::Smem sm;
  after_previous();
  const int tid = threadIdx.x;
  const float* Yb = Y + (long long)blockIdx.x * bsY;
  float a[RPT][T::NC];
  // rows of four columns as 16-byte accesses when they are contiguous and aligned
  const bool vin = ycs == 1 && (C & 3) == 0 && ((yrs | bsY) & 3) == 0 && (reinterpret_cast<uintptr_t>(Y) & 15u) == 0;
#pragma unroll
  for (int s = 0; s < RPT; ++s) {
    const int row = T::row_of(tid, s);
    const float* y = Yb + (long long)row * yrs;
    if (vin) {
#pragma unroll
      for (int k = 0; k < T::NC; k += 4) {
        const float4 f = (row < R && k < C) ? *reinterpret_cast<const float4*>(y + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        a[s][k] = f.x; a[s][k + 1] = f.y; a[s][k + 2] = f.z; a[s][k + 3] = f.w;
      }
    } else {
#pragma unroll
      for (int k = 0; k < T::NC; ++k) a[s][k] = (row < R && k < C) ? y[(long long)k * ycs] : 0.f;
    }
  }
  {
    float c0[RPT];
#pragma unroll
    for (int s = 0; s < RPT; ++s) c0[s] = a[s][0];
    T::put_norm(sm, c0, tid, 0);
  }
  T::template factor<0>(sm, a, tid, C);
  T::sync();
#pragma unroll
  for (int s = 0; s < RPT; ++s)
#pragma unroll
    for (int k = 0; k < T::NC; ++k) a[s][k] = 0.f;
  int par = 0;
  T::template accumulate<NB - 1>(sm, a, tid, C, par);
  float* Qb = Q + (long long)blockIdx.x * bsQ;
  const bool vout = qcs == 1 && (C & 3) == 0 && ((qrs | bsQ) & 3) == 0 && (reinterpret_cast<uintptr_t>(Q) & 15u) == 0;
#pragma unroll
  for (int s = 0; s < RPT; ++s) {
    const int row = T::row_of(tid, s);
    if (row >= R) continue;
    float* o = Qb + (long long)row * qrs;
#pragma unroll
    for (int k = 0; k < T::NC; k += 4) {
      float f[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) f[i] = (k + i < C && sm.flip[k + i]) ? -a[s][k + i] : a[s][k + i];
      if (vout) {
        if (k < C) *reinterpret_cast<float4*>(o + k) = make_float4(f[0], f[1], f[2], f[3]);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (k + i < C) o[(long long)(k + i) * qcs] = f[i];
      }
    }
  }
}

template <int RPT, int W>
cudaError_t launch_tree(const float* Y, long long bsY, long long yrs, long long ycs, float* Q, long long bsQ,
                        long long qrs, long long qcs, int rows, int cols, int batch, cudaStream_t st) {
  switch ((cols + 7) / 8) {
    case 1: return launch_early(qr_pos_tree_kernel<RPT, W, 1>, batch, 32 * W, 0, st, Y, bsY, yrs, ycs, Q, bsQ, qrs, qcs, rows, cols);
    case 2: return launch_early(qr_pos_tree_kernel<RPT, W, 2>, batch, 32 * W, 0, st, Y, bsY, yrs, ycs, Q, bsQ, qrs, qcs, rows, cols);
    case 3: return launch_early(qr_pos_tree_kernel<RPT, W, 3>, batch, 32 * W, 0, st, Y, bsY, yrs, ycs, Q, bsQ, qrs, qcs, rows, cols);
    default: return launch_early(qr_pos_tree_kernel<RPT, W, 4>, batch, 32 * W, 0, st, Y, bsY, yrs, ycs, Q, bsQ, qrs, qcs, rows, cols);
  }
}

}  // namespace

cudaError_t qr_pos_batched(const float* Y, long long bsY, long long yrs, long long ycs, float* Q,
                           long long bsQ, long long qrs, long long qcs, int rows, int cols, int batch,
                           cudaStream_t st) {
  if (g_dry_run || batch <= 0) return cudaSuccess;
  if (cols > kQrMaxCols || rows < cols || cols <= 0) return cudaErrorInvalidValue;
  if (rows <= 256 && cols <= kQrRegCols) {
    // the fewest warps that cover the rows with RPT = 2; RPT = 4 once an SM holds more than two
    // matrices of the full width (figures above)
    if (rows <= 64) return launch_tree<2, 1>(Y, bsY, yrs, ycs, Q, bsQ, qrs, qcs, rows, cols, batch, st);
    if (rows <= 128) return launch_tree<2, 2>(Y, bsY, yrs, ycs, Q, bsQ, qrs, qcs, rows, cols, batch, st);
    int sms = 0;
    PV_CUDA(sm_count(&sms));
    if (cols > 24 && batch > 2 * sms)
      return launch_early(qr_pos_tree_kernel<4, 2, 4>, batch, 64, 0, st, Y, bsY, yrs, ycs, Q, bsQ, qrs, qcs, rows, cols);
    return launch_tree<2, 4>(Y, bsY, yrs, ycs, Q, bsQ, qrs, qcs, rows, cols, batch, st);
  }
  const size_t smem = (size_t)2 * rows * cols * sizeof(float);
  constexpr size_t kMost = kCtaSmem - kQrMaxCols * (sizeof(float) + sizeof(int)) - kQrThreads / 32 * sizeof(float);
  if (smem > kMost) return cudaErrorInvalidValue;
  static SmemLimit limit{kMost, false};
  return launch_large(limit, false, qr_pos_kernel, batch, kQrThreads, smem, st, Y, bsY, yrs, ycs, Q, bsQ, qrs, qcs, rows, cols);
}

}  // namespace pv

extern "C" int pepsvmc_qr_pos(const float* Y, float* Q, int32_t batch, int32_t rows, int32_t cols, int32_t col_major,
                              void* stream) {
  if (!Y || !Q || batch < 1 || cols < 1 || cols > 64 || rows < cols) return PEPSVMC_EINVAL;
  const long long bs = (long long)rows * cols;
  const long long rs = col_major ? 1 : cols, cs = col_major ? rows : 1;
  const cudaError_t e =
      pv::qr_pos_batched(Y, bs, rs, cs, Q, bs, rs, cs, rows, cols, batch, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? PEPSVMC_OK : PEPSVMC_ECUDA;
}
