// Fused three-line column step and optimal site of the fit on the tcgen05 tensor cores
// (App. C, Fig. "contraction" (c); the same network closes the three-line environments of
// the sampler's ratios, Eq. (9), and of the measurement, Eqs. (3)-(7); App. B for the fit).
//
// Three-line step, per tile of 8 values of the outgoing top bond a' and 16 of the incoming
// bottom bond b:
//   S1  X[(b,l)][(a',u)]   = sum_a     E(a,l,b) T(a,u,a')          M 128, N 64, K 32
//   S2  Y[(b,a')][(r,d)]   = sum_(l,u) X A_s(l,u,r,d)              M 128, N 64, K 64
//   S3  O[(r,a')][b']     += sum_(b,d) Y B(b,d,b')                 M  64, N 32, K 128
// S3 accumulates over the b tiles in tensor memory.  The S1 and S2 accumulators are drained
// by the drain warps (one accumulator row per thread, tcgen05.ld) and stored, re-indexed
// and split into BF16 hi + lo, as the next product's A operand: S2's in the 128-byte
// swizzled layout, S3's without swizzle; in both the eight lanes that write one row group
// hit eight different bank groups.
//
// Split BF16 (x = hi + lo, the lo*lo term dropped) needs three BF16 products per step;
// they are merged into fewer, wider MMAs:
//   S1, S2: A_hi x [B_hi | B_lo] as one MMA of twice the width, plus A_lo x B_hi; the
//           drain adds the two column halves;
//   S3:     [Y_hi ; Y_lo] x [B_hi | B_lo] as one MMA of M 128, N 64 (the lo*lo quadrant
//           is computed and ignored); the final drain adds three quadrants.
// The lo copy of every operand tile directly follows its hi copy with the same row-group
// stride, so one descriptor addresses both.
//
// What bounds it: an MMA of N <= 128 costs its operands' shared-memory reads (measured 49,
// 51 and 67 cycles at N = 32, 64 and 128, M 128, K 16: 5, 6 and 8 KB at 128 B/cycle, in any
// layout), so a tile's products read 132 KB and its drains write 64 KB: ~1,600 cycles of
// shared memory, against ~4,500 cycles of dependent latency (product, drain, product, drain,
// product).  Hence one CTA per SM with two streams, each a chain of tiles with its own
// drain warps, accumulators and operand buffer: while one stream waits for a product the
// other drains.  The streams take the two a' tiles of a pair (the fit: the two v tiles) of
// the same chain, so E, T, A and B are converted and kept once for both.  What is left beside
// the drains' latency (~960 cycles each) is the change of chain, where the products wait for
// the conversion of the next operands (~4,000 of 25,000 cycles a chain at Dc 32, D 8).
// Launches of few tiles of bonds below the maxima, where there is nothing to overlap, go to
// fused_env3_tiles.cu (one tile per CTA, two CTAs per SM).
//
// Dc 32, D 8, split BF16, one tile per CTA -> this form: three-line step 128 chains 29.2 ->
// 21.1 us, 512 chains 90.9 -> 52.8 us, 2048 chains 364 -> 176 us (launched early, back to back,
// 19.7, 50.6 and 174: 109, 170 and 197 TFLOP/s; shared-memory data pipe 74 % busy); optimal site of
// the fit 512 chains 98.8 -> 66.9 us, 128 chains 33.2 -> 25 us.  Dc 24, D 6, 2048 chains 261 ->
// 188 us.  Tried and slower (512 chains): operands converted straight from global loads by
// eight warps and written out by the drains, 64.5 us; by two groups of four, 90 us; all of it
// unrolled in line (115 KB of code, instruction fetch at 79 % of its rate), 75 us; one rolled
// loop for all operand kinds, 76 us; results written by the converting warps, 68 us.
#include <math.h>

#include "fused.cuh"
#include "fused_pipe.cuh"

namespace pv {
namespace {

using namespace tc;

constexpr int kAT = 8;   // a' per tile
constexpr int kBT = 16;  // b per tile

// Byte offsets of the operand tiles (hi part; the lo part follows at + size).
constexpr uint32_t SZ_W = 128 * 128;                                  // X (S2 A, swizzled) or Y (S3 A)
constexpr uint32_t OFF_W = 0;                                         // [stream]
constexpr uint32_t SZ_E = 128 * 64;                                   // S1 A: 128 rows x 32 K
constexpr uint32_t SZ_T = 64 * 64;                                    // S1 B: 64 rows x 32 K
constexpr uint32_t SZ_A = 64 * 128;                                   // S2 B: 64 rows x 64 K
// S3 B: 32 rows (b') x 128 K ((b,d)) in the 128-byte swizzled layout, two K atoms of 64;
// with X3 the lo rows follow the hi rows inside each atom (one operand of 64 rows), so an
// atom holds 64 rows x 128 bytes.
constexpr uint32_t SZ_B = 2 * 64 * 128;
constexpr uint32_t B_ATOM = 64 * 128, B_LO = 32 * 128;
constexpr uint32_t OFF_B = OFF_W + 2 * 2 * SZ_W;                      // [b tile]
constexpr uint32_t OFF_E = OFF_B + 2 * SZ_B;                          // [b tile]
constexpr uint32_t OFF_T = OFF_E + 2 * 2 * SZ_E;                      // [a' tile]
constexpr uint32_t OFF_A = OFF_T + 4 * 2 * SZ_T;
constexpr uint32_t OFF_STAGE = OFF_A + 2 * SZ_A;
constexpr uint32_t OFF_XCH = OFF_STAGE + 2 * kStageBytes;             // 64 output rows
constexpr uint32_t SMEM_BYTES = OFF_XCH + 64 * kRowPitch * 4;
constexpr uint32_t TMEM_COLS = 512, TMEM_STREAM = 256;
constexpr uint32_t COL_S12 = 0, COL_S3 = 128;  // S1 and S2 share columns 0-127 (each is drained before the next)
static_assert(SMEM_BYTES + 1024 <= 232448, "the three-line CTA (with up to 1 KB of barriers) must fit an SM");

// This thread's accumulator row, columns 32 h .. 32 h + 31, as four K chunks of 8 at byte
// offsets off + i * stride (+ 16 ((lo3 ^ (4 h + i)) & 7): swz, the swizzled layout) of the
// operand tile.
template <bool X3>
__device__ __forceinline__ void drain_rows(uint32_t taddr, uint8_t* tile, uint32_t stride, bool swz, int lo3, int h4) {
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    float v[16];
    load_acc16<X3>(taddr + g * 16, v);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = g * 2 + k;
      put_split8<X3>(tile + i * stride + (swz ? ((lo3 ^ (h4 + i)) & 7) << 4 : 0), v + k * 8, SZ_W);
    }
  }
}

// ------------------------------------------------------------------ three-line step
struct Bars3 {
  Staging stage;
  uint64_t full[4];                          // loaders -> products, once per chain: E, T, A, B
  uint64_t free_[4];                         // products -> loaders, one arrival per stream and chain ([0]: E and T)
  uint64_t acc[2], w[2];                     // products <-> drain
  uint64_t o_full[2], o_free[2], fin[2];     // products <-> output
  uint64_t x_full, x_free;                   // output quarters 2, 3 <-> 0, 1
};

// Units: (chain, a' tiles of `step` streams); a CTA owns a contiguous range of items of `align`
// units, so consecutive units mostly share the chain and with it E, T, A and B.  Two streams
// per unit, except when that would leave SMs without work: then every a' tile is a unit of
// its own (first stream only; full bonds, 38 chains 10.2 us, with two streams 12.7).
// When the last unit of a chain has no tile for the second stream, an item is a whole chain.
struct Plan3 {
  Env3Fused a;
  PipeOp op[4];  // E, T, A, B in the order in which they are needed
  int n_at, n_bt, step, per_chain, streams, align;
  int share, rest;  // items per CTA, and how many CTAs take one more
};
struct Range3 {
  int c, p, units;  // first unit (chain, unit within it) and how many
};
__device__ __forceinline__ Range3 range_of(const Plan3& P) {
  const int i = blockIdx.x, items = P.share + (i < P.rest ? 1 : 0);
  const int u = (i * P.share + min(i, P.rest)) * P.align;
  return Range3{u / P.per_chain, u % P.per_chain, items * P.align};
}
Plan3 plan3(const Env3Fused& a, int sms, int& grid) {
  Plan3 P;
  P.a = a;
  P.n_at = (a.cT2 + kAT - 1) / kAT;
  P.n_bt = (a.cB + kBT - 1) / kBT;
  P.step = (long long)a.batch * P.n_at <= sms ? 1 : 2;
  P.per_chain = (P.n_at + P.step - 1) / P.step;
  P.streams = P.step < P.n_at ? P.step : P.n_at;
  P.align = P.n_at % P.step ? P.per_chain : 1;
  const int items = (int)((long long)a.batch * P.per_chain / P.align);
  grid = items < sms ? items : sms;
  P.share = items / grid;
  P.rest = items % grid;
  PipeOp &E = P.op[0], &T = P.op[1], &A = P.op[2], &B = P.op[3];
  auto set = [](PipeOp& o, int kind, const float* base, long long chain, int n0, long long s0, int n1, long long s1, int n2,
                long long s2) {
    o.kind = kind; o.base = base; o.chain = chain;
    o.n[0] = n0; o.s[0] = (int)s0; o.n[1] = n1; o.s[1] = (int)s1; o.n[2] = n2; o.s[2] = (int)s2;
  };
  set(E, OP_KXY, a.E, a.bsE, a.cT, a.sEa, a.Dl, a.sEl, a.cB, a.sEb);
  E.dst = OFF_E; E.tile = 2 * SZ_E; E.lo = SZ_E; E.ys = 4;
  set(T, a.sTa2 > a.sTa ? OP_YXK : OP_KXY, a.T, a.bsT, a.cT, a.sTa, a.Du, a.sTu, a.cT2, a.sTa2);
  T.dst = OFF_T; T.tile = 2 * SZ_T; T.lo = SZ_T; T.ys = 3;
  set(A, OP_SITE, a.A, a.ssA, a.Dl, a.sAl, a.Du, a.sAu, a.Dr, a.sAr);
  A.n[3] = a.Dd; A.s[3] = (int)a.sAd;
  A.dst = OFF_A; A.lo = SZ_A;
  set(B, a.sBb2 > a.sBb ? OP_YEO : OP_OE, a.B, a.bsB, a.cB, a.sBb, a.Dd, a.sBd, a.cB2, a.sBb2);
  B.dst = OFF_B; B.tile = SZ_B; B.lo = B_LO; B.swizzled = 1;
  for (PipeOp& o : P.op) finish_operand(o);
  return P;
}
__device__ __forceinline__ int slot_of(const int8_t* sel, long long stride, int flip, int c) {
  return sel ? ((sel[c * stride] < 0) ? 1 : 0) ^ flip : 0;
}

// Chains a CTA's range touches.
__device__ __forceinline__ int chains_of(const Plan3& P, const Range3& R) {
  return (R.p + R.units + P.per_chain - 1) / P.per_chain;
}

__device__ __forceinline__ void copy3(const Plan3& P, const Range3& R, uint32_t sbase, Bars3& bars, PipeWait wait) {
  Copier cp{bars.stage, sbase + OFF_STAGE, wait};
  const int last = R.c + chains_of(P, R);
  bool ok = true;
#pragma unroll 1
  for (int c = R.c; c < last && ok; ++c) {
    const int slot = slot_of(P.a.sel, P.a.sel_stride, P.a.sel_xor, c);
    if (c + 1 < last) {
      Copier::prefetch(P.op[0], c + 1);
      Copier::prefetch(P.op[1], c + 1);
      Copier::prefetch(P.op[3], c + 1);
    }
    ok = cp.operand(P.op[0], c) && cp.operand(P.op[1], c) && cp.operand(P.op[2], slot) && cp.operand(P.op[3], c);
  }
  cp.finish();
}

// Loader warps: E, T, A and B of every chain, each stored once the products have freed its
// buffer.
template <bool X3, bool FULL>
__device__ __forceinline__ void load3(const Plan3& P, const Range3& R, uint8_t* sm, Bars3& bars, PipeWait wait) {
  Loader ld{bars.stage, sm, OFF_STAGE, wait};
  const int chains = chains_of(P, R);
#pragma unroll 1
  for (int n = 0; n < chains; ++n) {
    const uint32_t prev = (uint32_t)(n - 1) & 1u;
    const int c = R.c + n, slot = slot_of(P.a.sel, P.a.sel_stride, P.a.sel_xor, c);
    if (n > 0 && !wait(&bars.free_[0], prev)) return;
    if (!ld.operand<X3, FULL, OP_KXY, OP_KXY>(P.op[0], c)) return;
    warp_publish(&bars.full[0]);
    if (!ld.operand<X3, FULL, OP_KXY, OP_YXK>(P.op[1], c)) return;
    warp_publish(&bars.full[1]);
    if (n > 0 && !wait(&bars.free_[2], prev)) return;
    if (!ld.operand<X3, FULL, OP_SITE, OP_SITE>(P.op[2], slot)) return;
    warp_publish(&bars.full[2]);
    if (n > 0 && !wait(&bars.free_[3], prev)) return;
    if (!ld.operand<X3, FULL, OP_OE, OP_YEO>(P.op[3], c)) return;
    warp_publish(&bars.full[3]);
  }
}

template <bool X3>
__device__ __forceinline__ void products3(const Plan3& P, const Range3& R, uint32_t sbase, uint32_t tmem, int s, Bars3& bars,
                                          PipeWait wait) {
  const uint32_t id_n = idesc<2>(128, 64), id_2n = idesc<2>(128, 128);
  const uint32_t id3 = X3 ? idesc<2>(128, 64) : idesc<2>(64, 32);
  const uint32_t W = sbase + OFF_W + s * 2 * SZ_W, d12 = tmem + COL_S12, d3 = tmem + COL_S3;
  const uint64_t w_sw = sdesc_sw128(W), w_sw_lo = sdesc_sw128(W + SZ_W), w_k = sdesc(W, 128, 2048);
  const uint64_t e0 = sdesc(sbase + OFF_E, 128, 512), e0_lo = sdesc(sbase + OFF_E + SZ_E, 128, 512);
  const uint64_t a0 = sdesc(sbase + OFF_A, 128, 1024), t0 = sdesc(sbase + OFF_T, 128, 512), b0 = sdesc_sw128(sbase + OFF_B);
  int m = 0, p = R.p;
  uint32_t sp = 0;  // parity of the chain's phases
  bool fresh = true;
#pragma unroll 1
  for (int u = 0; u < R.units; ++u) {
    const int t = p * P.step + s;
    if (t < P.n_at) {
      const bool chain_end = t + P.step >= P.n_at;  // this stream's last tile of the chain
      if (fresh && (!wait.one(&bars.full[0], sp) || !wait.one(&bars.full[1], sp))) return;
#pragma unroll 1
      for (int j = 0; j < P.n_bt; ++j) {
        const bool last = chain_end && j + 1 == P.n_bt, first = fresh && j == 0;
        const uint32_t je = j * (2 * SZ_E >> 4);
        tc_after_sync();
        mma_steps<X3, 2>(d12, e0 + je, e0_lo + je, t0 + t * (2 * SZ_T >> 4), 16, 16, id_n, id_2n, 0u);
        commit(&bars.acc[s]);
        if (last) commit(&bars.free_[0]);
        if (first && !wait.one(&bars.full[2], sp)) return;
        if (!wait.one(&bars.w[s], 0u)) return;
        tc_after_sync();
        mma_steps<X3, 4>(d12, w_sw, w_sw_lo, a0, 2, 16, id_n, id_2n, 0u);
        commit(&bars.acc[s]);
        if (last) commit(&bars.free_[2]);
        if (first && !wait.one(&bars.full[3], sp)) return;
        if (j == 0 && m >= 1 && !wait.one(&bars.o_free[s], (m - 1) & 1)) return;
        if (!wait.one(&bars.w[s], 1u)) return;
        tc_after_sync();
        // accumulated over the b tiles: with X3 [Y_hi ; Y_lo] x [B_hi | B_lo] (M 128, N 64),
        // else Y x B (M 64, N 32)
        const uint64_t b = b0 + j * (SZ_B >> 4);
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
          mma<2>(d3, w_k + ks * 16, b + (ks >> 2) * (B_ATOM >> 4) + (ks & 3) * 2, id3,
                 (j > 0 || ks > 0) ? 1u : 0u);
        if (last) commit(&bars.free_[3]);
      }
      commit(&bars.o_full[s]);
      ++m;
    }
    fresh = ++p == P.per_chain;
    if (fresh) {
      p = 0;
      sp ^= 1u;
    }
  }
}

// Outputs O[(r,a')][b'] of all units, by four warps (one per tensor-memory lane quarter).
template <bool X3>
__device__ __forceinline__ void output3(const Plan3& P, const Range3& R, uint8_t* sm, uint32_t tmem, Bars3& bars,
                                        PipeWait wait) {
  const int lane = threadIdx.x & 31, q = (threadIdx.x >> 5) & 3;
  const Env3Fused& a = P.a;
  const bool vec = a.sOb2 == 1 && ((a.bsO | a.sOa2 | a.sOr | a.cB2) & 3) == 0 && (reinterpret_cast<uintptr_t>(a.out) & 15) == 0;
  // with X3, lanes 0-63 hold [Y_hi B_hi | Y_hi B_lo] and lanes 64-127 [Y_lo B_hi | -]: the
  // warps of quarters 2 and 3 hand their first columns over through shared memory; an
  // M = 64 accumulator (plain BF16) keeps rows 16q..16q+15 in lanes 0-15 of quarter q
  float* buf = reinterpret_cast<float*>(sm + OFF_XCH) + (X3 ? (q & 1) * 32 : q * 16) * kRowPitch;
  float* mine = buf + (X3 ? lane : lane & 15) * kRowPitch;
  int c = R.c, p = R.p, m0 = 0, m1 = 0, k = 0;  // outputs of the two streams and of both so far
#pragma unroll 1
  for (int u = 0; u < R.units; ++u) {
#pragma unroll 1
    for (int s = 0; s < P.step; ++s) {
      const int t = p * P.step + s;
      if (t >= P.n_at) continue;
      const uint32_t taddr = tmem + s * TMEM_STREAM + COL_S3 + ((uint32_t)(q * 32) << 16);
      const uint32_t ph = (s == 0 ? m0 : m1) & 1, xph = k & 1;
      if (s == 0) ++m0; else ++m1;
      if (!wait(&bars.o_full[s], ph)) return;
      tc_after_sync();
      if (X3 && q >= 2 && k > 0 && !wait(&bars.x_free, xph ^ 1u)) return;
      if (X3 && q < 2 && !wait(&bars.x_full, xph)) return;
      ++k;
#pragma unroll 1
      for (int b0 = 0; b0 < 32; b0 += 16) {
        float v[16];
        tmem_ld16(taddr + b0, v);
        if (X3 && q < 2) {
          float lo[16];
          tmem_ld16(taddr + 32 + b0, lo);
          add_row16(mine + b0, lo);
#pragma unroll
          for (int e = 0; e < 16; ++e) v[e] += lo[e];
        }
        if (X3 || lane < 16) put_row16(mine + b0, v);
      }
      tc_before_sync();
      __syncwarp();
      if (lane == 0) {
        if (X3 && q >= 2) mbar_arrive(&bars.x_full);
        mbar_arrive(&bars.o_free[s]);
      }
      if (X3 && q >= 2) continue;
      // rows (r, a') to global memory along b'
      const int r0 = X3 ? q * 4 : q * 2;
      store_rows(buf, a.out + c * a.bsO + r0 * a.sOr + t * kAT * a.sOa2, a.sOr, a.sOa2, a.sOb2, min(X3 ? 4 : 2, a.Dr - r0),
                 min(kAT, a.cT2 - t * kAT), a.cB2, vec);
      __syncwarp();
      if (X3 && lane == 0) mbar_arrive(&bars.x_free);
    }
    if (++p == P.per_chain) {
      p = 0;
      ++c;
    }
  }
}

template <bool X3>
__device__ __forceinline__ void drain3(const Plan3& P, const Range3& R, uint8_t* sm, uint32_t tmem, int s, Bars3& bars,
                                       PipeWait wait) {
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) & 7, q = warp & 3, h = warp >> 2;
  const uint32_t row = tmem + COL_S12 + h * 32 + ((uint32_t)(q * 32) << 16);
  uint8_t* W = sm + OFF_W + s * 2 * SZ_W;
  const int m1 = q * 32 + lane, hi3 = m1 >> 3, lo3 = m1 & 7;
  int p = R.p;
#pragma unroll 1
  for (int u = 0; u < R.units; ++u) {
    const int n = p * P.step + s < P.n_at ? 2 * P.n_bt : 0;
    // per b tile: S1's row (b,l) -> S2 rows (b,a'), chunk l (swizzled); S2's row (b,a') -> S3
    // rows (r,a'), chunk b
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      if (!wait(&bars.acc[s], (uint32_t)i & 1u)) return;
      tc_after_sync();
      const bool x = (i & 1) == 0;
      drain_rows<X3>(row, W + (x ? (hi3 * 8 + h * 4) << 7 : (h * 64 + hi3) * 128 + lo3 * 16), x ? 128u : 2048u, x, lo3,
                     h * 4);
      warp_publish(&bars.w[s]);
    }
    if (++p == P.per_chain) p = 0;
  }
}

// Common end of a product-issuing thread: whatever it issued completes (bounded by at
// least the default budget) before the tensor memory is released.
__device__ __forceinline__ void finish_products(uint64_t* fin, long long budget) {
  commit(fin);
  wait_parity(fin, 0u, budget > kDefaultWaitCycles ? budget : kDefaultWaitCycles);
}

template <bool X3, bool FULL>
__global__ void __launch_bounds__(kPipeThreads, 1) env3_fused_kernel(const __grid_constant__ Plan3 P, unsigned* status) {
  extern __shared__ __align__(1024) uint8_t sm[];  // the swizzled tiles lie on 1 KB boundaries
  __shared__ __align__(8) Bars3 bars;
  __shared__ uint32_t tmem_base;
  __shared__ PipeCtl ctl;
  const Range3 R = range_of(P);
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    staging_init(bars.stage);
#pragma unroll 1
    for (int i = 0; i < 4; ++i) {
      mbar_init(&bars.full[i], kPipeLoadWarps);
      mbar_init(&bars.free_[i], P.streams);
    }
#pragma unroll 1
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars.acc[i], 1);
      mbar_init(&bars.w[i], kPipeDrainWarps);
      mbar_init(&bars.o_full[i], 1);
      mbar_init(&bars.o_free[i], 4);
      mbar_init(&bars.fin[i], 1);
    }
    mbar_init(&bars.x_full, 2);
    mbar_init(&bars.x_free, 2);
    mbar_fence_init();
    ctl.abort = 0;
    ctl.status = status;
    ctl.budget = P.a.wait_cycles > 0 ? P.a.wait_cycles : kDefaultWaitCycles;
  }
  if (warp == 0) tmem_alloc(&tmem_base, TMEM_COLS);
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  after_previous();
  const uint32_t tmem = tmem_base;
  const PipeWait wait{&ctl};
  switch (pipe_role(warp)) {
    case ROLE_DRAIN: {
      const int s = warp / kPipeDrainWarps;
      if (s < P.streams) drain3<X3>(P, R, sm, tmem + s * TMEM_STREAM, s, bars, wait);
      break;
    }
    case ROLE_LOAD: load3<X3, FULL>(P, R, sm, bars, wait); break;
    case ROLE_OUT: output3<X3>(P, R, sm, tmem, bars, wait); break;
    case ROLE_COPY:
      if ((threadIdx.x & 31) == 0) copy3(P, R, smem_u32(sm), bars, wait);
      break;
    case ROLE_PRODUCTS: {
      const int s = warp & 1;
      if ((threadIdx.x & 31) == 0 && s < P.streams) {
        products3<X3>(P, R, smem_u32(sm), tmem + s * TMEM_STREAM, s, bars, wait);
        finish_products(&bars.fin[s], ctl.budget);
      }
      break;
    }
  }
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

template <bool X3, bool FULL>
cudaError_t launch(const Plan3& P, int grid, unsigned* status, cudaStream_t st) {
  static SmemLimit limit{SMEM_BYTES, false};
  return launch_large(limit, true, env3_fused_kernel<X3, FULL>, grid, kPipeThreads, SMEM_BYTES, st, P, status);
}

// ------------------------------------------------------------ optimal site of the fit
// Fused optimal-site contraction of the variational fit (App. B): per unit (one chain) the
// two streams take the two tiles of 16 values of the new MPS's left bond v and walk the
// a' tiles of 8:
//   S1  X[(v,l)][(a',u)]    = sum_a     L(a,l,v) T(a,u,a')          M 128, N 64, K 32
//   S2  Y[(v,a')][(r,d)]    = sum_(l,u) X A_s(l,u,r,d)              M 128, N 64, K 64
//   S3  O[(v,d)][v']       += sum_(a',r) Y R(a',r,v')               M 128, N 32, K 64
// S3 accumulates over the a' tiles.  S1's drain is the three-line step's; S2's re-indexes
// each row (v,a') into rows (v,d) and K chunk a' of S3's operand, in the 128-byte swizzled
// layout (the eight lanes of one row group write eight different bank groups).  Split BF16
// products are merged as in the three-line step.
constexpr int kPV = 16;  // v per tile
constexpr uint32_t P_SZ_R = 32 * 128;                                  // S3 B: 32 rows x 64 K
constexpr uint32_t P_OFF_L = OFF_W + 2 * 2 * SZ_W;                     // [v tile], S1 A
constexpr uint32_t P_OFF_T = P_OFF_L + 2 * 2 * SZ_E;                   // [a' tile], S1 B
constexpr uint32_t P_OFF_R = P_OFF_T + 4 * 2 * SZ_T;                   // [a' tile]
constexpr uint32_t P_OFF_A = P_OFF_R + 4 * 2 * P_SZ_R;
constexpr uint32_t P_OFF_STAGE = P_OFF_A + 2 * SZ_A;
constexpr uint32_t P_OFF_BUF = P_OFF_STAGE + 2 * kStageBytes;            // output rows, 32 per warp
constexpr uint32_t P_SMEM_BYTES = P_OFF_BUF + 4 * 32 * kRowPitch * 4;
static_assert(P_SMEM_BYTES + 1024 <= 232448, "the optimal-site CTA must fit an SM");

struct BarsP {
  Staging stage;
  uint64_t full[4];                        // loaders -> products, once per unit: L, T, A, R
  uint64_t free_[4];                       // products -> loaders, one arrival per stream and unit ([0]: L and T)
  uint64_t acc[2], w[2];                   // products <-> drain
  uint64_t o_full[2], o_free[2], fin[2];   // products <-> output
};

// Units: (chain, v tiles of `step` streams), as in the three-line step.
struct PlanP {
  Proj3Fused a;
  PipeOp op[4];  // L, T, A, R
  int n_at, n_vt, step, per_chain, streams;
  int share, rest;
};
PlanP planp(const Proj3Fused& a, int sms, int& grid) {
  PlanP P;
  P.a = a;
  P.n_at = (a.cT2 + kAT - 1) / kAT;
  P.n_vt = (a.cV + kPV - 1) / kPV;
  P.step = (long long)a.batch * P.n_vt <= sms ? 1 : 2;
  P.per_chain = (P.n_vt + P.step - 1) / P.step;
  P.streams = P.step < P.n_vt ? P.step : P.n_vt;
  const int units = a.batch * P.per_chain;
  grid = units < sms ? units : sms;
  P.share = units / grid;
  P.rest = units % grid;
  PipeOp &L = P.op[0], &T = P.op[1], &A = P.op[2], &Rt = P.op[3];
  auto set = [](PipeOp& o, int kind, const float* base, long long chain, int n0, long long s0, int n1, long long s1, int n2,
                long long s2) {
    o.kind = kind; o.base = base; o.chain = chain;
    o.n[0] = n0; o.s[0] = (int)s0; o.n[1] = n1; o.s[1] = (int)s1; o.n[2] = n2; o.s[2] = (int)s2;
  };
  set(L, OP_KXY, a.L, a.bsL, a.cT, a.sLa, a.Dl, a.sLl, a.cV, a.sLv);
  L.dst = P_OFF_L; L.tile = 2 * SZ_E; L.lo = SZ_E; L.ys = 4;
  set(T, OP_KXY, a.T, a.bsT, a.cT, a.sTa, a.Du, a.sTu, a.cT2, a.sTa2);
  T.dst = P_OFF_T; T.tile = 2 * SZ_T; T.lo = SZ_T; T.ys = 3;
  set(A, OP_SITE, a.A, a.ssA, a.Dl, a.sAl, a.Du, a.sAu, a.Dr, a.sAr);
  A.n[3] = a.Dd; A.s[3] = (int)a.sAd;
  A.dst = P_OFF_A; A.lo = SZ_A;
  set(Rt, OP_OE, a.R, a.bsR, a.cT2, a.sRa, a.Dr, a.sRr, a.cV2, a.sRv);
  Rt.dst = P_OFF_R; Rt.tile = 2 * P_SZ_R; Rt.lo = P_SZ_R;
  for (PipeOp& o : P.op) finish_operand(o);
  return P;
}
struct RangeP {
  int first, units;
};

__device__ __forceinline__ void copyp(const PlanP& P, const RangeP& U, uint32_t sbase, BarsP& bars, PipeWait wait) {
  Copier cp{bars.stage, sbase + P_OFF_STAGE, wait};
  bool ok = true;
#pragma unroll 1
  for (int u = U.first; u < U.first + U.units && ok; ++u) {
    const int c = u / P.per_chain, slot = slot_of(P.a.sel, P.a.sel_stride, 0, c);
    const int next = (u + 1) / P.per_chain;
    if (next > c && u + 1 < U.first + U.units) {
      Copier::prefetch(P.op[0], next);
      Copier::prefetch(P.op[1], next);
      Copier::prefetch(P.op[3], next);
    }
    ok = cp.operand(P.op[0], c) && cp.operand(P.op[1], c) && cp.operand(P.op[2], slot) && cp.operand(P.op[3], c);
  }
  cp.finish();
}

template <bool X3>
__device__ __forceinline__ void productsp(const PlanP& P, const RangeP& U, uint32_t sbase, uint32_t tmem, int s, BarsP& bars,
                                          PipeWait wait) {
  const uint32_t id_n = idesc<2>(128, 64), id_2n = idesc<2>(128, 128);
  const uint32_t id3_n = idesc<2>(128, 32), id3_2n = idesc<2>(128, 64);
  const uint32_t W = sbase + OFF_W + s * 2 * SZ_W, d12 = tmem + COL_S12, d3 = tmem + COL_S3;
  const uint64_t w = sdesc_sw128(W), w_lo = sdesc_sw128(W + SZ_W);
  const uint64_t l0 = sdesc(sbase + P_OFF_L, 128, 512), t0 = sdesc(sbase + P_OFF_T, 128, 512),
                 a0 = sdesc(sbase + P_OFF_A, 128, 1024), r0 = sdesc(sbase + P_OFF_R, 128, 1024);
#pragma unroll 1
  for (int n = 0; n < U.units; ++n) {
    const uint32_t ph = (uint32_t)n & 1u;
    if (!wait.one(&bars.full[0], ph) || !wait.one(&bars.full[1], ph)) return;
    const uint64_t l = l0 + ((U.first + n) % P.per_chain * P.step + s) * (2 * SZ_E >> 4);
#pragma unroll 1
    for (int t = 0; t < P.n_at; ++t) {
      const bool last = t + 1 == P.n_at;
      tc_after_sync();
      mma_steps<X3, 2>(d12, l, l + (SZ_E >> 4), t0 + t * (2 * SZ_T >> 4), 16, 16, id_n, id_2n, 0u);
      commit(&bars.acc[s]);
      if (last) commit(&bars.free_[0]);
      if (t == 0 && !wait.one(&bars.full[2], ph)) return;
      if (!wait.one(&bars.w[s], 0u)) return;
      tc_after_sync();
      mma_steps<X3, 4>(d12, w, w_lo, a0, 2, 16, id_n, id_2n, 0u);
      commit(&bars.acc[s]);
      if (last) commit(&bars.free_[2]);
      if (t == 0 && (!wait.one(&bars.full[3], ph) || (n > 0 && !wait.one(&bars.o_free[s], ph ^ 1u)))) return;
      if (!wait.one(&bars.w[s], 1u)) return;
      tc_after_sync();
      mma_steps<X3, 4>(d3, w, w_lo, r0 + t * (2 * P_SZ_R >> 4), 2, 16, id3_n, id3_2n, t > 0 ? 1u : 0u);
    }
    commit(&bars.free_[3]);
    commit(&bars.o_full[s]);
  }
}

// Outputs Y(v,d,v') of all units.
template <bool X3>
__device__ __forceinline__ void outputp(const PlanP& P, const RangeP& U, uint8_t* sm, uint32_t tmem, BarsP& bars,
                                        PipeWait wait) {
  const int lane = threadIdx.x & 31, q = (threadIdx.x >> 5) & 3;
  const Proj3Fused& a = P.a;
  const bool vec = a.sOv2 == 1 && ((a.bsO | a.sOv | a.sOd | a.cV2) & 3) == 0 && (reinterpret_cast<uintptr_t>(a.out) & 15) == 0;
  float* buf = reinterpret_cast<float*>(sm + P_OFF_BUF) + q * 32 * kRowPitch;
  float* mine = buf + lane * kRowPitch;
#pragma unroll 1
  for (int n = 0; n < U.units; ++n) {
    const int u = U.first + n;
#pragma unroll 1
    for (int s = 0; s < P.streams; ++s) {
      const uint32_t taddr = tmem + s * TMEM_STREAM + COL_S3 + ((uint32_t)(q * 32) << 16);
      if (!wait(&bars.o_full[s], n & 1)) return;
      tc_after_sync();
#pragma unroll 1
      for (int b0 = 0; b0 < 32; b0 += 16) {
        float v[16];
        tmem_ld16(taddr + b0, v);
        if constexpr (X3) {
          float w[16];
          tmem_ld16(taddr + 32 + b0, w);
#pragma unroll
          for (int e = 0; e < 16; ++e) v[e] += w[e];
        }
        put_row16(mine + b0, v);
      }
      tc_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars.o_free[s]);
      // rows (v, d) to global memory along v'
      const int v0 = (u % P.per_chain * P.step + s) * kPV + q * 4;
      store_rows(buf, a.out + u / P.per_chain * a.bsO + v0 * a.sOv, a.sOv, a.sOd, a.sOv2, min(4, a.cV - v0), a.Dd, a.cV2,
                 vec);
      __syncwarp();
    }
  }
}

// Loader warps: L, T, A and R of every unit.
template <bool X3, bool FULL>
__device__ __forceinline__ void loadp(const PlanP& P, const RangeP& U, uint8_t* sm, BarsP& bars, PipeWait wait) {
  Loader ld{bars.stage, sm, P_OFF_STAGE, wait};
#pragma unroll 1
  for (int n = 0; n < U.units; ++n) {
    const int c = (U.first + n) / P.per_chain, slot = slot_of(P.a.sel, P.a.sel_stride, 0, c);
    const uint32_t prev = (uint32_t)(n - 1) & 1u;
    if (n > 0 && !wait(&bars.free_[0], prev)) return;
    if (!ld.operand<X3, FULL, OP_KXY, OP_KXY>(P.op[0], c)) return;
    warp_publish(&bars.full[0]);
    if (!ld.operand<X3, FULL, OP_KXY, OP_KXY>(P.op[1], c)) return;
    warp_publish(&bars.full[1]);
    if (n > 0 && !wait(&bars.free_[2], prev)) return;
    if (!ld.operand<X3, FULL, OP_SITE, OP_SITE>(P.op[2], slot)) return;
    warp_publish(&bars.full[2]);
    if (n > 0 && !wait(&bars.free_[3], prev)) return;
    if (!ld.operand<X3, FULL, OP_OE, OP_OE>(P.op[3], c)) return;
    warp_publish(&bars.full[3]);
  }
}

template <bool X3>
__device__ __forceinline__ void drainp(const PlanP& P, const RangeP& U, uint8_t* sm, uint32_t tmem, int s, BarsP& bars,
                                       PipeWait wait) {
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) & 7, q = warp & 3, h = warp >> 2;
  const uint32_t row = tmem + COL_S12 + ((uint32_t)(q * 32) << 16);
  uint8_t* W = sm + OFF_W + s * 2 * SZ_W;
  const int m1 = q * 32 + lane, hi3 = m1 >> 3, lo3 = m1 & 7;
  const int tiles = U.units * P.n_at;
#pragma unroll 1
  for (int i = 0; i < tiles; ++i) {
    if (!wait(&bars.acc[s], 0u)) return;
    tc_after_sync();
    // S1: row (v,l) -> S2 rows (v,a'), chunk l (swizzled)
    drain_rows<X3>(row + h * 32, W + ((hi3 * 8 + h * 4) << 7), 128u, true, lo3, h * 4);
    warp_publish(&bars.w[s]);
    if (!wait(&bars.acc[s], 1u)) return;
    tc_after_sync();
    // S2: row (v,a') -> S3 rows (v,d) for d in [4h, 4h+4), chunk a' (swizzled)
    float x[8][4];  // [r][d - 4h]
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      float v[16];  // columns (r, d) with r in [2p, 2p+2)
      load_acc16<X3>(row + p * 16, v);
#pragma unroll
      for (int rr = 0; rr < 2; ++rr)
#pragma unroll
        for (int dd = 0; dd < 4; ++dd) x[p * 2 + rr][dd] = h ? v[rr * 8 + 4 + dd] : v[rr * 8 + dd];
    }
#pragma unroll
    for (int dd = 0; dd < 4; ++dd) {
      float col[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) col[r] = x[r][dd];
      put_split8<X3>(W + sw128_chunk_off(hi3 * 8 + h * 4 + dd, lo3), col, SZ_W);
    }
    warp_publish(&bars.w[s]);
  }
}

template <bool X3, bool FULL>
__global__ void __launch_bounds__(kPipeThreads, 1) proj3_fused_kernel(const __grid_constant__ PlanP P, unsigned* status) {
  extern __shared__ __align__(1024) uint8_t sm[];  // the swizzled tiles lie on 1 KB boundaries
  __shared__ __align__(8) BarsP bars;
  __shared__ uint32_t tmem_base;
  __shared__ PipeCtl ctl;
  const int bi = blockIdx.x;
  const RangeP U{bi * P.share + min(bi, P.rest), P.share + (bi < P.rest ? 1 : 0)};
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    staging_init(bars.stage);
#pragma unroll 1
    for (int i = 0; i < 4; ++i) {
      mbar_init(&bars.full[i], kPipeLoadWarps);
      mbar_init(&bars.free_[i], P.streams);
    }
#pragma unroll 1
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars.acc[i], 1);
      mbar_init(&bars.w[i], kPipeDrainWarps);
      mbar_init(&bars.o_full[i], 1);
      mbar_init(&bars.o_free[i], 4);
      mbar_init(&bars.fin[i], 1);
    }
    mbar_fence_init();
    ctl.abort = 0;
    ctl.status = status;
    ctl.budget = P.a.wait_cycles > 0 ? P.a.wait_cycles : kDefaultWaitCycles;
  }
  if (warp == 0) tmem_alloc(&tmem_base, TMEM_COLS);
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  after_previous();
  const uint32_t tmem = tmem_base;
  const PipeWait wait{&ctl};
  switch (pipe_role(warp)) {
    case ROLE_DRAIN: {
      const int s = warp / kPipeDrainWarps;
      if (s < P.streams) drainp<X3>(P, U, sm, tmem + s * TMEM_STREAM, s, bars, wait);
      break;
    }
    case ROLE_LOAD: loadp<X3, FULL>(P, U, sm, bars, wait); break;
    case ROLE_OUT: outputp<X3>(P, U, sm, tmem, bars, wait); break;
    case ROLE_COPY:
      if ((threadIdx.x & 31) == 0) copyp(P, U, smem_u32(sm), bars, wait);
      break;
    case ROLE_PRODUCTS: {
      const int s = warp & 1;
      if ((threadIdx.x & 31) == 0 && s < P.streams) {
        productsp<X3>(P, U, smem_u32(sm), tmem + s * TMEM_STREAM, s, bars, wait);
        finish_products(&bars.fin[s], ctl.budget);
      }
      break;
    }
  }
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

template <bool X3, bool FULL>
cudaError_t launch_proj3(const PlanP& P, int grid, unsigned* status, cudaStream_t st) {
  static SmemLimit limit{P_SMEM_BYTES, false};
  return launch_large(limit, true, proj3_fused_kernel<X3, FULL>, grid, kPipeThreads, P_SMEM_BYTES, st, P, status);
}

bool all_full(const PipeOp (&op)[4]) {
  for (const PipeOp& o : op)
    if (!full_operand(o)) return false;
  return true;
}

// Whether the pipeline is faster than one tile per CTA with bonds below the maxima (with full bonds it
// is at every number of chains: 1 chain 10.3 / 9.7 us, one tile per CTA / pipeline, split BF16, 38
// 10.8 / 10.2, 50 14.2 / 12.8, 512 90.9 / 52.8).  With one a' tile per chain a stream idles (Dc 8, D 2,
// 1024 chains 29.2 / 43.5), and few tiles leave nothing to overlap.  Above that both forms run
// in whole rounds of CTAs, so which is faster changes back and forth with the number of chains
// (Dc 24, D 6, 152 chains 21.3 / 17.6, 184 25.9 / 30.3, 256 37.1 / 30.4, 2048 261 / 188; Dc 16, D 4 in
// BF16 640 23.8 / 27.1): the rule compares estimates (us), fitted to 219 launches of bonds up to 32
// and 8 and 150 to 2048 chains (rms error 4 % for one tile per CTA, 7 % for the pipeline).  One tile per
// CTA: by rounds of two CTAs per SM and, if the last round needs one only, that.  Pipeline: by
// a CTA's chains and tiles.  Of the 219, two sizes remain that the choice makes slower than one tile
// per CTA by more than 3 %, by 7 and 11 %.
bool pipeline_pays(const Plan3& P, int sms, bool split) {
  const Env3Fused& a = P.a;
  const long long tiles = (long long)a.batch * P.n_at;
  if (P.n_at < 2 || tiles * P.n_bt * 152 < 1100LL * sms) return false;
  const double rounds = (double)(tiles / (2 * sms)), last = (double)(tiles % (2 * sms)), n = P.n_bt;
  const double whole = rounds + (last > sms), half = last > 0 && last <= sms;
  const double units = (double)(P.share + (P.rest > 0)) * P.align, chains = ceil(units / P.per_chain);
  const double v = 1e-4 * (a.cT * (a.Dl * a.cB + a.Du * a.cT2) + a.Dl * a.Du * a.Dr * a.Dd + a.cB * a.Dd * a.cB2);  // operands
  const double per_tile = split ? 2.2 + whole * (3.4 + 3.85 * n + 0.76 * v) + half * (3.5 * n - 1.1)
                                : 2.9 + whole * (2.2 + 2.65 * n + 0.84 * v) + half * (1.45 * n + 0.25);
  const double pipe = split ? 4.7 + chains * (4.1 + 1.9 * v) + 1.8 * units * n : 4.9 + chains * (2.9 + 1.2 * v) + 1.35 * units * n;
  return 1.03 * pipe < per_tile;
}

}  // namespace

cudaError_t env3_fused(const Env3Fused& a, bool split, unsigned* status, cudaStream_t st) {
  if (g_dry_run || a.batch <= 0) return cudaSuccess;
  if (!env3_fused_fits(a.cT, a.cB, a.cT2, a.cB2, a.Dl, a.Dr, a.Du, a.Dd)) return cudaErrorInvalidValue;
  if ((long long)a.batch * 4 > 0x7fffffffLL) return cudaErrorInvalidValue;
  int grid = 0, sms = 0;
  PV_CUDA(sm_count(&sms));
  const Plan3 P = plan3(a, sms, grid);
  const bool full = all_full(P.op);
  if (!full && !pipeline_pays(P, sms, split)) return env3_tiles(a, split, sms, status, st);
  if (full) return split ? launch<true, true>(P, grid, status, st) : launch<false, true>(P, grid, status, st);
  return split ? launch<true, false>(P, grid, status, st) : launch<false, false>(P, grid, status, st);
}

cudaError_t proj3_fused(const Proj3Fused& a, bool split, unsigned* status, cudaStream_t st) {
  if (g_dry_run || a.batch <= 0) return cudaSuccess;
  if (!proj3_fused_fits(a)) return cudaErrorInvalidValue;
  if ((long long)a.batch * 2 > 0x7fffffffLL) return cudaErrorInvalidValue;
  int grid = 0, sms = 0;
  PV_CUDA(sm_count(&sms));
  const PlanP P = planp(a, sms, grid);
  // With one or two a' tiles there is too little per unit to overlap.  Measured, one tile per
  // CTA / pipeline, split BF16: full bonds 16 chains 22.5 / 18.3 us, 512 chains 98.8 / 66.9;
  // Dc 16, D 4 (two a' tiles) 64 chains 14.3 / 14.3, 512 chains 32.0 / 33.2.
  // One tile of v leaves a stream idle, which costs where each chain would still have a CTA in the
  // one round of two per SM: cV 12, 192 chains 20.0 / 22.4; 152 chains 18.9 / 15.3, 580 chains 30.2 / 28.6.
  if (P.n_at < 3 || (P.n_vt == 1 && a.batch > sms && a.batch <= 2 * sms)) return proj3_tiles(a, split, sms, status, st);
  if (all_full(P.op))
    return split ? launch_proj3<true, true>(P, grid, status, st) : launch_proj3<false, true>(P, grid, status, st);
  return split ? launch_proj3<true, false>(P, grid, status, st) : launch_proj3<false, false>(P, grid, status, st);
}

}  // namespace pv
