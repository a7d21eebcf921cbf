// Fused four-line column step at full bonds (Dc 32, D 8, b-major environments) as a pipeline
// of three streams: the products, operand layouts and summation order of fused_env4.cu, roles
// and hand-overs as in fused_pipe.cuh.
//
// Per tile of 8 values of a' and 2 of the incoming bottom bond b:
//   S1  X[(b,l2,l1)][(a',u1)]   = sum_a       E(a,l1,l2,b) T(a,u1,a')     M 128, N 64, K 32
//   S2  Y[(l2,b,a')][(r1,d1)]   = sum_(l1,u1) X a1(l1,u1,r1,d1)           M 128, N 64, K 64
//   S3  Z[(b,r1,a')][(r2,d2)]   = sum_(l2,d1) Y a2(l2,d1,r2,d2)           M 128, N 64, K 64
//   S4  O[(r1,r2,a')][b']      += sum_(b,d2)  Z B(b,d2,b')                M 512, N 32, K 16
// A unit is a chain and one a' tile; its 16 b tiles go to the three streams in turn, so that
// three tiles are in flight, and S4 of all of them accumulates into one region of tensor
// memory, in the order of b.  That region (128 columns) and one of 128 columns for each
// stream's S1-S3 fill the tensor memory; a1, a2 and B are converted once per chain.
//
// Bound (split format): shared memory.  A tile's products read their operands for ~1,770 cycles
// (128 B/cycle), its drains write for ~770, E's staging and conversion take ~400; measured
// 3,760 cycles per tile with the data pipe 84 % busy (ncu: 40 % products, 44 % loads and
// stores), the rest hand-over latency (drain ~1,100 cycles, products ~1,600, beside the two
// other streams).  Two streams, each with an S4 region of its own and E shared by two a'
// tiles, were at 4,150 cycles: too few tiles in flight.  Measured, one-tile-per-CTA kernel ->
// this: 1 chain 61 -> 39 us, 76 chains 87 -> 72, 128 chains 165 -> 130, 512 chains 566 -> 438
// (236 TFLOP/s), 1001 chains 1080 -> 831; plain BF16 1 chain 40 -> 30, 512 chains 350 -> 293
// (there the loaders set the pace).
#include <new>

#include "fused.cuh"
#include "fused_pipe.cuh"

namespace pv {
namespace {

using namespace tc;

constexpr int kAT = 8, kBT = 2, kNB = 32 / kBT;

constexpr int kStreams = 3, kDrainWarps = 8, kLoadWarps = 4;  // drain warps per stream
constexpr int kThreads = (kStreams * kDrainWarps + kLoadWarps + 1 + kStreams) * 32;

constexpr uint32_t SZ_W = 128 * 128, OFF_W = 0;                     // [stream] X (swizzled), Y or Z
constexpr uint32_t SZ_E = 128 * 64, OFF_E = OFF_W + kStreams * 2 * SZ_W;  // [tile parity]
constexpr uint32_t SZ_T = 64 * 64, OFF_T = OFF_E + 4 * SZ_E;        // [unit parity]
constexpr uint32_t SZ_A = 64 * 128, OFF_A1 = OFF_T + 4 * SZ_T, OFF_A2 = OFF_A1 + 2 * SZ_A;
constexpr uint32_t SZ_B = 32 * 32, OFF_B = OFF_A2 + 2 * SZ_A;       // [b tile], hi then lo
constexpr uint32_t kPiece = 8192, OFF_STAGE = OFF_B + kNB * 2 * SZ_B;
constexpr uint32_t SMEM_BYTES = OFF_STAGE + 2 * kPiece;
constexpr uint32_t TMEM_COLS = 512, COL_S4 = 0, COL_S123 = 128;     // S1-S3: 128 columns per stream
static_assert(SMEM_BYTES + 1024 <= 232448 && kThreads == 1024, "the four-line CTA must fit an SM");

struct Bars4 {
  uint64_t full[2], empty[2];                     // staging buffers: copy <-> loaders
  uint64_t t_full[2], t_free[2];                  // per unit
  uint64_t e_full[kStreams], e_free[2];           // per tile: of the stream; of the buffer
  uint64_t a_full[2], a_free[2], b_full, b_free;  // per chain: a1, a2; B
  uint64_t acc[kStreams], w[kStreams], fin[kStreams];  // products <-> drain
  uint64_t s4[kStreams], o_free;                  // S4 of a tile complete; results of a unit read
};

// Units (chain, a' tile), a contiguous range per CTA; operands in bulk pieces of 8 KB.
struct Plan4 {
  Env4Fused a;
  PipeOp T, A1, A2, B;
  int share, rest;
};
struct Range4 {
  int c, p, units;  // first chain, its first a' tile
};

// Conversions of an 8 KB piece by the four loader warps (w).  E: one b, [a][l1][l2], rows
// b*64 + l2*8 + l1, K = a; lanes over l1 and half of l2, l2 shifted by four where l1 >= 4:
// 32 different banks.
template <bool X3>
__device__ __forceinline__ void convert_e(uint32_t src, int b, uint8_t* dst) {
  const int lane = threadIdx.x & 31, kc = (threadIdx.x >> 5) & 3, l1 = lane & 7;
  float v[2][8];
  uint32_t off[2];
#pragma unroll
  for (int n = 0; n < 2; ++n) {
    const int l2 = ((lane >> 3) + 4 * (l1 >> 2) + 4 * n) & 7;
    const uint32_t s = src + (kc * 8 * 64 + l1 * 8 + l2) * 4;
#pragma unroll
    for (int e = 0; e < 8; ++e) v[n][e] = lds(s + e * 256);
    off[n] = kmajor_off(b * 64 + l2 * 8 + l1, kc * 8, 4);
  }
#pragma unroll
  for (int n = 0; n < 2; ++n) put_split8<X3>(dst + off[n], v[n], SZ_E);
}
// T, rows a'*8 + u, K = a: the tile itself ([a'][u][a]), or piece kc of [a][u][a'].
template <bool X3>
__device__ __forceinline__ void convert_t(uint32_t src, int kc, bool rows, int tile, uint8_t* dst) {
  const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) & 3;
  float v[8];
  if (rows) {
    const int u = lane & 7, h = lane & 1, k = (w + (u >> 1)) & 3;
#pragma unroll 1
    for (int n = 0; n < 2; ++n) {
      const int y = (lane >> 3) + 4 * n;
      const uint32_t s = src + (y * 256 + u * 32 + k * 8) * 4;
      const float4 f = lds4(s + 16 * h), g = lds4(s + 16 - 16 * h);
      const float4 a = h ? g : f, b = h ? f : g;
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
      v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
      put_split8<X3>(dst + kmajor_off(y * 8 + u, k * 8, 4), v, SZ_T);
    }
  } else if ((w >> 1) == (kc & 1)) {
    const int u = (lane >> 3) + 4 * (w & 1), y = lane & 7;
    const uint32_t s = src + (u * 32 + tile * 8 + y) * 4;
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = lds(s + e * 1024);
    put_split8<X3>(dst + kmajor_off(y * 8 + u, kc * 8, 4), v, SZ_T);
  }
}
// Site tensor, half p of its outermost index (l, or r of a mirrored view): rows r*8 + d, K = (l, u).
template <bool X3>
__device__ __forceinline__ void convert_a(uint32_t src, int p, bool mirrored, uint8_t* dst) {
  const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) & 3, d = lane & 7, out = 4 * p + w;
#pragma unroll 1
  for (int n = 0; n < 2; ++n) {
    const int in = (lane >> 3) + 4 * n;
    const uint32_t s = src + (w * 512 + in * 8 + d) * 4;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = lds(s + e * 256);
    put_split8<X3>(dst + kmajor_off((mirrored ? out : in) * 8 + d, (mirrored ? in : out) * 8, 8), v, SZ_A);
  }
}
// B, piece p (8 values of its outermost index, b or b'): rows b', K = (b, d2), b tiles of 2.
template <bool X3>
__device__ __forceinline__ void convert_b(uint32_t src, int p, bool rows, uint8_t* dst) {
  const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) & 3;
#pragma unroll 1
  for (int n = 0; n < 2; ++n) {
    const int i = 2 * w + n, b = rows ? lane : 8 * p + i, y = rows ? 8 * p + i : lane;
    const uint32_t s = src + (i * 256 + lane) * 4;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = lds(s + e * 128);
    put_split8<X3>(dst + (b >> 1) * 2 * SZ_B + kmajor_off(y, (b & 1) * 8, 2), v, SZ_B);
  }
}
__device__ __forceinline__ int slot_of(const int8_t* sel, long long stride, int flip, int c) {
  return sel ? ((sel[c * stride] < 0) ? 1 : 0) ^ flip : 0;
}

__device__ __forceinline__ void prefetch_l2(const float* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ void copy4(const Plan4& P, const Range4& R, uint32_t stage, Bars4& bars, PipeWait wait) {
  const Env4Fused& a = P.a;
  int c = R.c, p = R.p, n = 0;  // n: pieces issued
  auto pieces = [&](const float* src, int count) {
#pragma unroll 1
    for (int i = 0; i < count; ++i, ++n) {
      const int k = n & 1;
      if (n >= 2 && !wait.one(&bars.empty[k], ((n >> 1) - 1) & 1)) return false;
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&bars.full[k])), "r"(kPiece)
                   : "memory");
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                       stage + k * kPiece),
                   "l"(src + i * (kPiece / 4)), "r"(kPiece), "r"(smem_u32(&bars.full[k]))
                   : "memory");
    }
    return true;
  };
  const bool t_rows = P.T.kind == OP_YXK;
  bool ok = true;
#pragma unroll 1
  for (int u = 0; u < R.units && ok; ++u) {
    const bool fresh = u == 0 || p == 0;
    const float* E = a.E + c * a.bsE;
    const float* T = a.T + c * a.bsT;
    if (u == 0) prefetch_l2(E, 8 * kPiece);
    ok = t_rows ? pieces(T + p * (kPiece / 4), 1) : pieces(T, 4);
#pragma unroll 1
    for (int j = 0; j < kNB && ok; ++j) {
      // device memory is asked four tiles ahead (the staging buffers hold half a tile each)
      if (fresh && j + 4 < kNB) prefetch_l2(E + (j + 4) * (kPiece / 2), 2 * kPiece);
      if (p == 3 && u + 1 < R.units) {
        if (j < 4) prefetch_l2(E + a.bsE + j * (kPiece / 2), 2 * kPiece);
        if (j == 4) prefetch_l2(T + a.bsT, 4 * kPiece);
        if (j == 5) prefetch_l2(a.B + (c + 1) * a.bsB, 4 * kPiece);
      }
      ok = pieces(E + j * (kPiece / 2), 2);
      if (j == 0 && fresh && ok)
        ok = pieces(a.A1 + slot_of(a.sel1, a.sel_stride, a.xor1, c) * a.ss1, 2) &&
             pieces(a.A2 + slot_of(a.sel2, a.sel_stride, a.xor2, c) * a.ss2, 2) && pieces(a.B + c * a.bsB, 4);
    }
    if (++p == 4) {
      p = 0;
      ++c;
    }
  }
  // whatever was issued lands (with a limit) before the shared memory is given up
#pragma unroll 1
  for (int k = max(0, n - 2); k < n; ++k) wait_parity(&bars.full[k & 1], (k >> 1) & 1, kDefaultWaitCycles);
}

template <bool X3>
__device__ __forceinline__ void load4(const Plan4& P, const Range4& R, uint8_t* sm, Bars4& bars, PipeWait wait) {
  const uint32_t stage = smem_u32(sm) + OFF_STAGE;
  int n = 0, p = R.p;        // pieces taken; a' tile
  int chain = 0, s_e = 0;    // chains begun; stream of the next b tile
  auto take = [&]() { return wait(&bars.full[n & 1], (n >> 1) & 1); };
  auto done = [&]() {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&bars.empty[n & 1]);
    ++n;
  };
  auto src = [&]() { return stage + (n & 1) * kPiece; };
  const bool t_rows = P.T.kind == OP_YXK, b_rows = P.B.kind == OP_YEO;
#pragma unroll 1
  for (int u = 0; u < R.units; ++u) {
    const bool fresh = u == 0 || p == 0;
    if (u >= 2 && !wait(&bars.t_free[u & 1], ((u >> 1) - 1) & 1)) return;
#pragma unroll 1
    for (int h = 0; h < (t_rows ? 1 : 4); ++h) {
      if (!take()) return;
      convert_t<X3>(src(), h, t_rows, p, sm + OFF_T + (u & 1) * 2 * SZ_T);
      done();
    }
    warp_publish(&bars.t_full[u & 1]);
#pragma unroll 1
    for (int j = 0; j < kNB; ++j) {
      const int g = u * kNB + j;
      if (g >= 2 && !wait(&bars.e_free[g & 1], ((g >> 1) - 1) & 1)) return;
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        if (!take()) return;
        convert_e<X3>(src(), h, sm + OFF_E + (g & 1) * 2 * SZ_E);
        done();
      }
      warp_publish(&bars.e_full[s_e]);
      s_e = s_e + 1 == kStreams ? 0 : s_e + 1;
      if (j > 0 || !fresh) continue;
      const uint32_t prev = (uint32_t)(chain - 1) & 1u;
#pragma unroll 1
      for (int s = 0; s < 2; ++s) {
        if (chain > 0 && !wait(&bars.a_free[s], prev)) return;
        const bool mirrored = s ? P.A2.s[0] < P.A2.s[2] : P.A1.s[0] < P.A1.s[2];
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          if (!take()) return;
          convert_a<X3>(src(), h, mirrored, sm + (s ? OFF_A2 : OFF_A1));
          done();
        }
        warp_publish(&bars.a_full[s]);
      }
      if (chain > 0 && !wait(&bars.b_free, prev)) return;
#pragma unroll 1
      for (int h = 0; h < 4; ++h) {
        if (!take()) return;
        convert_b<X3>(src(), h, b_rows, sm + OFF_B);
        done();
      }
      warp_publish(&bars.b_full);
      ++chain;
    }
    p = (p + 1) & 3;
  }
}

template <bool X3>
__device__ __forceinline__ void products4(const Range4& R, uint32_t sbase, uint32_t tmem, int s, Bars4& bars, PipeWait wait) {
  const uint32_t id_n = idesc<2>(128, 64), id_2n = idesc<2>(128, 128), id4 = idesc<2>(128, 32);
  const uint32_t W = sbase + OFF_W + s * 2 * SZ_W, d = tmem + COL_S123 + s * 128;
  const uint64_t w_sw = sdesc_sw128(W), w_k = sdesc(W, 128, 1024), w_4 = sdesc(W, 128, 256);
  const uint64_t e0 = sdesc(sbase + OFF_E, 128, 512), t0 = sdesc(sbase + OFF_T, 128, 512),
                 a1 = sdesc(sbase + OFF_A1, 128, 1024), a2 = sdesc(sbase + OFF_A2, 128, 1024), b0 = sdesc(sbase + OFF_B, 128, 256);
  constexpr uint32_t LO = SZ_W >> 4;
  const int tiles = R.units * kNB;
  uint64_t* const s4_before = &bars.s4[(s + kStreams - 1) % kStreams];
  uint32_t wph = 0;  // parity of this stream's tile; of the first of its three phases of w
#pragma unroll 1
  for (int g = s; g < tiles; g += kStreams) {
    const int u = g >> 4, j = g & 15, p = (R.p + u) & 3;
    const uint32_t cp = (uint32_t)((R.p + u) >> 2) & 1u;             // the chain's parity
    const bool first = j < kStreams && (u == 0 || p == 0);          // this stream's first tile of a chain
    const bool t_last = j >= kNB - kStreams, last = t_last && p == 3;  // its last one of a unit, of a chain
    if (j < kStreams && !wait.one(&bars.t_full[u & 1], (u >> 1) & 1)) return;
    if (!wait.one(&bars.e_full[s], wph)) return;
    tc_after_sync();
    const uint64_t e = e0 + (g & 1) * (2 * SZ_E >> 4);
    mma_steps<X3, 2>(d, e, e + (SZ_E >> 4), t0 + (u & 1) * (2 * SZ_T >> 4), 16, 16, id_n, id_2n, 0u);
    commit(&bars.acc[s]);
    commit(&bars.e_free[g & 1]);
    if (t_last) commit(&bars.t_free[u & 1]);
    if (first && !wait.one(&bars.a_full[0], cp)) return;
    if (!wait.one(&bars.w[s], wph)) return;
    tc_after_sync();
    mma_steps<X3, 4>(d, w_sw, w_sw + LO, a1, 2, 16, id_n, id_2n, 0u);
    commit(&bars.acc[s]);
    if (last) commit(&bars.a_free[0]);
    if (first && !wait.one(&bars.a_full[1], cp)) return;
    if (!wait.one(&bars.w[s], wph ^ 1u)) return;
    tc_after_sync();
    mma_steps<X3, 4>(d, w_k, w_k + LO, a2, 16, 16, id_n, id_2n, 0u);
    commit(&bars.acc[s]);
    if (last) commit(&bars.a_free[1]);
    if (first && !wait.one(&bars.b_full, cp)) return;
    // S4 of the tile before this one (the stream before, whose parity differs for stream 0) is
    // complete: one accumulator, in order
    if (g > 0 && !wait.one(s4_before, s == 0 ? wph ^ 1u : wph)) return;
    if (j == 0 && u > 0 && !wait.one(&bars.o_free, (uint32_t)(u - 1) & 1u)) return;
    if (!wait.one(&bars.w[s], wph)) return;
    wph ^= 1u;
    tc_after_sync();
    const uint64_t b = b0 + j * (2 * SZ_B >> 4);
    const uint32_t acc = j > 0 ? 1u : 0u;
#pragma unroll
    for (int qq = 0; qq < 4; ++qq) {
      const uint32_t d4 = tmem + COL_S4 + qq * 32;
      mma<2>(d4, w_4 + qq * 256, b, id4, acc);
      if constexpr (X3) {
        mma<2>(d4, w_4 + qq * 256, b + (SZ_B >> 4), id4, 1u);
        mma<2>(d4, w_4 + LO + qq * 256, b, id4, 1u);
      }
    }
    commit(&bars.s4[s]);
    if (last) commit(&bars.b_free);
  }
}

// The drains of one stream, and the results of the units that end in it.  Z stays in W until
// S4 has read it: the commit of the next S1, issued behind S4, covers that.
template <bool X3>
__device__ __forceinline__ void drain4(const Plan4& P, const Range4& R, uint8_t* sm, uint32_t tmem, int s, Bars4& bars,
                                       PipeWait wait) {
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) & 7, q = warp & 3, h = warp >> 2;
  const uint32_t row = tmem + COL_S123 + s * 128 + h * 32 + ((uint32_t)(q * 32) << 16);
  uint8_t* W = sm + OFF_W + s * 2 * SZ_W;
  const int m = q * 32 + lane, lo3 = m & 7, mid = (m >> 3) & 7, top = m >> 6;
  // S1: row (b,l2,l1) -> S2 rows (l2,b,a'), chunk l1 (swizzled); S2: row (l2,b,a') -> S3 rows
  // (b,r1,a'), chunk l2; S3: row (b,r1,a') -> S4 rows (r1,r2,a'), chunk b
  const uint32_t base0 = (mid * 16 + top * 8 + h * 4) << 7;
  const uint32_t base1 = ((((m >> 3) & 1) * 8 + h * 4) * 8 + (m >> 4)) * 128 + lo3 * 16;
  const uint32_t base2 = ((mid * 8 + h * 4) * 2 + top) * 128 + lo3 * 16;
  const int tiles = R.units * kNB;
  uint32_t ph = 0;  // of acc: odd number of phases per tile
#pragma unroll 1
  for (int t = s; t < tiles; t += kStreams) {
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
      if (!wait(&bars.acc[s], ph)) return;
      ph ^= 1u;
      tc_after_sync();
      uint8_t* dst = W + (k == 0 ? base0 : k == 1 ? base1 : base2);
      const uint32_t stride = k == 0 ? 128u : k == 1 ? 1024u : 256u;
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        float v[16];
        load_acc16<X3>(row + g * 16, v);
#pragma unroll
        for (int i2 = 0; i2 < 2; ++i2) {
          const int i = g * 2 + i2;
          put_split8<X3>(dst + i * stride + (k == 0 ? ((lo3 ^ (h * 4 + i)) & 7) << 4 : 0), v + i2 * 8, SZ_W);
        }
      }
      warp_publish(&bars.w[s]);
    }
    if ((t & (kNB - 1)) != kNB - 1) continue;
    // results O[(r1,r2,a')][b'] of the unit
    if (!wait(&bars.s4[s], ph ^ 1u)) return;
    tc_after_sync();
    const Env4Fused& a = P.a;
    const int v0 = R.p + (t >> 4);
    float* O = a.out + (R.c + (v0 >> 2)) * a.bsO + ((v0 & 3) * kAT + lo3) * a.sOa2;
#pragma unroll 1
    for (int i = 0; i < 4; ++i) {
      const int qq = h + (i & 2), b0 = (i & 1) * 16, m4 = qq * 128 + m;
      float v[16];
      tmem_ld16(tmem + COL_S4 + qq * 32 + b0 + ((uint32_t)(q * 32) << 16), v);
      float* d = O + (m4 >> 6) * a.sOr1 + mid * a.sOr2 + b0 * a.sOb2;
#pragma unroll
      for (int e = 0; e < 16; ++e) d[e * a.sOb2] = v[e];
    }
    tc_before_sync();
    __syncwarp();
    if (lane == 0) mbar_arrive(&bars.o_free);
  }
}

template <bool X3>
__global__ void __launch_bounds__(kThreads, 1) env4_pipe_kernel(const __grid_constant__ Plan4 P, unsigned* status) {
  extern __shared__ __align__(1024) uint8_t sm[];  // the swizzled tiles lie on 1 KB boundaries
  __shared__ __align__(8) Bars4 bars;
  __shared__ uint32_t tmem_base;
  __shared__ PipeCtl ctl;
  const int bi = blockIdx.x, u0 = bi * P.share + min(bi, P.rest);
  const Range4 R{u0 >> 2, u0 & 3, P.share + (bi < P.rest ? 1 : 0)};
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    mbar_init(&bars.b_full, kLoadWarps);
    mbar_init(&bars.b_free, kStreams);
    mbar_init(&bars.o_free, kDrainWarps);
#pragma unroll 1
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars.full[i], 1);
      mbar_init(&bars.empty[i], kLoadWarps);
      mbar_init(&bars.t_full[i], kLoadWarps);
      mbar_init(&bars.t_free[i], kStreams);
      mbar_init(&bars.e_free[i], 1);
      mbar_init(&bars.a_full[i], kLoadWarps);
      mbar_init(&bars.a_free[i], kStreams);
    }
#pragma unroll 1
    for (int i = 0; i < kStreams; ++i) {
      mbar_init(&bars.e_full[i], kLoadWarps);
      mbar_init(&bars.s4[i], 1);
      mbar_init(&bars.acc[i], 1);
      mbar_init(&bars.w[i], kDrainWarps);
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
  constexpr int LOAD0 = kStreams * kDrainWarps, COPY0 = LOAD0 + kLoadWarps;
  if (warp < LOAD0) {
    drain4<X3>(P, R, sm, tmem, warp / kDrainWarps, bars, wait);
  } else if (warp < COPY0) {
    load4<X3>(P, R, sm, bars, wait);
  } else if ((threadIdx.x & 31) == 0) {
    if (warp == COPY0) {
      copy4(P, R, smem_u32(sm) + OFF_STAGE, bars, wait);
    } else {
      const int s = warp - COPY0 - 1;
      products4<X3>(R, smem_u32(sm), tmem, s, bars, wait);
      commit(&bars.fin[s]);  // whatever was issued completes before the tensor memory is released
      wait_parity(&bars.fin[s], 0u, ctl.budget > kDefaultWaitCycles ? ctl.budget : kDefaultWaitCycles);
    }
  }
  __syncwarp();
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

void set3(PipeOp& o, int kind, const float* base, long long chain, int n0, long long s0, int n1, long long s1, int n2,
          long long s2) {
  o.kind = kind; o.base = base; o.chain = chain;
  o.n[0] = n0; o.s[0] = (int)s0; o.n[1] = n1; o.s[1] = (int)s1; o.n[2] = n2; o.s[2] = (int)s2;
  finish_operand(o);
}
void set_site(PipeOp& o, const float* base, long long slot, int nl, long long sl, int nu, long long su, int nr, long long sr,
              int nd, long long sd) {
  o.n[3] = nd;
  o.s[3] = (int)sd;
  set3(o, OP_SITE, base, slot, nl, sl, nu, su, nr, sr);
}

template <bool X3>
cudaError_t launch(const Plan4& P, int grid, unsigned* status, cudaStream_t st) {
  static SmemLimit limit{SMEM_BYTES, false};
  return launch_large(limit, true, env4_pipe_kernel<X3>, grid, kThreads, SMEM_BYTES, st, P, status);
}

}  // namespace

bool env4_pipe_fits(const Env4Fused& a, void* plan) {
  static_assert(sizeof(Plan4) <= kEnv4PlanBytes);
  Plan4& P = *new (plan) Plan4;
  P.a = a;
  if (a.batch >= 1 << 28 || a.cT != 32 || a.cB != 32 || a.cT2 != 32 || a.cB2 != 32 || a.D1r != 8 || a.D2r != 8) return false;
  set3(P.T, a.sTa2 > a.sTa ? OP_YXK : OP_KXY, a.T, a.bsT, a.cT, a.sTa, a.Du1, a.sTu, a.cT2, a.sTa2);
  set_site(P.A1, a.A1, a.ss1, a.D1l, a.s1l, a.Du1, a.s1u, a.D1r, a.s1r, a.Dd1, a.s1d);
  set_site(P.A2, a.A2, a.ss2, a.D2l, a.s2l, a.Dd1, a.s2u, a.D2r, a.s2r, a.Dd2, a.s2d);
  set3(P.B, a.sBb2 > a.sBb ? OP_YEO : OP_OE, a.B, a.bsB, a.cB, a.sBb, a.Dd2, a.sBd, a.cB2, a.sBb2);
  return full_operand(P.T) && full_operand(P.A1) && full_operand(P.A2) && full_operand(P.B) &&
         a.sEb == 2048 && a.sEa == 64 && a.sEl1 == 8 && a.sEl2 == 1 && (a.bsE & 3) == 0 &&
         (reinterpret_cast<uintptr_t>(a.E) & 15) == 0;
}

cudaError_t env4_pipe(const void* plan, bool split, unsigned* status, cudaStream_t st) {
  Plan4 P = *static_cast<const Plan4*>(plan);
  int sms = 0;
  PV_CUDA(sm_count(&sms));
  const int units = 4 * P.a.batch, grid = units < sms ? units : sms;
  P.share = units / grid;
  P.rest = units % grid;
  return split ? launch<true>(P, grid, status, st) : launch<false>(P, grid, status, st);
}

}  // namespace pv
