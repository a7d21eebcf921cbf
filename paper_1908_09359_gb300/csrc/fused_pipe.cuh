// Shared pieces of the warp-specialised fused column-step kernels (sm_103a): one CTA per
// SM runs two independent streams of tiles, so that one stream's accumulator drains
// overlap the other's products.  Warps: 8 drain warps per stream, 8 loader warps, 4 that write
// the results, one product-issuing warp per stream and one that issues bulk copies; all
// hand-overs are mbarriers with a clock budget.
//
// Operands arrive as float32: a bulk copy brings a 16 KB piece of a chain's operand, as it
// lies in memory, into one of two staging buffers, and the loader warps convert it into the
// operand's layout.  (Converted straight from global loads, 26 warps' tiles leave 28 KB of
// first-level cache, too few lines for the loads in flight: measured ~5,000 cycles per round
// trip, and the loaders, not the products, set the pace.)
#pragma once
#include "tc_util.cuh"

namespace pv {
namespace tc {

constexpr int kPipeDrainWarps = 8;   // per stream
constexpr int kPipeLoadWarps = 8;    // convert operands
constexpr int kPipeOutWarps = 4;     // write the results, one per tensor-memory lane quarter
constexpr int kPipeThreads = (2 * kPipeDrainWarps + kPipeLoadWarps + kPipeOutWarps + 3) * 32;
enum PipeRole { ROLE_DRAIN, ROLE_LOAD, ROLE_OUT, ROLE_PRODUCTS, ROLE_COPY };
__device__ __forceinline__ PipeRole pipe_role(int warp) {
  return warp < 2 * kPipeDrainWarps                        ? ROLE_DRAIN
         : warp < 2 * kPipeDrainWarps + kPipeLoadWarps     ? ROLE_LOAD
         : warp < 2 * kPipeDrainWarps + kPipeLoadWarps + kPipeOutWarps ? ROLE_OUT
         : warp < 2 * kPipeDrainWarps + kPipeLoadWarps + kPipeOutWarps + 2 ? ROLE_PRODUCTS : ROLE_COPY;
}

// Waits of one kernel, set up once per CTA in shared memory.  A wait that runs out of budget
// sets `abort` for the whole CTA (every other wait then returns false at its next poll) and
// ST_TIMEOUT in the status word.  One out-of-line copy: the code of all roles has to stay in
// the SM's instruction cache.
struct PipeCtl {
  int abort;
  unsigned* status;
  long long budget;
};
static __device__ __noinline__ bool pipe_wait(uint32_t bar, uint32_t parity, PipeCtl* ctl) {
  uint32_t done;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  if (done) return true;
  const long long t0 = clock64(), budget = ctl->budget;
  const uint32_t ns = (uint32_t)(budget < 40000 ? budget >> 1 : 20000);  // how long one try may suspend the warp
  while (true) {
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(ns)
        : "memory");
    if (done) return true;
    if (*reinterpret_cast<volatile int*>(&ctl->abort)) return false;
    if (clock64() - t0 > budget) {
      *reinterpret_cast<volatile int*>(&ctl->abort) = 1;
      atomicOr(ctl->status, ST_TIMEOUT);
      return false;
    }
  }
}
struct PipeWait {
  PipeCtl* ctl;
  // every lane of the warp waits; all lanes get the same answer
  __device__ __forceinline__ bool operator()(uint64_t* bar, uint32_t parity) const {
    return __all_sync(0xffffffffu, pipe_wait(smem_u32(bar), parity, ctl));
  }
  // a single thread waits
  __device__ __forceinline__ bool one(uint64_t* bar, uint32_t parity) const { return pipe_wait(smem_u32(bar), parity, ctl); }
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Shared-memory writes of this warp are handed to the products: every lane orders its own
// writes (and tensor-memory loads) first, then one lane arrives for the warp.
__device__ __forceinline__ void warp_publish(uint64_t* bar) {
  fence_async_smem();
  tc_before_sync();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
}

// Eight values split into BF16 hi + lo (put16's split: hi = bf16(x), lo = bf16(x - hi), the
// remainder formed exactly by a fused multiply-add that takes hi as BF16) or, without X3,
// rounded to BF16; 16 bytes each at dst and dst + lo_off.
template <bool X3>
__device__ __forceinline__ void put_split8(uint8_t* dst, const float* f, int lo_off) {
  uint32_t w[4], wl[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[i]) : "f"(f[2 * i + 1]), "f"(f[2 * i]));
    if constexpr (X3) {
      float l0, l1;
      asm("{\n.reg .b16 h0, h1, m1;\nmov.b32 {h0, h1}, %2;\nmov.b16 m1, 0xBF80;\n"
          "fma.rn.f32.bf16 %0, h0, m1, %3;\nfma.rn.f32.bf16 %1, h1, m1, %4;\n}\n"
          : "=&f"(l0), "=f"(l1)
          : "r"(w[i]), "f"(f[2 * i]), "f"(f[2 * i + 1]));
      asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(wl[i]) : "f"(l1), "f"(l0));
    }
  }
  *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
  if constexpr (X3) *reinterpret_cast<uint4*>(dst + lo_off) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
}

// 16 accumulator columns of this thread's row; with X3 the columns 64 further on (the
// products with the B operand's lo part) are added.
template <bool X3>
__device__ __forceinline__ void load_acc16(uint32_t taddr, float* v) {
  if constexpr (X3) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]), "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]), "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]), "=&r"(r[15]), "=&r"(r[16]), "=&r"(r[17]), "=&r"(r[18]), "=&r"(r[19]), "=&r"(r[20]), "=&r"(r[21]), "=&r"(r[22]), "=&r"(r[23]), "=&r"(r[24]), "=&r"(r[25]), "=&r"(r[26]), "=&r"(r[27]), "=&r"(r[28]), "=&r"(r[29]), "=&r"(r[30]), "=&r"(r[31])
        : "r"(taddr), "r"(taddr + 64)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
      const float2 s = __fadd2_rn(make_float2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])),
                                  make_float2(__uint_as_float(r[16 + i]), __uint_as_float(r[17 + i])));
      v[i] = s.x;
      v[i + 1] = s.y;
    }
  } else {
    tmem_ld16(taddr, v);
  }
}

// n K steps of a split (or plain) BF16 product into accumulator d (N columns; with X3 columns
// N..2N-1 receive A_hi x B_lo); the descriptors advance by da and db (units of 16 bytes) per
// step; acc: whether the first step accumulates.
template <bool X3, int n>
__device__ __forceinline__ void mma_steps(uint32_t d, uint64_t a_hi, uint64_t a_lo, uint64_t b, uint32_t da, uint32_t db,
                                          uint32_t id_n, uint32_t id_2n, uint32_t acc) {
#pragma unroll
  for (int k = 0; k < n; ++k) {
    if constexpr (X3) {
      mma<2>(d, a_hi, b, id_2n, acc);  // [hi x hi | hi x lo]
      mma<2>(d, a_lo, b, id_n, 1u);    // lo x hi into the first half
    } else {
      mma<2>(d, a_hi, b, id_n, acc);
    }
    acc = 1u;
    a_hi += da;
    a_lo += da;
    b += db;
  }
}

// 32 rows x 32 columns of results in shared memory, rows kRowPitch floats apart (16-byte
// accesses of eight rows, and of one row's 128 bytes, are free of bank conflicts).
constexpr int kRowPitch = 36;
__device__ __forceinline__ void put_row16(float* row, const float* v) {
#pragma unroll
  for (int e = 0; e < 16; e += 4) *reinterpret_cast<float4*>(row + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
}
__device__ __forceinline__ void add_row16(const float* row, float* v) {
#pragma unroll
  for (int e = 0; e < 16; e += 4) {
    const float4 f = *reinterpret_cast<const float4*>(row + e);
    v[e] += f.x; v[e + 1] += f.y; v[e + 2] += f.z; v[e + 3] += f.w;
  }
}
// Store rows i = 8 g + k (g < groups, k < 8) at dst + g * s_group + k * s_row, n_cols columns
// s_col apart; only k < n_rows and the first n_groups groups exist.  vec: columns contiguous,
// everything on 16 bytes and n_cols a multiple of 4.
__device__ __forceinline__ void store_rows(const float* buf, float* dst, long long s_group, long long s_row, long long s_col,
                                           int n_groups, int n_rows, int n_cols, bool vec) {
  const int lane = threadIdx.x & 31;
  if (vec) {
    // eight lanes per row, four rows per step
    const int k = lane >> 3, col = (lane & 7) * 4;
    const float* b = buf + k * kRowPitch + col;
    float* d0 = dst + k * s_row + col;
    float* d1 = d0 + 4 * s_row;
    const bool v0 = k < n_rows && col < n_cols, v1 = k + 4 < n_rows && col < n_cols;
#pragma unroll 1
    for (int g = 0; g < n_groups; ++g) {
      const float4 x = *reinterpret_cast<const float4*>(b), y = *reinterpret_cast<const float4*>(b + 4 * kRowPitch);
      if (v0) *reinterpret_cast<float4*>(d0) = x;
      if (v1) *reinterpret_cast<float4*>(d1) = y;
      b += 8 * kRowPitch;
      d0 += s_group;
      d1 += s_group;
    }
  } else {
#pragma unroll 1
    for (int g = 0; g < n_groups; ++g)
#pragma unroll 1
      for (int k = 0; k < n_rows; ++k)
        if (lane < n_cols) dst[g * s_group + k * s_row + lane * s_col] = buf[(g * 8 + k) * kRowPitch + lane];
  }
}

// ------------------------------------------------------------------ operand staging
constexpr uint32_t kStageBytes = 16384;

// One operand of a unit, described on the host: where its pieces lie in global memory and how
// they become a K-major operand of 16-byte chunks (8 K values each).  An operand has an
// outermost index of at most 32 values and is taken in pieces of 16 of them.
enum OperandKind : int {
  OP_KXY,   // rows y*8 + x, K = k; k outermost, y innermost: dims (k, x, y)
  OP_YXK,   // the same rows from memory with y outermost, k innermost
  OP_OE,    // rows y, K = (o, e); o outermost: dims (o, e, y)
  OP_YEO,   // the same from memory with y outermost, o innermost
  OP_SITE,  // site tensor, rows r*8 + d, K = (l, u), 64 x 64, one piece: dims (l, u, r, d)
};
struct PipeOp {
  const float* base = nullptr;
  long long chain = 0;          // floats between chains (site tensor: between slots)
  int s[4] = {}, n[4] = {};     // strides (floats) and extents in the order of the kind's dims
  int kind = 0, pieces = 1, bulk = 0;
  int piece = 0;                // floats from one piece to the next
  uint32_t bytes[2] = {};       // of each piece
  // destination: byte offset in shared memory, bytes between tiles of 2^ys rows' y (KXY, YXK) or
  // of 8 (16 when swizzled) o, and from the hi to the lo part
  uint32_t dst = 0, tile = 0, lo = 0;
  int ys = 0, swizzled = 0;
};

// Fill in pieces and bulk: a bulk copy needs dense pieces that start and end on 16 bytes.
inline void finish_operand(PipeOp& o) {
  const bool y_outer = o.kind == OP_YXK || o.kind == OP_YEO;
  const int d = o.kind == OP_SITE ? 4 : 3;
  long long total = 1, extent = 1;
  for (int i = 0; i < d; ++i) {
    total *= o.n[i];
    extent += (long long)(o.n[i] - 1) * o.s[i];
  }
  const int outer = o.kind == OP_SITE ? 0 : y_outer ? 2 : 0;
  const int n = o.kind == OP_SITE ? 1 : o.n[outer], step = o.kind == OP_SITE ? (int)total : o.s[outer];
  o.pieces = n > 16 ? 2 : 1;
  o.piece = 16 * step;
  const long long f0 = (long long)(n > 16 ? 16 : n) * step, f1 = n > 16 ? (long long)(n - 16) * step : 0;
  o.bytes[0] = (uint32_t)(f0 * 4);
  o.bytes[1] = (uint32_t)(f1 * 4);
  o.bulk = extent == total && (long long)n * step == total && (f0 & 3) == 0 && (f1 & 3) == 0 && (o.chain & 3) == 0 &&
           (reinterpret_cast<uintptr_t>(o.base) & 15) == 0 && f0 * 4 <= kStageBytes && f1 * 4 <= kStageBytes;
}

// The two staging buffers: filled by the copy thread, emptied by the loader warps.
struct Staging {
  uint64_t full[2], empty[2];
};
__device__ __forceinline__ void staging_init(Staging& g) {
  for (int i = 0; i < 2; ++i) {
    mbar_init(&g.full[i], 1);
    mbar_init(&g.empty[i], kPipeLoadWarps);
  }
}

// Copy thread: pieces in the order in which the loader warps convert them.
struct Copier {
  Staging& g;
  uint32_t stage;  // shared address of the buffers
  PipeWait wait;
  int n = 0;       // pieces issued
  __device__ __forceinline__ bool operand(const PipeOp& o, int c) {
    if (!o.bulk) return true;
    const float* src = o.base + c * o.chain;
#pragma unroll 1
    for (int p = 0; p < o.pieces; ++p, src += o.piece) {
      const int st = n & 1;
      if (n >= 2 && !wait.one(&g.empty[st], ((n >> 1) - 1) & 1)) return false;
      const uint32_t bytes = p ? o.bytes[1] : o.bytes[0];
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&g.full[st])), "r"(bytes)
                   : "memory");
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                       stage + st * kStageBytes),
                   "l"(src), "r"(bytes), "r"(smem_u32(&g.full[st]))
                   : "memory");
      ++n;
    }
    return true;
  }
  // ask for chain c's operand in the second-level cache (the staging buffers hold two pieces
  // only, too few to cover the latency of device memory)
  __device__ __forceinline__ static void prefetch(const PipeOp& o, int c) {
    if (o.bulk)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(o.base + c * o.chain), "r"(o.bytes[0] + o.bytes[1])
                   : "memory");
  }
  // whatever was issued lands (with a limit) before the shared memory is given up
  __device__ __forceinline__ void finish() {
#pragma unroll 1
    for (int k = max(0, n - 2); k < n; ++k) wait_parity(&g.full[k & 1], (k >> 1) & 1, kDefaultWaitCycles);
  }
};

// Piece p of an operand at src (its own element offsets apply) to shared memory, two chunks
// per loader thread (256 threads: warp w, lane).  Lane mappings keep the reads of a dense
// 32 x 8 x 32 operand and the stores free of bank conflicts; each store phase of eight lanes
// writes the eight rows of a row group.  Out of line, one copy per kind and scalar arguments
// (a descriptor behind a pointer costs a load per field and call).
struct Dims4 {
  int s0, s1, s2, s3, n0, n1, n2, n3;
};
template <bool X3, int KIND>
__device__ __noinline__ void convert_piece(const float* src, int p, Dims4 d, uint8_t* base, uint32_t tile, uint32_t lo,
                                           int arg) {
  const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) & 7;
  float v[2][8];
  uint32_t dst[2];
#pragma unroll
  for (int n = 0; n < 2; ++n) {
    int off, sk, left;   // offset of the chunk's first element, its stride, valid elements
    bool vec = false;
    if constexpr (KIND == OP_SITE) {
      // lanes along (r, d), or (the mirrored view, whose l runs inside r) along d and l
      const int i = 2 * w + n, dd = lane & 7, in = (lane >> 3) + 4 * (i & 1), out = i >> 1;
      const int l = d.s0 > d.s2 ? out : in, r = d.s0 > d.s2 ? in : out;
      off = l * d.s0 + r * d.s2 + dd * d.s3;
      sk = d.s1;
      left = l < d.n0 && r < d.n2 && dd < d.n3 ? d.n1 : 0;
      dst[n] = kmajor_off(r * 8 + dd, l * 8, 8);
    } else if constexpr (KIND == OP_OE || KIND == OP_YEO) {
      const int i = 16 * p + 2 * w + n, k = KIND == OP_OE ? i : lane, y = KIND == OP_OE ? lane : i;
      off = k * d.s0 + y * d.s2;
      sk = d.s1;
      left = k < d.n0 && y < d.n2 ? d.n1 : 0;
      // swizzled (arg): atoms of 64 rows x 8 o, two to a tile
      dst[n] = arg ? (k >> 4) * tile + ((k >> 3) & 1) * (tile >> 1) + sw128_chunk_off(y, k & 7)
                   : (k >> 3) * tile + kmajor_off(y, (k & 7) * 8, 8);
    } else {
      int kc, x, y;
      if constexpr (KIND == OP_KXY) {  // lane = y, and x rotates with the lane
        kc = 2 * p + (w & 1);
        x = (lane + (w >> 1) + 4 * n) & 7;
        y = lane;
      } else {  // lanes x, then four y; a lane's two 16-byte reads rotate with x
        x = lane & 7;
        y = 16 * p + (lane >> 3) + 4 * (w & 3);
        kc = ((w >> 2) + 2 * n + (x >> 1)) & 3;
        vec = d.s0 == 1 && ((d.s1 | d.s2) & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
      }
      off = kc * 8 * d.s0 + x * d.s1 + y * d.s2;
      sk = d.s0;
      left = x < d.n1 && y < d.n2 ? d.n0 - kc * 8 : 0;
      dst[n] = (y >> arg) * tile + ((((y & ((1 << arg) - 1)) * 4 + kc) << 7) + (x << 4));
    }
    const float* s = src + off;
    if (KIND == OP_YXK && vec && left >= 8) {
      const int h = lane & 1;
      const float4 f = *reinterpret_cast<const float4*>(s + 4 * h), g = *reinterpret_cast<const float4*>(s + 4 - 4 * h);
      const float4 a = h ? g : f, b = h ? f : g;
      v[n][0] = a.x; v[n][1] = a.y; v[n][2] = a.z; v[n][3] = a.w;
      v[n][4] = b.x; v[n][5] = b.y; v[n][6] = b.z; v[n][7] = b.w;
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e, s += sk) v[n][e] = e < left ? *s : 0.f;
    }
  }
#pragma unroll
  for (int n = 0; n < 2; ++n) put_split8<X3>(base + dst[n], v[n], lo);
}

// The same for a staged piece of an operand with every extent at its maximum (32 x 8 x 32, site
// 8 x 8 x 8 x 8) and dense: no bounds and constant strides, a third of the instructions.
// Conversions are a chain of dependent instructions in a few warps (about 1,000 cycles a piece
// in the general form, twice that beside busy drains), and the products wait for them at
// every chain.
__device__ __forceinline__ float lds(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ float4 lds4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
template <bool X3, int KIND>
__device__ __forceinline__ void convert_full(uint32_t src, int p, bool mirrored, uint8_t* base, uint32_t tile, uint32_t lo,
                                             int ys, bool swizzled) {
  const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) & 7;
  float v[2][8];
  uint32_t dst[2];
#pragma unroll
  for (int n = 0; n < 2; ++n) {
    constexpr int SK = KIND == OP_KXY ? 256 : KIND == OP_SITE ? 64 : 32;
    uint32_t off;
    if constexpr (KIND == OP_SITE) {
      const int i = 2 * w + n, d = lane & 7, in = (lane >> 3) + 4 * (i & 1), out = i >> 1;
      off = out * 512 + in * 8 + d;
      dst[n] = kmajor_off((mirrored ? out : in) * 8 + d, (mirrored ? in : out) * 8, 8);
    } else if constexpr (KIND == OP_OE || KIND == OP_YEO) {
      const int i = 2 * w + n, k = KIND == OP_OE ? 16 * p + i : lane, y = KIND == OP_OE ? lane : 16 * p + i;
      off = i * 256 + lane;
      dst[n] = swizzled ? (k >> 4) * tile + ((k >> 3) & 1) * (tile >> 1) + sw128_chunk_off(y, k & 7)
                        : (k >> 3) * tile + kmajor_off(y, (k & 7) * 8, 8);
    } else {
      int kc, x, y;
      if constexpr (KIND == OP_KXY) {
        kc = 2 * p + (w & 1);
        x = (lane + (w >> 1) + 4 * n) & 7;
        y = lane;
        off = (w & 1) * 8 * 256 + x * 32 + y;
      } else {
        x = lane & 7;
        y = 16 * p + (lane >> 3) + 4 * (w & 3);
        kc = ((w >> 2) + 2 * n + (x >> 1)) & 3;
        off = (y & 15) * 256 + x * 32 + kc * 8;
      }
      dst[n] = (y >> ys) * tile + ((((y & ((1 << ys) - 1)) * 4 + kc) << 7) + (x << 4));
    }
    if constexpr (KIND == OP_YXK) {
      const int h = lane & 1;
      const float4 f = lds4(src + off * 4 + 16 * h), g = lds4(src + off * 4 + 16 - 16 * h);
      const float4 a = h ? g : f, b = h ? f : g;
      v[n][0] = a.x; v[n][1] = a.y; v[n][2] = a.z; v[n][3] = a.w;
      v[n][4] = b.x; v[n][5] = b.y; v[n][6] = b.z; v[n][7] = b.w;
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[n][e] = lds(src + off * 4 + e * SK * 4);
    }
  }
#pragma unroll
  for (int n = 0; n < 2; ++n) put_split8<X3>(base + dst[n], v[n], lo);
}
// An operand of convert_full.
inline bool full_operand(const PipeOp& o) {
  if (!o.bulk) return false;
  if (o.kind == OP_SITE)
    return o.n[0] == 8 && o.n[1] == 8 && o.n[2] == 8 && o.n[3] == 8 && o.s[1] == 64 && o.s[3] == 1 &&
           ((o.s[0] == 512 && o.s[2] == 8) || (o.s[0] == 8 && o.s[2] == 512));
  const bool k_outer = o.kind == OP_KXY || o.kind == OP_OE;
  return o.n[0] == 32 && o.n[1] == 8 && o.n[2] == 32 && o.s[1] == 32 && o.s[0] == (k_outer ? 256 : 1) &&
         o.s[2] == (k_outer ? 1 : 256);
}

// Loader warps' side of the staging buffers.
struct Loader {
  Staging& g;
  uint8_t* sm;
  uint32_t stage;  // byte offset of the buffers
  PipeWait wait;
  int n = 0;       // pieces taken
  // both pieces of chain (slot) c's operand; those a bulk copy cannot take are read from
  // global memory.  Pieces beyond the operand give zeros.
  template <bool X3, bool FULL, int KIND, int KIND2>
  __device__ __forceinline__ bool operand(const PipeOp& o, int c) {
    const Dims4 d{o.s[0], o.s[1], o.s[2], o.s[3], o.n[0], o.n[1], o.n[2], o.n[3]};
    const int arg = KIND == OP_KXY ? o.ys : o.swizzled;
#pragma unroll 1
    for (int p = 0; p < (KIND == OP_SITE ? 1 : 2); ++p) {
      const bool staged = FULL || (o.bulk && p < o.pieces);
      if (staged && !wait(&g.full[n & 1], (n >> 1) & 1)) return false;
      if constexpr (FULL) {
        const uint32_t src = smem_u32(sm) + stage + (n & 1) * kStageBytes;
        const bool mirrored = KIND == OP_SITE && o.s[0] < o.s[2];
        if (KIND == KIND2 || o.kind == KIND)
          convert_full<X3, KIND>(src, p, mirrored, sm + o.dst, o.tile, o.lo, o.ys, o.swizzled);
        else
          convert_full<X3, KIND2>(src, p, mirrored, sm + o.dst, o.tile, o.lo, o.ys, o.swizzled);
      } else {
        const float* src = staged ? reinterpret_cast<const float*>(sm + stage + (n & 1) * kStageBytes) - p * o.piece
                                  : o.base + c * o.chain;
        if (KIND == KIND2 || o.kind == KIND) convert_piece<X3, KIND>(src, p, d, sm + o.dst, o.tile, o.lo, arg);
        else convert_piece<X3, KIND2>(src, p, d, sm + o.dst, o.tile, o.lo, arg);
      }
      if (staged) {
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive(&g.empty[n & 1]);
        ++n;
      }
    }
    return true;
  }
};

}  // namespace tc
}  // namespace pv
