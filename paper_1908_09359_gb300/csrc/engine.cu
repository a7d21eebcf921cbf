// Host engine and C ABI of the VMC-PEPS hot path (arXiv:1908.09359).
//
// The engine issues the device work of one context on one CUDA stream.  All
// chains advance in lock step: every contraction is one batched launch over
// the chains, and per-chain choices (the spin of a site, accept/reject) are
// data on the device, never host branches.
//
// Lattice orientations.  Everything is written for rows swept top-down (the
// boundary-MPS scheme of App. B); the other directions reuse it on re-oriented
// lattices: O1 = upside down (bottom environments), O2 = transposed (columns,
// for vertical bonds), O3 = transposed and upside down.  Each orientation has
// its own permuted float copies of the site tensors.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <string>
#include <vector>

#include "common.cuh"
#include "fused.cuh"
#include "fused_f32.cuh"
#include "kernels.cuh"
#include "pepsvmc.h"
#include "proposal.cuh"
#include "stages.cuh"

using namespace pv;

namespace {

struct Orient {
  int Ly, Lx;       // rows and columns in this orientation
  bool tr, vf;      // transposed, upside down
};

// One site tensor of an oriented row: both spin slots, two permuted layouts.
struct SiteOp {
  const float* lurd;  // [(l,u)][(r,d)], slot 1 at +size
  const float* urld;  // [(u,r)][(l,d)]
  long long size;
  int Dl, Dr, Du, Dd;
  int spin;           // original lattice index k*Lx + m (selects the slot per chain)
};

// One boundary MPS for all chains: site m of chain c at base + m*site_stride + c*chain_stride.
struct View {
  const float* base;
  long long site_stride, chain_stride;
  const std::vector<int>* bond;  // L+1 bond dimensions
  const double* logs;            // per chain log of the norm factored out
  const float* site(int m) const { return base + (long long)m * site_stride; }
};

struct Store {
  float* base = nullptr;
  double* logs = nullptr;  // [rows][C]
  int rows = 0, L = 0;
  std::vector<std::vector<int>> bond;
  float* row_ptr(int r, long long C, long long S) const { return base + (long long)r * L * C * S; }
};

struct Sketch {
  float* dev = nullptr;
  std::vector<long long> off;  // per site
};

std::vector<int> bond_caps(const std::vector<int>& chiX, const std::vector<int>& phys, int chi) {
  const int L = (int)phys.size();
  std::vector<int> r(L > 0 ? L - 1 : 0);
  for (int i = 0; i < L - 1; ++i) r[i] = std::min(chi, chiX[i]);
  int prev = 1;
  for (int i = 0; i < L - 1; ++i) {
    r[i] = std::min(r[i], prev * phys[i]);
    prev = r[i];
  }
  int nxt = 1;
  for (int i = L - 2; i >= 0; --i) {
    r[i] = std::min(r[i], nxt * phys[i + 1]);
    nxt = r[i];
  }
  return r;
}

}  // namespace

struct pepsvmc_ctx {
  pepsvmc_config cfg{};
  cudaStream_t st = nullptr;
  std::string err;
  int C = 0, Ly = 0, Lx = 0, D = 0, chi = 0, nfit = 1, Lmax = 0;
  // chi: the cutoff the fit uses now; the sampler's (chi_s) except inside a measurement
  // with its own cutoff (chi_m); chi_x = max of both sizes the buffers and the sketch
  int chi_s = 0, chi_m = 0, chi_x = 0;
  long long P = 0, Ph = 0, S = 0, S4 = 0, SI = 0;
  Orient O[4];
  std::vector<long long> site_off, site_half_off;  // original sites
  std::vector<int> site_size;
  std::vector<long long> perm_site_off[4];
  long long launches = 0;
  long long wait_budget = 0;  // device wait budget in clock cycles (0 = default)
  unsigned chain_base = 0;    // global index of chain 0 in the Philox counters
  unsigned long long sweep_counter = 0;
  bool top_valid = false, have_grad = false, have_measure = false;
  int trace_on = 0;
  std::vector<double> sketch_host;
  std::map<std::string, Sketch> sketches;
  std::vector<int> trivial_bond;

  // device memory
  std::vector<void*> allocs;
  double* master = nullptr;
  double* grad = nullptr;
  double* sumG = nullptr;
  double* sumGE = nullptr;
  double* sums = nullptr;
  float* perm[4][2] = {};
  int* perm_map[4][2] = {};
  int8_t* spins = nullptr;
  float* ones = nullptr;
  double* zeros_d = nullptr;
  Store st_top, st_bot, st_colbot, st_coltop;
  float *envL = nullptr, *envR = nullptr, *envRf = nullptr;
  float *l3[2] = {}, *fl = nullptr;
  float *tmp1 = nullptr, *tmp2 = nullptr;
  float *tmp3 = nullptr, *tmp4 = nullptr;  // the two shared four-line intermediates Y(f1 = 0, 1)
  float *R4 = nullptr, *l4[2] = {}, *fl4 = nullptr, *ptop[2] = {}, *pbot[2] = {};
  float* G = nullptr;
  double *eloc = nullptr, *den = nullptr, *logpsi = nullptr;
  int8_t* sign = nullptr;
  int* exps = nullptr;
  unsigned* status = nullptr;
  unsigned long long* counters = nullptr;
  unsigned long long* d_sweep = nullptr;
  double* trace_ratio = nullptr;
  int8_t* trace_dec = nullptr;
  int* elem_site = nullptr;
  long long *d_site_half_off = nullptr, *d_site_full_off = nullptr;
  int *d_site_size = nullptr, *d_site_spin = nullptr;

  // ------------------------------------------------------------------ helpers
  bool dry = false;                                      // no device: validate only
  uintptr_t fake_next = (uintptr_t)1 << 44;
  std::vector<std::pair<uintptr_t, size_t>> regions;     // every allocation (bounds checks)

  template <typename T>
  cudaError_t alloc(T** p, size_t n) {
    void* q = nullptr;
    const size_t bytes = n * sizeof(T);
    if (dry) {
      q = reinterpret_cast<void*>(fake_next);
      fake_next += (bytes + 4096) & ~(size_t)255;
    } else {
      cudaError_t e = cudaMalloc(&q, bytes + 256);
      if (e != cudaSuccess) return e;
      allocs.push_back(q);
    }
    regions.push_back({reinterpret_cast<uintptr_t>(q), bytes});
    *p = reinterpret_cast<T*>(q);
    return cudaSuccess;
  }

  // True when elements [0, max_off] of p (element size esz) lie in one allocation.
  bool span(const void* p, long long max_off, size_t esz, const char* what) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    if (!p || max_off < 0) {
      err = std::string("bounds check failed (null or negative span): ") + what;
      return false;
    }
    const uintptr_t end = a + (uintptr_t)(max_off + 1) * esz;
    for (const auto& r : regions)
      if (a >= r.first && a < r.first + r.second) {
        if (end <= r.first + r.second) return true;
        break;
      }
    char buf[256];
    snprintf(buf, sizeof(buf), "bounds check failed: %s (max offset %lld)", what, max_off);
    err = buf;
    return false;
  }

  cudaError_t cp(void* dst, const void* src, size_t bytes, cudaMemcpyKind k) {
    if (dry || bytes == 0) return cudaSuccess;
    return cudaMemcpyAsync(dst, src, bytes, k, st);
  }
  cudaError_t ms(void* dst, int v, size_t bytes) { return dry ? cudaSuccess : cudaMemsetAsync(dst, v, bytes, st); }
  cudaError_t sync() { return dry ? cudaSuccess : cudaStreamSynchronize(st); }
  cudaError_t cps(void* dst, const void* src, size_t bytes, cudaMemcpyKind k) {
    cudaError_t e = cp(dst, src, bytes, k);
    return e == cudaSuccess ? sync() : e;
  }

  int nbonds() const { return 2 * Lx * Ly - Lx - Ly; }

  void orig(int o, int kp, int mp, int& k, int& m) const {
    const Orient& Ob = O[o];
    const int kk = Ob.vf ? (Ob.Ly - 1 - kp) : kp;
    if (!Ob.tr) { k = kk; m = mp; } else { k = mp; m = kk; }
  }

  SiteOp site(int o, int kp, int mp) const {
    const Orient& Ob = O[o];
    SiteOp s;
    s.Dl = mp == 0 ? 1 : D;
    s.Dr = mp == Ob.Lx - 1 ? 1 : D;
    s.Du = kp == 0 ? 1 : D;
    s.Dd = kp == Ob.Ly - 1 ? 1 : D;
    s.size = (long long)s.Dl * s.Dr * s.Du * s.Dd;
    const long long off = perm_site_off[o][(size_t)kp * Ob.Lx + mp];
    s.lurd = perm[o][0] + off;
    s.urld = perm[o][1] + off;
    int k, m;
    orig(o, kp, mp, k, m);
    s.spin = k * Lx + m;
    return s;
  }

  View trivial_view() const { return View{ones, 0, 1, &trivial_bond, zeros_d}; }

  View view(const Store& s, int row, int slot) const {
    if (row == 0) return trivial_view();
    return View{s.row_ptr(slot, C, S), (long long)C * S, S, &s.bond[row], s.logs + (size_t)slot * C};
  }

  static long long scatter_max(int M, int c2, int c3, long long s1, long long s2, long long s3) {
    const int c23 = c2 * c3;
    return (long long)((M - 1) / c23) * s1 + (long long)(c2 - 1) * s2 + (long long)(c3 - 1) * s3;
  }

  // ----------------------------------------------- optional per-launch event timing
  bool prof = false;
  std::vector<cudaEvent_t> ev_pool;
  struct Pending { cudaEvent_t a, b; int kind; std::string shape; double flops; };
  struct ShapeStat { long long n = 0; double flops = 0, ms = 0; };
  std::map<std::string, ShapeStat> shape_stats;
  std::vector<Pending> pending;
  double prof_acc[6] = {0, 0, 0, 0, 0, 0};  // gemm launches, flops, ms, qr launches, qr ms, gemm bytes

  // Algorithmic bytes of one contraction launch: every FP32 operand read once (an
  // operand shared by all chains once, both spin slots of a selected site tensor), the
  // result written once (read and written when accumulating).
  double gemm_bytes(const GemmDesc& g) const {
    const double a = (g.bsA ? (double)C : 1.0) * g.M * g.K;
    const double b = (g.bsB ? (double)C : (g.sel ? 2.0 : 1.0)) * g.K * g.N;
    const double c = (g.accumulate ? 2.0 : 1.0) * C * (double)g.M * g.N;
    return 4.0 * (a + b + c);
  }

  cudaEvent_t ev() {
    if (ev_pool.empty()) {
      cudaEvent_t e;
      cudaEventCreate(&e);
      return e;
    }
    cudaEvent_t e = ev_pool.back();
    ev_pool.pop_back();
    return e;
  }
  cudaError_t collect() {
    if (pending.empty() || dry) return cudaSuccess;
    PV_CUDA(cudaEventSynchronize(pending.back().b));
    for (const Pending& p : pending) {
      float ms = 0.f;
      PV_CUDA(cudaEventElapsedTime(&ms, p.a, p.b));
      if (p.kind < 2) prof_acc[p.kind == 0 ? 2 : 4] += ms;  // kind 2: per-chain reductions (shape table only)
      ShapeStat& ss = shape_stats[p.shape];
      ss.n += 1;
      ss.flops += p.flops;
      ss.ms += ms;
      ev_pool.push_back(p.a);
      ev_pool.push_back(p.b);
    }
    pending.clear();
    return cudaSuccess;
  }
  template <typename F>
  cudaError_t timed(int kind, F&& launch, const std::string& shape = "", double flops = 0.0) {
    if (!prof || dry) return launch();
    cudaEvent_t a = ev(), b = ev();
    PV_CUDA(cudaEventRecord(a, st));
    PV_CUDA(launch());
    PV_CUDA(cudaEventRecord(b, st));
    pending.push_back({a, b, kind, shape, flops});
    if (pending.size() >= 16384) return collect();
    return cudaSuccess;
  }

  cudaError_t gemm(GemmDesc& g) {
    g.batch = C;
    if (g.M % (g.cm2 * g.cm3) || g.N % (g.cn2 * g.cn3)) {
      err = "contraction layout: scattered extents do not divide M or N";
      return cudaErrorInvalidValue;
    }
    const long long b1 = C - 1;
    if (!span(g.A, b1 * g.bsA + (long long)(g.M - 1) * g.sAm + (long long)(g.K - 1) * g.sAk, 4, "gemm A") ||
        !span(g.B, (g.sel ? g.ssB : 0) + b1 * g.bsB + (long long)(g.K - 1) * g.sBk + (long long)(g.N - 1) * g.sBn, 4,
              "gemm B") ||
        !span(g.C, b1 * g.bsC + scatter_max(g.M, g.cm2, g.cm3, g.sCm1, g.sCm2, g.sCm3) +
                       scatter_max(g.N, g.cn2, g.cn3, g.sCn1, g.sCn2, g.sCn3), 4, "gemm C") ||
        (g.sel && !span(g.sel, b1 * g.sel_stride, 1, "gemm spin selector")) ||
        (g.inv_scale && !span(g.inv_scale, b1, 8, "gemm scale")))
      return cudaErrorInvalidValue;
    ++launches;
    if (prof) {
      prof_acc[0] += 1;
      prof_acc[1] += 2.0 * g.M * g.N * g.K * (double)C;
      prof_acc[5] += gemm_bytes(g);
    }
    if (!prof) return launch_gemm(g);
    char key[96];
    snprintf(key, sizeof(key), "gemm %s M%d N%d K%d", tc_route(g) ? "tc" : "f32", g.M, g.N, g.K);
    return timed(0, [&] { return launch_gemm(g); }, key, 2.0 * g.M * g.N * g.K * (double)C);
  }

  // Tensor cores for contractions big enough to fill a 128-row tile, CUDA cores otherwise.
  int tc_mode() const {
    switch (cfg.precision) {
      case PEPSVMC_MIXED_BF16: return 2;
      case PEPSVMC_MIXED_BF16X3: return 3;
      case PEPSVMC_MIXED_TF32: return 4;
      default: return 0;
    }
  }
  bool tc_route(const GemmDesc& g) const {
    const auto it = tuned.find(tune_key(g));
    if (it != tuned.end()) return it->second >= 100;
    return tc_mode() && (long long)g.M * g.N * g.K >= kTcMinWork && g.M >= 64 && g.K >= 8;
  }

  // ---------------------------------------------------------------- autotuner
  // Per contraction shape (dims, strides, scatter), every candidate kernel -- the six
  // FP32 tile shapes and, in the tensor-core modes, the four TC tile widths -- is timed
  // once with CUDA events on its first use; the fastest is kept for the context.
  // Candidates compute the same product, so the timing runs are harmless.
  bool autotune = true;
  bool capturing = false;
  std::map<std::string, int> tuned;  // choice: f32 config, 100 + TC tile width, 1000 + two-stage split tile width
  std::map<std::string, std::vector<float>> tune_ms;

  static std::string tune_key(const GemmDesc& g) {
    char k[320];
    snprintf(k, sizeof(k), "%d %d %d|%lld %lld|%lld %lld %d|%d %d %lld %lld %lld|%d %d %lld %lld %lld", g.M, g.N, g.K,
             g.sAm, g.sAk, g.sBk, g.sBn, g.sel != nullptr, g.cm2, g.cm3, g.sCm1, g.sCm2, g.sCm3, g.cn2, g.cn3, g.sCn1,
             g.sCn2, g.sCn3);
    return k;
  }
  cudaError_t run_choice(const GemmDesc& g0, int choice) {
    GemmDesc g = g0;
    g.wait_cycles = wait_budget;
    if (choice >= 1000) return gemm_tc(g, 6, choice - 1000, status, st);  // split BF16, two stages
    if (choice >= 100) return gemm_tc(g, tc_mode(), choice - 100, status, st);
    return gemm_f32(g, choice, st);
  }
  cudaError_t tune(const GemmDesc& g, const std::string& key) {
    std::vector<int> cand;
    for (int c = 0; c < gemm_f32_num_configs(); ++c) cand.push_back(c);
    if (tc_mode() && g.K >= 8)
      for (int bn : {32, 64, 128, 256}) {
        if (bn / 2 < g.N || bn == 32) cand.push_back(100 + bn);
        // the double-buffered split form, for products with more than one K stage
        if (tc_mode() == 3 && bn <= 64 && g.K > 64 && (bn / 2 < g.N || bn == 32)) cand.push_back(1000 + bn);
      }
    cudaEvent_t e0 = ev(), e1 = ev();
    int best = -1;
    float best_ms = 0.f;
    std::vector<float> times;
    for (int c : cand) {
      PV_CUDA(run_choice(g, c));  // warm
      PV_CUDA(cudaEventRecord(e0, st));
      PV_CUDA(run_choice(g, c));
      PV_CUDA(cudaEventRecord(e1, st));
      PV_CUDA(cudaEventSynchronize(e1));
      float ms = 0.f;
      PV_CUDA(cudaEventElapsedTime(&ms, e0, e1));
      times.push_back(ms);
      if (best < 0 || ms < best_ms) {
        best = c;
        best_ms = ms;
      }
    }
    ev_pool.push_back(e0);
    ev_pool.push_back(e1);
    tuned[key] = best;
    tune_ms[key] = times;
    return cudaSuccess;
  }
  int forced = -1;  // a choice code fixed by pepsvmc_set_contraction_kernel, or -1
  cudaError_t launch_gemm(const GemmDesc& g) {
    if (forced >= 0) return run_choice(g, forced);
    if (!dry && (autotune || !tuned.empty())) {
      const std::string key = tune_key(g);
      auto it = tuned.find(key);
      if (it == tuned.end() && autotune && !capturing && !g.accumulate) {
        PV_CUDA(tune(g, key));
        it = tuned.find(key);
      }
      if (it != tuned.end()) return run_choice(g, it->second);
    }
    if (tc_mode() && (long long)g.M * g.N * g.K >= kTcMinWork && g.M >= 64 && g.K >= 8)
      return run_choice(g, 100);
    return gemm_f32(g, gemm_f32_pick(g), st);
  }
  static constexpr long long kTcMinWork = 1 << 15;

  cudaError_t qr(const float* Y, long long bsY, long long yrs, long long ycs, float* Q, long long bsQ, long long qrs,
                 long long qcs, int rows, int cols, int batch) {
    const long long b1 = batch - 1;
    if (!span(Y, b1 * bsY + (long long)(rows - 1) * yrs + (long long)(cols - 1) * ycs, 4, "qr input") ||
        !span(Q, b1 * bsQ + (long long)(rows - 1) * qrs + (long long)(cols - 1) * qcs, 4, "qr output"))
      return cudaErrorInvalidValue;
    if (rows < cols) {
      err = "qr: fewer rows than columns";
      return cudaErrorInvalidValue;
    }
    ++launches;
    if (prof) prof_acc[3] += 1;
    char key[64];
    snprintf(key, sizeof(key), "qr %dx%d", rows, cols);
    return timed(1, [&] { return qr_pos_batched(Y, bsY, yrs, ycs, Q, bsQ, qrs, qcs, rows, cols, batch, st); },
                 key, 0.0);
  }

  // Per-chain array span: chains 0..C-1 with stride bs, n entries each.
  bool chains(const void* p, long long bs, long long n, size_t esz, const char* what) {
    return span(p, (long long)(C - 1) * bs + n - 1, esz, what);
  }

  cudaError_t dot(const float* a, long long bsa, const float* b, long long bsb, int n, double* out) {
    if (!chains(a, bsa, n, 4, "dot a") || !chains(b, bsb, n, 4, "dot b") || !chains(out, 1, 1, 8, "dot out"))
      return cudaErrorInvalidValue;
    ++launches;
    return timed(2, [&] { return k_dot(a, bsa, b, bsb, n, out, C, status, st); }, "dot");
  }

  // rho_export (nullable): [chain][2][Ly][Lx] receives each NN ratio at (channel, site).
  float* rho_export = nullptr;
  cudaError_t ratio(const float* a, long long bsa, const float* b, long long bsb, int n, int si, int sj,
                    double halfJ, long long export_idx = -1) {
    if (!chains(a, bsa, n, 4, "ratio a") || !chains(b, bsb, n, 4, "ratio b") ||
        !chains(spins, (long long)Ly * Lx, (long long)std::max(si, sj) + 1, 1, "ratio spins"))
      return cudaErrorInvalidValue;
    ++launches;
    float* ro = (rho_export && export_idx >= 0) ? rho_export : nullptr;
    return timed(2, [&] {
      return k_ratio_accum(a, bsa, b, bsb, n, den, spins, (long long)Ly * Lx, si, sj, halfJ, eloc, C, status, st, ro,
                           2LL * Ly * Lx, export_idx);
    }, "ratio_accum");
  }

  cudaError_t logpsi_of(const float* x, long long bs, const double* logT, const double* logB) {
    if (!chains(x, bs, 1, 4, "logpsi x") || !chains(logT, 1, 1, 8, "logT") || !chains(logB, 1, 1, 8, "logB"))
      return cudaErrorInvalidValue;
    ++launches;
    return timed(2, [&] { return k_logpsi(x, bs, exps, logT, logB, logpsi, sign, C, status, st); }, "logpsi");
  }

  const int8_t* sel_base = nullptr;  // spin array the site tensors are selected from (default: spins)
  void sel(GemmDesc& g, const SiteOp& a, const float* base, int flip) const {
    g.B = base;
    g.ssB = a.size;
    g.bsB = 0;
    g.sel = (sel_base ? sel_base : spins) + a.spin;
    g.sel_stride = (long long)Ly * Lx;
    g.sel_xor = flip;
  }

  // --------------------------------------------------------- contractions
  // Fused three-line step (all three products in one tensor-core kernel, intermediates
  // on chip) for the tensor-core precisions; on by default, switchable for comparisons.
  bool fused_on = true;
  bool fused_ok(int cT, int cB, int cT2, int cB2, const SiteOp& a) const {
    return fused_on && forced < 0 && (tc_mode() == 2 || tc_mode() == 3) &&
           env3_fused_fits(cT, cB, cT2, cB2, a.Dl, a.Dr, a.Du, a.Dd);
  }
  bool spans3(const Env3Fused& f) {
    const long long b1 = f.batch - 1;
    return span(f.E, b1 * f.bsE + (f.cT - 1) * f.sEa + (f.Dl - 1) * f.sEl + (f.cB - 1) * f.sEb, 4, "fused E") &&
           span(f.T, b1 * f.bsT + (f.cT - 1) * f.sTa + (f.Du - 1) * f.sTu + (f.cT2 - 1) * f.sTa2, 4, "fused T") &&
           span(f.A, f.ssA + (f.Dl - 1) * f.sAl + (f.Du - 1) * f.sAu + (f.Dr - 1) * f.sAr + (f.Dd - 1) * f.sAd, 4,
                "fused A") &&
           span(f.B, b1 * f.bsB + (f.cB - 1) * f.sBb + (f.Dd - 1) * f.sBd + (f.cB2 - 1) * f.sBb2, 4, "fused B") &&
           span(f.out, b1 * f.bsO + (f.cT2 - 1) * f.sOa2 + (f.Dr - 1) * f.sOr + (f.cB2 - 1) * f.sOb2, 4, "fused out") &&
           (!f.sel || span(f.sel, b1 * f.sel_stride, 1, "fused spin selector"));
  }
  // caller_memory: the operands are the caller's (the C-ABI step), not the context's
  // allocations, so the context's bounds table does not cover them
  cudaError_t fused3(Env3Fused f, int batch = 0, bool caller_memory = false) {
    f.batch = batch > 0 ? batch : C;
    f.wait_cycles = wait_budget;
    if (!caller_memory && !spans3(f)) return cudaErrorInvalidValue;
    ++launches;
    const double nb = f.batch;
    const double flops = 2.0 * nb *
        ((double)f.Dl * f.cB * f.Du * f.cT2 * f.cT + (double)f.cB * f.cT2 * f.Dr * f.Dd * f.Dl * f.Du +
         (double)f.cT2 * f.Dr * f.cB2 * f.cB * f.Dd);
    if (prof) {
      prof_acc[0] += 1;
      prof_acc[1] += flops;
      // algorithmic bytes of the fused step: E, T, B and the result per chain, both slots of A once
      prof_acc[5] += 4.0 * ((f.bsE ? nb : 1.0) * f.cT * f.Dl * f.cB + (f.bsT ? nb : 1.0) * f.cT * f.Du * f.cT2 +
                            (f.bsB ? nb : 1.0) * f.cB * f.Dd * f.cB2 + nb * f.cT2 * f.Dr * f.cB2 +
                            2.0 * f.Dl * f.Du * f.Dr * f.Dd);
    }
    char key[96];
    snprintf(key, sizeof(key), "fused3 %d %d %d %d x %d %d %d %d", f.cT, f.cB, f.cT2, f.cB2, f.Dl, f.Dr, f.Du, f.Dd);
    const bool split = tc_mode() == 3;
    return timed(0, [&] { return env3_fused(f, split, status, st); }, key, flops);
  }
  // left step: E (cT,Dl,cB), T (cT,Du,cT2), B (cB,Dd,cB2) -> out (cT2,Dr,cB2)
  Env3Fused fused_left(const float* E, long long bsE, int cT, int cB, const float* T, long long bsT, int cT2,
                       const SiteOp& a, int flip, const float* B, long long bsB, int cB2, float* out,
                       long long bsO) const {
    Env3Fused f;
    f.cT = cT; f.cB = cB; f.cT2 = cT2; f.cB2 = cB2; f.Dl = a.Dl; f.Dr = a.Dr; f.Du = a.Du; f.Dd = a.Dd;
    f.E = E; f.bsE = bsE; f.sEa = (long long)a.Dl * cB; f.sEl = cB; f.sEb = 1;
    f.T = T; f.bsT = bsT; f.sTa = (long long)a.Du * cT2; f.sTu = cT2; f.sTa2 = 1;
    f.A = a.lurd; f.ssA = a.size;
    f.sAl = (long long)a.Du * a.Dr * a.Dd; f.sAu = (long long)a.Dr * a.Dd; f.sAr = a.Dd; f.sAd = 1;
    f.sel = (sel_base ? sel_base : spins) + a.spin; f.sel_stride = (long long)Ly * Lx; f.sel_xor = flip;
    f.B = B; f.bsB = bsB; f.sBb = (long long)a.Dd * cB2; f.sBd = cB2; f.sBb2 = 1;
    f.out = out; f.bsO = bsO; f.sOa2 = (long long)a.Dr * cB2; f.sOr = cB2; f.sOb2 = 1;
    return f;
  }
  // right step as a mirrored left step: E (cT2,Dr,cB2), T (cT,Du,cT2), B (cB,Dd,cB2) -> out (cT,Dl,cB)
  Env3Fused fused_right(const float* E, long long bsE, int cT2, int cB2, const float* T, long long bsT, int cT,
                        const SiteOp& a, int flip, const float* B, long long bsB, int cB, float* out,
                        long long bsO) const {
    Env3Fused f;
    f.cT = cT2; f.cB = cB2; f.cT2 = cT; f.cB2 = cB; f.Dl = a.Dr; f.Dr = a.Dl; f.Du = a.Du; f.Dd = a.Dd;
    f.E = E; f.bsE = bsE; f.sEa = (long long)a.Dr * cB2; f.sEl = cB2; f.sEb = 1;
    f.T = T; f.bsT = bsT; f.sTa = 1; f.sTu = cT2; f.sTa2 = (long long)a.Du * cT2;
    f.A = a.lurd; f.ssA = a.size;
    f.sAl = a.Dd; f.sAu = (long long)a.Dr * a.Dd; f.sAr = (long long)a.Du * a.Dr * a.Dd; f.sAd = 1;
    f.sel = (sel_base ? sel_base : spins) + a.spin; f.sel_stride = (long long)Ly * Lx; f.sel_xor = flip;
    f.B = B; f.bsB = bsB; f.sBb = 1; f.sBd = cB2; f.sBb2 = (long long)a.Dd * cB2;
    f.out = out; f.bsO = bsO; f.sOa2 = (long long)a.Dl * cB; f.sOr = cB; f.sOb2 = 1;
    return f;
  }

  // FP32 three-line step in one kernel (intermediates in shared memory): the same sums in the
  // same order as the separate products (rev: those of the right step).  out1: the result with
  // the other slot of the site, sharing E . T.
  bool f32_fused() const { return fused_on && forced < 0 && tc_mode() == 0; }
  bool f32_ok(const Env3Fused& f) const { return f32_fused() && env3_f32_fits(f); }
  cudaError_t step3_f32(Env3Fused f, float* out1, bool rev, int batch = 0, bool caller_memory = false) {
    f.batch = batch > 0 ? batch : C;
    if (!caller_memory) {
      Env3Fused g = f;
      g.out = out1 ? out1 : f.out;
      if (!spans3(f) || !spans3(g)) return cudaErrorInvalidValue;
    }
    ++launches;
    const double nb = f.batch, nv = out1 ? 2.0 : 1.0;
    const double flops = 2.0 * nb *
        ((double)f.Dl * f.cB * f.Du * f.cT2 * f.cT +
         nv * ((double)f.cB * f.cT2 * f.Dr * f.Dd * f.Dl * f.Du + (double)f.cT2 * f.Dr * f.cB2 * f.cB * f.Dd));
    if (prof) {
      prof_acc[0] += 1;
      prof_acc[1] += flops;
      prof_acc[5] += 4.0 * ((f.bsE ? nb : 1.0) * f.cT * f.Dl * f.cB + (f.bsT ? nb : 1.0) * f.cT * f.Du * f.cT2 +
                            (f.bsB ? nb : 1.0) * f.cB * f.Dd * f.cB2 + nv * nb * f.cT2 * f.Dr * f.cB2 +
                            2.0 * f.Dl * f.Du * f.Dr * f.Dd);
    }
    char key[96];
    snprintf(key, sizeof(key), "step3 f32 %d %d %d %d x %d %d %d %d", f.cT, f.cB, f.cT2, f.cB2, f.Dl, f.Dr, f.Du, f.Dd);
    return timed(0, [&] { return env3_f32(f, out1, rev, rev, Mid3(), st); }, key, flops);
  }
  // FP32 optimal site of the fit, Y (cV,Dd,cV2) = L . T . a . R, in one kernel: the same chain
  // of products with one of the boundary bonds in the place of a'.  From the left (the sums
  // and the copy in tmp2 are proj3's) that is v, from the right (proj3_right's) v2.
  Env3Fused proj_f32(bool right, const float* Lf, long long bsL, int cT, int cV, const float* T, long long bsT, int cT2,
                     const SiteOp& a, const float* Rf, long long bsR, int cV2, float* Y, long long bsY, Mid3& mid) const {
    const int Dl = a.Dl, Dr = a.Dr, Du = a.Du, Dd = a.Dd;
    Env3Fused f;
    f.A = a.lurd; f.ssA = a.size; f.sAl = (long long)Dr * Dd; f.sAr = 1;
    f.sel = (sel_base ? sel_base : spins) + a.spin; f.sel_stride = (long long)Ly * Lx;
    f.Dl = Du; f.Dr = Dd;
    f.E = T; f.bsE = bsT; f.sEl = cT2;
    f.out = Y; f.bsO = bsY; f.sOr = cV2;
    mid.p = tmp2; mid.bs = SI;
    if (!right) {
      f.cT = cT; f.cB = cT2; f.cT2 = cV; f.cB2 = cV2; f.Du = Dl; f.Dd = Dr;
      f.sEa = (long long)Du * cT2; f.sEb = 1;
      f.T = Lf; f.bsT = bsL; f.sTa = (long long)Dl * cV; f.sTu = cV; f.sTa2 = 1;
      f.sAu = (long long)Du * Dr * Dd; f.sAd = Dd;
      f.B = Rf; f.bsB = bsR; f.sBb = (long long)Dr * cV2; f.sBd = cV2; f.sBb2 = 1;
      f.sOa2 = (long long)Dd * cV2; f.sOb2 = 1;
      mid.sj = Dd * cT2 * Dr; mid.sr = cT2 * Dr; mid.sb = Dr; mid.sd = 1;
    } else {
      f.cT = cT2; f.cB = cT; f.cT2 = cV2; f.cB2 = cV; f.Du = Dr; f.Dd = Dl;
      f.sEa = 1; f.sEb = (long long)Du * cT2;
      f.T = Rf; f.bsT = bsR; f.sTa = (long long)Dr * cV2; f.sTu = cV2; f.sTa2 = 1;
      f.sAu = Dd; f.sAd = (long long)Du * Dr * Dd;
      f.B = Lf; f.bsB = bsL; f.sBb = (long long)Dl * cV; f.sBd = cV; f.sBb2 = 1;
      f.sOa2 = 1; f.sOb2 = (long long)Dd * cV2;
      mid.sj = 1; mid.sr = cV2; mid.sb = Dl * Dd * cV2; mid.sd = Dd * cV2;
    }
    return f;
  }
  cudaError_t proj_step_f32(Env3Fused f, const Mid3& mid, bool right) {
    f.batch = C;
    if (!spans3(f) || !chains(mid.p, mid.bs, (long long)f.cB * f.Dd * f.Dr * f.cT2, 4, "fit intermediate"))
      return cudaErrorInvalidValue;
    ++launches;
    const double nb = f.batch;
    const double flops = 2.0 * nb *
        ((double)f.Dl * f.cB * f.Du * f.cT2 * f.cT + (double)f.cB * f.cT2 * f.Dr * f.Dd * f.Dl * f.Du +
         (double)f.cT2 * f.Dr * f.cB2 * f.cB * f.Dd);
    if (prof) {
      prof_acc[0] += 1;
      prof_acc[1] += flops;
      prof_acc[5] += 4.0 * ((f.bsE ? nb : 1.0) * f.cT * f.Dl * f.cB + (f.bsT ? nb : 1.0) * f.cT * f.Du * f.cT2 +
                            (f.bsB ? nb : 1.0) * f.cB * f.Dd * f.cB2 + nb * f.cT2 * f.Dr * (f.cB2 + (double)f.cB * f.Dd) +
                            2.0 * f.Dl * f.Du * f.Dr * f.Dd);
    }
    char key[96];
    snprintf(key, sizeof(key), "proj f32 %d %d %d %d x %d %d %d %d", f.cT, f.cB, f.cT2, f.cB2, f.Dl, f.Dr, f.Du, f.Dd);
    return timed(0, [&] { return env3_f32(f, nullptr, !right, false, mid, st); }, key, flops);
  }
  // FP32 four-line step, one to four flip variants (see Env4Outs) of it in one kernel.
  cudaError_t step4_f32(Env4Fused f, const Env4Outs& o, bool rev) {
    f.batch = C;
    for (float* p : o.p) {
      f.out = p;
      if (p && !spans4(f)) return cudaErrorInvalidValue;
    }
    ++launches;
    const double nb = C, s1 = (double)f.D1l * f.D2l * f.cB * f.Du1 * f.cT2 * f.cT,
                 s2 = (double)f.D2l * f.cB * f.cT2 * f.D1r * f.Dd1 * f.D1l * f.Du1,
                 s34 = (double)f.cB * f.cT2 * f.D1r * f.D2r * f.Dd2 * f.D2l * f.Dd1 +
                       (double)f.cT2 * f.D1r * f.D2r * f.cB2 * f.cB * f.Dd2;
    const int n0 = (o.p[0] != nullptr) + (o.p[1] != nullptr), n1 = (o.p[2] != nullptr) + (o.p[3] != nullptr);
    const double flops = 2.0 * nb * (s1 + ((n0 > 0) + (n1 > 0)) * s2 + (n0 + n1) * s34);
    if (prof) {
      prof_acc[0] += 1;
      prof_acc[1] += flops;
      prof_acc[5] += 4.0 * ((f.bsE ? nb : 1.0) * f.cT * f.D1l * f.D2l * f.cB + (f.bsT ? nb : 1.0) * f.cT * f.Du1 * f.cT2 +
                            (f.bsB ? nb : 1.0) * f.cB * f.Dd2 * f.cB2 + (n0 + n1) * nb * f.cT2 * f.D1r * f.D2r * f.cB2 +
                            2.0 * f.D1l * f.Du1 * f.D1r * f.Dd1 + 2.0 * f.D2l * f.Dd1 * f.D2r * f.Dd2);
    }
    char key[96];
    snprintf(key, sizeof(key), "step4 f32 %d %d %d %d (%d)", f.cT, f.cB, f.cT2, f.cB2, n0 + n1);
    return timed(0, [&] { return env4_f32(f, o, rev, st); }, key, flops);
  }

  // Fused four-line step (four products in one tensor-core kernel).
  bool spans4(const Env4Fused& f) {
    const long long b1 = C - 1;
    return span(f.E, b1 * f.bsE + (f.cT - 1) * f.sEa + (f.D1l - 1) * f.sEl1 + (f.D2l - 1) * f.sEl2 + (f.cB - 1) * f.sEb, 4,
                "fused4 E") &&
           span(f.T, b1 * f.bsT + (f.cT - 1) * f.sTa + (f.Du1 - 1) * f.sTu + (f.cT2 - 1) * f.sTa2, 4, "fused4 T") &&
           span(f.A1, f.ss1 + (f.D1l - 1) * f.s1l + (f.Du1 - 1) * f.s1u + (f.D1r - 1) * f.s1r + (f.Dd1 - 1) * f.s1d, 4,
                "fused4 a1") &&
           span(f.A2, f.ss2 + (f.D2l - 1) * f.s2l + (f.Dd1 - 1) * f.s2u + (f.D2r - 1) * f.s2r + (f.Dd2 - 1) * f.s2d, 4,
                "fused4 a2") &&
           span(f.B, b1 * f.bsB + (f.cB - 1) * f.sBb + (f.Dd2 - 1) * f.sBd + (f.cB2 - 1) * f.sBb2, 4, "fused4 B") &&
           span(f.out, b1 * f.bsO + (f.cT2 - 1) * f.sOa2 + (f.D1r - 1) * f.sOr1 + (f.D2r - 1) * f.sOr2 + (f.cB2 - 1) * f.sOb2,
                4, "fused4 out") &&
           span(f.sel1, b1 * f.sel_stride, 1, "fused4 spin 1") && span(f.sel2, b1 * f.sel_stride, 1, "fused4 spin 2");
  }
  cudaError_t fused4(Env4Fused f) {
    f.batch = C;
    f.wait_cycles = wait_budget;
    if (!spans4(f)) return cudaErrorInvalidValue;
    ++launches;
    const double nb = C;
    const double flops = 2.0 * nb *
        ((double)f.D1l * f.D2l * f.cB * f.Du1 * f.cT2 * f.cT + (double)f.D2l * f.cB * f.cT2 * f.D1r * f.Dd1 * f.D1l * f.Du1 +
         (double)f.cB * f.cT2 * f.D1r * f.D2r * f.Dd2 * f.D2l * f.Dd1 + (double)f.cT2 * f.D1r * f.D2r * f.cB2 * f.cB * f.Dd2);
    if (prof) {
      prof_acc[0] += 1;
      prof_acc[1] += flops;
      prof_acc[5] += 4.0 * ((f.bsE ? nb : 1.0) * f.cT * f.D1l * f.D2l * f.cB + (f.bsT ? nb : 1.0) * f.cT * f.Du1 * f.cT2 +
                            (f.bsB ? nb : 1.0) * f.cB * f.Dd2 * f.cB2 + nb * f.cT2 * f.D1r * f.D2r * f.cB2 +
                            2.0 * f.D1l * f.Du1 * f.D1r * f.Dd1 + 2.0 * f.D2l * f.Dd1 * f.D2r * f.Dd2);
    }
    char key[96];
    snprintf(key, sizeof(key), "fused4 %d %d %d %d", f.cT, f.cB, f.cT2, f.cB2);
    const bool split = tc_mode() == 3;
    return timed(0, [&] { return env4_fused(f, split, status, st); }, key, flops);
  }
  bool fused4_ok(const Env4Fused& f) const {
    return fused_on && forced < 0 && (tc_mode() == 2 || tc_mode() == 3) && env4_fused_fits(f);
  }
  // Every four-line step of this context runs fused (all bonds within the kernel's
  // maxima): the four-line environments are then stored b-major, E(a,l1,l2,b) at
  // [b][a][l1][l2], so that the kernel's slices of consecutive b are contiguous.  The
  // consumers of these environments (dot, ratio, normalisation) are element-wise over
  // matching layouts, so only the fused steps see the order.
  bool four_bmajor() const {
    return fused_on && forced < 0 && (tc_mode() == 2 || tc_mode() == 3) && chi_x <= kFusedChi && D <= kFusedD;
  }
  // left step of rows (k,k+1): E (cT,D1l,D2l,cB), T (cT,Du1,cT2), B (cB,Dd2,cB2) -> out (cT2,D1r,D2r,cB2)
  Env4Fused fused4_left(const float* E, long long bsE, int cT, int cB, const float* T, long long bsT, int cT2,
                        const SiteOp& a1, int f1, const SiteOp& a2, int f2, const float* B, long long bsB, int cB2,
                        float* out, long long bsO) const {
    Env4Fused f;
    f.cT = cT; f.cB = cB; f.cT2 = cT2; f.cB2 = cB2;
    f.D1l = a1.Dl; f.D1r = a1.Dr; f.Du1 = a1.Du; f.Dd1 = a1.Dd; f.D2l = a2.Dl; f.D2r = a2.Dr; f.Dd2 = a2.Dd;
    f.E = E; f.bsE = bsE;
    if (four_bmajor()) {
      f.sEb = (long long)cT * a1.Dl * a2.Dl; f.sEa = (long long)a1.Dl * a2.Dl; f.sEl1 = a2.Dl; f.sEl2 = 1;
    } else {
      f.sEa = (long long)a1.Dl * a2.Dl * cB; f.sEl1 = (long long)a2.Dl * cB; f.sEl2 = cB; f.sEb = 1;
    }
    f.T = T; f.bsT = bsT; f.sTa = (long long)a1.Du * cT2; f.sTu = cT2; f.sTa2 = 1;
    f.A1 = a1.lurd; f.ss1 = a1.size;
    f.s1l = (long long)a1.Du * a1.Dr * a1.Dd; f.s1u = (long long)a1.Dr * a1.Dd; f.s1r = a1.Dd; f.s1d = 1;
    f.A2 = a2.lurd; f.ss2 = a2.size;
    f.s2l = (long long)a2.Du * a2.Dr * a2.Dd; f.s2u = (long long)a2.Dr * a2.Dd; f.s2r = a2.Dd; f.s2d = 1;
    const int8_t* sb = sel_base ? sel_base : spins;
    f.sel1 = sb + a1.spin; f.sel2 = sb + a2.spin; f.sel_stride = (long long)Ly * Lx; f.xor1 = f1; f.xor2 = f2;
    f.B = B; f.bsB = bsB; f.sBb = (long long)a2.Dd * cB2; f.sBd = cB2; f.sBb2 = 1;
    f.out = out; f.bsO = bsO;
    if (four_bmajor()) {
      f.sOb2 = (long long)cT2 * a1.Dr * a2.Dr; f.sOa2 = (long long)a1.Dr * a2.Dr; f.sOr1 = a2.Dr; f.sOr2 = 1;
    } else {
      f.sOa2 = (long long)a1.Dr * a2.Dr * cB2; f.sOr1 = (long long)a2.Dr * cB2; f.sOr2 = cB2; f.sOb2 = 1;
    }
    return f;
  }
  // right step as a mirrored left step: E (cT2,D1r,D2r,cB2) -> out (cT,D1l,D2l,cB)
  Env4Fused fused4_right(const float* E, long long bsE, int cT2, int cB2, const float* T, long long bsT, int cT,
                         const SiteOp& a1, int f1, const SiteOp& a2, int f2, const float* B, long long bsB, int cB,
                         float* out, long long bsO) const {
    Env4Fused f;
    f.cT = cT2; f.cB = cB2; f.cT2 = cT; f.cB2 = cB;
    f.D1l = a1.Dr; f.D1r = a1.Dl; f.Du1 = a1.Du; f.Dd1 = a1.Dd; f.D2l = a2.Dr; f.D2r = a2.Dl; f.Dd2 = a2.Dd;
    f.E = E; f.bsE = bsE;
    if (four_bmajor()) {
      f.sEb = (long long)cT2 * a1.Dr * a2.Dr; f.sEa = (long long)a1.Dr * a2.Dr; f.sEl1 = a2.Dr; f.sEl2 = 1;
    } else {
      f.sEa = (long long)a1.Dr * a2.Dr * cB2; f.sEl1 = (long long)a2.Dr * cB2; f.sEl2 = cB2; f.sEb = 1;
    }
    f.T = T; f.bsT = bsT; f.sTa = 1; f.sTu = cT2; f.sTa2 = (long long)a1.Du * cT2;
    f.A1 = a1.lurd; f.ss1 = a1.size;
    f.s1l = a1.Dd; f.s1u = (long long)a1.Dr * a1.Dd; f.s1r = (long long)a1.Du * a1.Dr * a1.Dd; f.s1d = 1;
    f.A2 = a2.lurd; f.ss2 = a2.size;
    f.s2l = a2.Dd; f.s2u = (long long)a2.Dr * a2.Dd; f.s2r = (long long)a2.Du * a2.Dr * a2.Dd; f.s2d = 1;
    const int8_t* sb = sel_base ? sel_base : spins;
    f.sel1 = sb + a1.spin; f.sel2 = sb + a2.spin; f.sel_stride = (long long)Ly * Lx; f.xor1 = f1; f.xor2 = f2;
    f.B = B; f.bsB = bsB; f.sBb = 1; f.sBd = cB2; f.sBb2 = (long long)a2.Dd * cB2;
    f.out = out; f.bsO = bsO;
    if (four_bmajor()) {
      f.sOb2 = (long long)cT * a1.Dl * a2.Dl; f.sOa2 = (long long)a1.Dl * a2.Dl; f.sOr1 = a2.Dl; f.sOr2 = 1;
    } else {
      f.sOa2 = (long long)a1.Dl * a2.Dl * cB; f.sOr1 = (long long)a2.Dl * cB; f.sOr2 = cB; f.sOb2 = 1;
    }
    return f;
  }

  // Fused optimal site of the fit: Y (cV,Dd,cV2) = L (cT,Dl,cV) . T (cT,Du,cT2) . a . R (cT2,Dr,cV2).
  bool proj_fused_ok(int cT, int cV, int cT2, int cV2, const SiteOp& a) const {
    return fused_ok(cT, cV, cT2, cV2, a);
  }
  cudaError_t fused_proj3(const float* Lf, long long bsL, int cT, int cV, const float* T, long long bsT, int cT2,
                          const SiteOp& a, const float* Rf, long long bsR, int cV2, float* Y, long long bsY) {
    Proj3Fused f;
    f.cT = cT; f.cV = cV; f.cT2 = cT2; f.cV2 = cV2; f.Dl = a.Dl; f.Dr = a.Dr; f.Du = a.Du; f.Dd = a.Dd;
    f.batch = C;
    f.L = Lf; f.bsL = bsL; f.sLa = (long long)a.Dl * cV; f.sLl = cV; f.sLv = 1;
    f.T = T; f.bsT = bsT; f.sTa = (long long)a.Du * cT2; f.sTu = cT2; f.sTa2 = 1;
    f.A = a.lurd; f.ssA = a.size;
    f.sAl = (long long)a.Du * a.Dr * a.Dd; f.sAu = (long long)a.Dr * a.Dd; f.sAr = a.Dd; f.sAd = 1;
    f.sel = (sel_base ? sel_base : spins) + a.spin; f.sel_stride = (long long)Ly * Lx;
    f.R = Rf; f.bsR = bsR; f.sRa = (long long)a.Dr * cV2; f.sRr = cV2; f.sRv = 1;
    f.out = Y; f.bsO = bsY; f.sOv = (long long)a.Dd * cV2; f.sOd = cV2; f.sOv2 = 1;
    f.wait_cycles = wait_budget;
    const long long b1 = C - 1;
    if (!span(f.L, b1 * f.bsL + (cT - 1) * f.sLa + (a.Dl - 1) * f.sLl + (cV - 1) * f.sLv, 4, "proj L") ||
        !span(f.T, b1 * f.bsT + (cT - 1) * f.sTa + (a.Du - 1) * f.sTu + (cT2 - 1) * f.sTa2, 4, "proj T") ||
        !span(f.A, f.ssA + (a.Dl - 1) * f.sAl + (a.Du - 1) * f.sAu + (a.Dr - 1) * f.sAr + (a.Dd - 1) * f.sAd, 4,
              "proj A") ||
        !span(f.R, b1 * f.bsR + (cT2 - 1) * f.sRa + (a.Dr - 1) * f.sRr + (cV2 - 1) * f.sRv, 4, "proj R") ||
        !span(f.out, b1 * f.bsO + (cV - 1) * f.sOv + (a.Dd - 1) * f.sOd + (cV2 - 1) * f.sOv2, 4, "proj out") ||
        !span(f.sel, b1 * f.sel_stride, 1, "proj spin selector"))
      return cudaErrorInvalidValue;
    ++launches;
    const double nb = C;
    const double flops = 2.0 * nb *
        ((double)a.Dl * cV * a.Du * cT2 * cT + (double)cV * cT2 * a.Dr * a.Dd * a.Dl * a.Du +
         (double)cV * a.Dd * cV2 * cT2 * a.Dr);
    if (prof) {
      prof_acc[0] += 1;
      prof_acc[1] += flops;
      prof_acc[5] += 4.0 * ((bsL ? nb : 1.0) * cT * a.Dl * cV + (bsT ? nb : 1.0) * cT * a.Du * cT2 +
                            (bsR ? nb : 1.0) * cT2 * a.Dr * cV2 + nb * cV * a.Dd * cV2 + 2.0 * a.size);
    }
    char key[96];
    snprintf(key, sizeof(key), "fusedP %d %d %d %d x %d %d %d %d", cT, cV, cT2, cV2, a.Dl, a.Dr, a.Du, a.Dd);
    const bool split = tc_mode() == 3;
    return timed(0, [&] { return proj3_fused(f, split, status, st); }, key, flops);
  }

  // Three-line left step (App. C, Fig. "contraction" (c)): E (cT,Dl,cB) -> out (cT2,Dr,cB2).
  cudaError_t left3(const float* E, long long bsE, int cT, int cB, const float* T, long long bsT, int cT2,
                    const SiteOp& a, int flip, const float* B, long long bsB, int cB2, float* out,
                    long long bsO) {
    if (fused_ok(cT, cB, cT2, cB2, a))
      return fused3(fused_left(E, bsE, cT, cB, T, bsT, cT2, a, flip, B, bsB, cB2, out, bsO));
    const Env3Fused f = fused_left(E, bsE, cT, cB, T, bsT, cT2, a, flip, B, bsB, cB2, out, bsO);
    if (f32_ok(f)) return step3_f32(f, nullptr, false);
    GemmDesc g[3];
    env3_left_descs(g, Env3Dims{cT, cB, cT2, cB2, a.Dl, a.Dr, a.Du, a.Dd}, E, bsE, T, bsT, a.lurd, a.size,
                    (sel_base ? sel_base : spins) + a.spin, (long long)Ly * Lx, flip, B, bsB, out, bsO, tmp1, tmp2, SI);
    for (int i = 0; i < 3; ++i) PV_CUDA(gemm(g[i]));
    return cudaSuccess;
  }
  // Left step for the configuration and, when out1 is given, with the spin of the site
  // flipped: the first product E . T does not depend on the spin and is done once;
  // tmp1 keeps it afterwards (delta3_after_left3 reads it; keep_et asks for it when the
  // fused kernel, which keeps E . T on chip, computes the step).
  cudaError_t left3_pair(const float* E, long long bsE, int cT, int cB, const float* T, long long bsT, int cT2,
                         const SiteOp& a, const float* B, long long bsB, int cB2, float* out0, float* out1,
                         long long bsO, bool keep_et = false) {
    GemmDesc g[3];
    const Env3Dims d{cT, cB, cT2, cB2, a.Dl, a.Dr, a.Du, a.Dd};
    if (fused_ok(cT, cB, cT2, cB2, a)) {
      PV_CUDA(fused3(fused_left(E, bsE, cT, cB, T, bsT, cT2, a, 0, B, bsB, cB2, out0, bsO)));
      if (out1) PV_CUDA(fused3(fused_left(E, bsE, cT, cB, T, bsT, cT2, a, 1, B, bsB, cB2, out1, bsO)));
      if (!keep_et) return cudaSuccess;
      env3_left_descs(g, d, E, bsE, T, bsT, a.lurd, a.size, (sel_base ? sel_base : spins) + a.spin, (long long)Ly * Lx, 0, B, bsB, out0,
                      bsO, tmp1, tmp2, SI);
      return gemm(g[0]);
    }
    env3_left_descs(g, d, E, bsE, T, bsT, a.lurd, a.size, (sel_base ? sel_base : spins) + a.spin, (long long)Ly * Lx, 0, B, bsB, out0, bsO,
                    tmp1, tmp2, SI);
    const Env3Fused f = fused_left(E, bsE, cT, cB, T, bsT, cT2, a, 0, B, bsB, cB2, out0, bsO);
    if (f32_ok(f)) {
      PV_CUDA(step3_f32(f, out1, false));
      return keep_et ? gemm(g[0]) : cudaSuccess;
    }
    for (int i = 0; i < 3; ++i) PV_CUDA(gemm(g[i]));
    if (!out1) return cudaSuccess;
    env3_left_descs(g, d, E, bsE, T, bsT, a.lurd, a.size, (sel_base ? sel_base : spins) + a.spin, (long long)Ly * Lx, 1, B, bsB, out1, bsO,
                    tmp1, tmp2, SI);
    PV_CUDA(gemm(g[1]));
    return gemm(g[2]);
  }

  // Three-line right step: E (cT2,Dr,cB2) -> out (cT,Dl,cB).
  cudaError_t right3(const float* E, long long bsE, int cT2, int cB2, const float* T, long long bsT, int cT,
                     const SiteOp& a, int flip, const float* B, long long bsB, int cB, float* out,
                     long long bsO) {
    if (fused_ok(cT2, cB2, cT, cB, a))
      return fused3(fused_right(E, bsE, cT2, cB2, T, bsT, cT, a, flip, B, bsB, cB, out, bsO));
    const Env3Fused f = fused_right(E, bsE, cT2, cB2, T, bsT, cT, a, flip, B, bsB, cB, out, bsO);
    if (f32_ok(f)) return step3_f32(f, nullptr, true);
    PV_CUDA(right3_head(E, bsE, cT2, cB2, T, bsT, cT, a, flip));
    return right3_tail(a, cT, cB2, B, bsB, cB, out, bsO);
  }
  // First two products of the right step: tmp2 [cT][Dl][Dd][cB2] = T . E . a (E on the right).
  cudaError_t right3_head(const float* E, long long bsE, int cT2, int cB2, const float* T, long long bsT, int cT,
                          const SiteOp& a, int flip, bool first = true) {
    const int Dl = a.Dl, Dr = a.Dr, Du = a.Du, Dd = a.Dd;
    GemmDesc g;
    g.M = cT * Du; g.N = Dr * cB2; g.K = cT2;
    g.A = T; g.sAm = cT2; g.sAk = 1; g.bsA = bsT;
    g.B = E; g.sBk = (long long)Dr * cB2; g.sBn = 1; g.bsB = bsE;
    g.C = tmp1; g.bsC = SI;
    g.cm2 = Du; g.sCm1 = (long long)cB2 * Du * Dr; g.sCm2 = Dr;
    g.cn2 = cB2; g.sCn1 = 1; g.sCn2 = (long long)Du * Dr;
    if (first) PV_CUDA(gemm(g));  // else tmp1 still holds T . E from the previous call
    GemmDesc h;
    h.M = cT * cB2; h.N = Dl * Dd; h.K = Du * Dr;
    h.A = tmp1; h.sAm = (long long)Du * Dr; h.sAk = 1; h.bsA = SI;
    sel(h, a, a.urld, flip); h.sBk = (long long)Dl * Dd; h.sBn = 1;
    h.C = tmp2; h.bsC = SI;
    h.cm2 = cB2; h.sCm1 = (long long)Dl * Dd * cB2; h.sCm2 = 1;
    h.cn2 = Dd; h.sCn1 = (long long)Dd * cB2; h.sCn2 = cB2;
    return gemm(h);
  }
  // Right step for the configuration and with the spin of the site flipped, sharing T . E.
  cudaError_t right3_pair(const float* E, long long bsE, int cT2, int cB2, const float* T, long long bsT, int cT,
                          const SiteOp& a, const float* B, long long bsB, int cB, float* out0, float* out1,
                          long long bsO) {
    if (fused_ok(cT2, cB2, cT, cB, a)) {
      PV_CUDA(fused3(fused_right(E, bsE, cT2, cB2, T, bsT, cT, a, 0, B, bsB, cB, out0, bsO)));
      return fused3(fused_right(E, bsE, cT2, cB2, T, bsT, cT, a, 1, B, bsB, cB, out1, bsO));
    }
    const Env3Fused f = fused_right(E, bsE, cT2, cB2, T, bsT, cT, a, 0, B, bsB, cB, out0, bsO);
    if (f32_ok(f)) return step3_f32(f, out1, true);
    PV_CUDA(right3_head(E, bsE, cT2, cB2, T, bsT, cT, a, 0));
    PV_CUDA(right3_tail(a, cT, cB2, B, bsB, cB, out0, bsO));
    PV_CUDA(right3_head(E, bsE, cT2, cB2, T, bsT, cT, a, 1, false));
    return right3_tail(a, cT, cB2, B, bsB, cB, out1, bsO);
  }
  // Last product of the right step: out (cT,Dl,cB) = tmp2 [cT][Dl][Dd][cB2] . B (cB,Dd,cB2).
  cudaError_t right3_tail(const SiteOp& a, int cT, int cB2, const float* B, long long bsB, int cB, float* out,
                          long long bsO) {
    const int Dl = a.Dl, Dd = a.Dd;
    GemmDesc q;
    q.M = cT * Dl; q.N = cB; q.K = Dd * cB2;
    q.A = tmp2; q.sAm = (long long)Dd * cB2; q.sAk = 1; q.bsA = SI;
    q.B = B; q.sBk = 1; q.sBn = (long long)Dd * cB2; q.bsB = bsB;
    q.C = out; q.bsC = bsO; q.sCm1 = cB; q.sCn1 = 1;
    return gemm(q);
  }
  // Last product of the left step from the fit's intermediate: after proj3, tmp2 holds
  // [cV][Dd][cT2][Dr] = L . T . a, so the new left environment of the fitted site V
  // (cV,Dd,cV2) is out (cT2,Dr,cV2) = tmp2 . V -- the step's first two products are
  // the optimal-site products already done.
  cudaError_t left3_tail_after_proj(const SiteOp& a, int cV, int cT2, const float* V, long long bsV, int cV2,
                                    float* out, long long bsO) {
    const int Dr = a.Dr, Dd = a.Dd;
    GemmDesc q;
    q.M = cT2 * Dr; q.N = cV2; q.K = cV * Dd;
    q.A = tmp2; q.sAm = 1; q.sAk = (long long)cT2 * Dr; q.bsA = SI;
    q.B = V; q.sBk = cV2; q.sBn = 1; q.bsB = bsV;
    q.C = out; q.bsC = bsO; q.sCm1 = cV2; q.sCn1 = 1;
    return gemm(q);
  }
  // Optimal site contracted from the right (for right-to-left half-sweeps): tmp2
  // [cT][Dl][Dd][cV2] = T . R . a as in the right step, then Y (cV,Dd,cV2) = L . tmp2;
  // right3_tail then gives the new right environment without repeating those products.
  cudaError_t proj3_right(const float* Lf, long long bsL, int cT, int cV, const float* T, long long bsT, int cT2,
                          const SiteOp& a, const float* Rf, long long bsR, int cV2, float* Y, long long bsY) {
    Mid3 mid;
    const Env3Fused f = proj_f32(true, Lf, bsL, cT, cV, T, bsT, cT2, a, Rf, bsR, cV2, Y, bsY, mid);
    if (f32_ok(f)) return proj_step_f32(f, mid, true);
    PV_CUDA(right3_head(Rf, bsR, cT2, cV2, T, bsT, cT, a, 0));
    const int Dl = a.Dl, Dd = a.Dd;
    GemmDesc q;
    q.M = Dd * cV2; q.N = cV; q.K = cT * Dl;
    q.A = tmp2; q.sAm = 1; q.sAk = (long long)Dd * cV2; q.bsA = SI;
    q.B = Lf; q.sBk = cV; q.sBn = 1; q.bsB = bsL;
    q.C = Y; q.bsC = bsY; q.sCm1 = 1; q.sCn1 = (long long)Dd * cV2;
    return gemm(q);
  }

  // Optimal site of the fit (App. B): Y (cV,Dd,cV2) = L (cT,Dl,cV) . T . a . R (cT2,Dr,cV2),
  // contracted from the left; tmp2 keeps L . T . a for left3_tail_after_proj.
  cudaError_t proj3(const float* Lf, long long bsL, int cT, int cV, const float* T, long long bsT, int cT2,
                    const SiteOp& a, const float* Rf, long long bsR, int cV2, float* Y, long long bsY) {
    Mid3 mid;
    const Env3Fused f = proj_f32(false, Lf, bsL, cT, cV, T, bsT, cT2, a, Rf, bsR, cV2, Y, bsY, mid);
    if (f32_ok(f)) return proj_step_f32(f, mid, false);
    const int Dl = a.Dl, Dr = a.Dr, Du = a.Du, Dd = a.Dd;
    GemmDesc g;
    g.M = Dl * cV; g.N = Du * cT2; g.K = cT;
    g.A = Lf; g.sAm = 1; g.sAk = (long long)Dl * cV; g.bsA = bsL;
    g.B = T; g.sBk = (long long)Du * cT2; g.sBn = 1; g.bsB = bsT;
    g.C = tmp1; g.bsC = SI;
    g.cm2 = cV; g.sCm1 = Du; g.sCm2 = (long long)cT2 * Dl * Du;
    g.cn2 = cT2; g.sCn1 = 1; g.sCn2 = (long long)Dl * Du;
    PV_CUDA(gemm(g));
    GemmDesc h;
    h.M = cV * cT2; h.N = Dr * Dd; h.K = Dl * Du;
    h.A = tmp1; h.sAm = (long long)Dl * Du; h.sAk = 1; h.bsA = SI;
    sel(h, a, a.lurd, 0); h.sBk = (long long)Dr * Dd; h.sBn = 1;
    h.C = tmp2; h.bsC = SI;
    h.cm2 = cT2; h.sCm1 = (long long)Dd * cT2 * Dr; h.sCm2 = Dr;
    h.cn2 = Dd; h.sCn1 = 1; h.sCn2 = (long long)cT2 * Dr;
    PV_CUDA(gemm(h));
    GemmDesc q;
    q.M = cV * Dd; q.N = cV2; q.K = cT2 * Dr;
    q.A = tmp2; q.sAm = (long long)cT2 * Dr; q.sAk = 1; q.bsA = SI;
    q.B = Rf; q.sBk = cV2; q.sBn = 1; q.bsB = bsR;
    q.C = Y; q.bsC = bsY; q.sCm1 = cV2; q.sCn1 = 1;
    return gemm(q);
  }

  // Defect network (Eq. (7)) divided by Psi, G[l][r][u][d] = L.T.B.R / den, after
  // left3_pair on the same site: tmp1 holds L . T as [cB][cT2][Dl][Du].
  cudaError_t delta3_after_left3(int cB, int cT2, const SiteOp& a, const float* B, long long bsB, int cB2,
                                 const float* Rf, long long bsR, const double* dn, float* Gout, long long bsG) {
    const int Dl = a.Dl, Dr = a.Dr, Du = a.Du, Dd = a.Dd;
    GemmDesc p;
    p.M = cB * Dd; p.N = cT2 * Dr; p.K = cB2;
    p.A = B; p.sAm = cB2; p.sAk = 1; p.bsA = bsB;
    p.B = Rf; p.sBk = 1; p.sBn = cB2; p.bsB = bsR;
    p.C = tmp2; p.bsC = SI;
    p.cm2 = Dd; p.sCm1 = (long long)cT2 * Dd * Dr; p.sCm2 = Dr;
    p.cn2 = Dr; p.sCn1 = (long long)Dd * Dr; p.sCn2 = 1;
    PV_CUDA(gemm(p));
    GemmDesc q;
    q.M = Dl * Du; q.N = Dd * Dr; q.K = cB * cT2;
    q.A = tmp1; q.sAm = 1; q.sAk = (long long)Dl * Du; q.bsA = SI;
    q.B = tmp2; q.sBk = (long long)Dd * Dr; q.sBn = 1; q.bsB = SI;
    q.C = Gout; q.bsC = bsG;
    q.cm2 = Du; q.sCm1 = (long long)Dr * Du * Dd; q.sCm2 = Dd;
    q.cn2 = Dr; q.sCn1 = 1; q.sCn2 = (long long)Du * Dd;
    q.inv_scale = dn;
    return gemm(q);
  }

  // Four-line left step of rows (k, k+1): E (cT,D1l,D2l,cB) -> out (cT2,D1r,D2r,cB2),
  // as four products: (1) E . T -> X; (2) X . a1 -> Y; (3) Y . a2 -> Z; (4) Z . B -> out.
  // Only (2) depends on the spin of (k, m) and only (3) on that of (k+1, m), so the
  // measurement shares (1) over its four spin-flip variants and (2) over pairs of them.
  cudaError_t left4(const float* E, long long bsE, int cT, int cB, const float* T, long long bsT, int cT2,
                    const SiteOp& a1, int f1, const SiteOp& a2, int f2, const float* B, long long bsB, int cB2,
                    float* out, long long bsO) {
    if (four_bmajor())
      return fused4(fused4_left(E, bsE, cT, cB, T, bsT, cT2, a1, f1, a2, f2, B, bsB, cB2, out, bsO));
    const Env4Fused f = fused4_left(E, bsE, cT, cB, T, bsT, cT2, a1, f1, a2, f2, B, bsB, cB2, out, bsO);
    const Env4Outs o{{out}};
    if (f32_fused() && env4_f32_takes(f, o, C)) return step4_f32(f, o, false);
    PV_CUDA(left4_x(E, bsE, cT, cB, T, bsT, cT2, a1, a2, tmp1));
    PV_CUDA(left4_y(tmp1, cB, cT2, a1, f1, a2, tmp2));
    return left4_zw(tmp2, cB, cT2, a1, a2, f2, B, bsB, cB2, out, bsO, tmp1);
  }
  // (1): X [(D2l,cB)][cT2][D1l][Du1] = E . T over cT.
  cudaError_t left4_x(const float* E, long long bsE, int cT, int cB, const float* T, long long bsT, int cT2,
                      const SiteOp& a1, const SiteOp& a2, float* X) {
    const int D1l = a1.Dl, Du1 = a1.Du, D2l = a2.Dl;
    GemmDesc g;
    g.M = D1l * D2l * cB; g.N = Du1 * cT2; g.K = cT;
    g.A = E; g.sAm = 1; g.sAk = (long long)D1l * D2l * cB; g.bsA = bsE;
    g.B = T; g.sBk = (long long)Du1 * cT2; g.sBn = 1; g.bsB = bsT;
    g.C = X; g.bsC = SI;
    g.cm2 = D2l * cB; g.sCm1 = Du1; g.sCm2 = (long long)cT2 * D1l * Du1;
    g.cn2 = cT2; g.sCn1 = 1; g.sCn2 = (long long)D1l * Du1;
    return gemm(g);
  }
  // (2): Y [(cB,cT2)][D1r][D2l][Dd1] = X . a1 (spin of (k, m), flipped when f1).
  cudaError_t left4_y(const float* X, int cB, int cT2, const SiteOp& a1, int f1, const SiteOp& a2, float* Y) {
    const int D1l = a1.Dl, D1r = a1.Dr, Du1 = a1.Du, Dd1 = a1.Dd, D2l = a2.Dl;
    GemmDesc h;
    h.M = D2l * cB * cT2; h.N = D1r * Dd1; h.K = D1l * Du1;
    h.A = X; h.sAm = (long long)D1l * Du1; h.sAk = 1; h.bsA = SI;
    sel(h, a1, a1.lurd, f1); h.sBk = (long long)D1r * Dd1; h.sBn = 1;
    h.C = Y; h.bsC = SI;
    h.cm2 = cB * cT2; h.sCm1 = Dd1; h.sCm2 = (long long)D1r * D2l * Dd1;
    h.cn2 = Dd1; h.sCn1 = (long long)D2l * Dd1; h.sCn2 = 1;
    return gemm(h);
  }
  // (3) and (4): Z = Y . a2 (spin of (k+1, m), flipped when f2) into scratch, out = Z . B.
  cudaError_t left4_zw(const float* Y, int cB, int cT2, const SiteOp& a1, const SiteOp& a2, int f2,
                       const float* B, long long bsB, int cB2, float* out, long long bsO, float* scratch) {
    const int D1r = a1.Dr, Dd1 = a1.Dd, D2l = a2.Dl, D2r = a2.Dr, Dd2 = a2.Dd;
    GemmDesc q;
    q.M = cB * cT2 * D1r; q.N = D2r * Dd2; q.K = D2l * Dd1;
    q.A = Y; q.sAm = (long long)D2l * Dd1; q.sAk = 1; q.bsA = SI;
    sel(q, a2, a2.lurd, f2); q.sBk = (long long)D2r * Dd2; q.sBn = 1;
    q.C = scratch; q.bsC = SI;
    q.cm2 = cT2 * D1r; q.sCm1 = Dd2; q.sCm2 = (long long)D2r * cB * Dd2;
    q.cn2 = Dd2; q.sCn1 = (long long)cB * Dd2; q.sCn2 = 1;
    PV_CUDA(gemm(q));
    GemmDesc w;
    w.M = cT2 * D1r * D2r; w.N = cB2; w.K = cB * Dd2;
    w.A = scratch; w.sAm = (long long)cB * Dd2; w.sAk = 1; w.bsA = SI;
    w.B = B; w.sBk = cB2; w.sBn = 1; w.bsB = bsB;
    w.C = out; w.bsC = bsO; w.sCm1 = cB2; w.sCn1 = 1;
    return gemm(w);
  }

  // Four-line right step: E (cT2,D1r,D2r,cB2) -> out (cT,D1l,D2l,cB).
  cudaError_t right4(const float* E, long long bsE, int cT2, int cB2, const float* T, long long bsT, int cT,
                     const SiteOp& a1, int f1, const SiteOp& a2, int f2, const float* B, long long bsB, int cB,
                     float* out, long long bsO) {
    if (four_bmajor())
      return fused4(fused4_right(E, bsE, cT2, cB2, T, bsT, cT, a1, f1, a2, f2, B, bsB, cB, out, bsO));
    const Env4Fused f = fused4_right(E, bsE, cT2, cB2, T, bsT, cT, a1, f1, a2, f2, B, bsB, cB, out, bsO);
    const Env4Outs o{{out}};
    if (f32_fused() && env4_f32_takes(f, o, C)) return step4_f32(f, o, true);
    const int D1l = a1.Dl, D1r = a1.Dr, Du1 = a1.Du, Dd1 = a1.Dd;
    const int D2l = a2.Dl, D2r = a2.Dr, Dd2 = a2.Dd;
    GemmDesc g;
    g.M = cT * Du1; g.N = D1r * D2r * cB2; g.K = cT2;
    g.A = T; g.sAm = cT2; g.sAk = 1; g.bsA = bsT;
    g.B = E; g.sBk = (long long)D1r * D2r * cB2; g.sBn = 1; g.bsB = bsE;
    g.C = tmp1; g.bsC = SI;
    g.cm2 = Du1; g.sCm1 = (long long)D2r * cB2 * Du1 * D1r; g.sCm2 = D1r;
    g.cn2 = D2r * cB2; g.sCn1 = 1; g.sCn2 = (long long)Du1 * D1r;
    PV_CUDA(gemm(g));
    GemmDesc h;
    h.M = cT * D2r * cB2; h.N = D1l * Dd1; h.K = Du1 * D1r;
    h.A = tmp1; h.sAm = (long long)Du1 * D1r; h.sAk = 1; h.bsA = SI;
    sel(h, a1, a1.urld, f1); h.sBk = (long long)D1l * Dd1; h.sBn = 1;
    h.C = tmp2; h.bsC = SI;
    h.cm2 = D2r; h.cm3 = cB2;
    h.sCm1 = (long long)D1l * cB2 * Dd1 * D2r; h.sCm2 = 1; h.sCm3 = (long long)Dd1 * D2r;
    h.cn2 = Dd1; h.sCn1 = (long long)cB2 * Dd1 * D2r; h.sCn2 = D2r;
    PV_CUDA(gemm(h));
    GemmDesc q;
    q.M = cT * D1l * cB2; q.N = D2l * Dd2; q.K = Dd1 * D2r;
    q.A = tmp2; q.sAm = (long long)Dd1 * D2r; q.sAk = 1; q.bsA = SI;
    sel(q, a2, a2.urld, f2); q.sBk = (long long)D2l * Dd2; q.sBn = 1;
    q.C = tmp1; q.bsC = SI;
    q.cm2 = cB2; q.sCm1 = (long long)D2l * Dd2 * cB2; q.sCm2 = 1;
    q.cn2 = Dd2; q.sCn1 = (long long)Dd2 * cB2; q.sCn2 = cB2;
    PV_CUDA(gemm(q));
    GemmDesc w;
    w.M = cT * D1l * D2l; w.N = cB; w.K = Dd2 * cB2;
    w.A = tmp1; w.sAm = (long long)Dd2 * cB2; w.sAk = 1; w.bsA = SI;
    w.B = B; w.sBk = 1; w.sBn = (long long)Dd2 * cB2; w.bsB = bsB;
    w.C = out; w.bsC = bsO; w.sCm1 = cB; w.sCn1 = 1;
    return gemm(w);
  }

  cudaError_t norm2(float* x, long long bs, int n, float* x2 = nullptr, int n2 = 0, float* x3 = nullptr,
                    int n3 = 0, int* ex = nullptr) {
    if (!chains(x, bs, n, 4, "normalize x") || (x2 && !chains(x2, bs, n2, 4, "normalize x2")) ||
        (x3 && !chains(x3, bs, n3, 4, "normalize x3")))
      return cudaErrorInvalidValue;
    ++launches;
    return timed(2, [&] { return k_normalize_pow2(x, bs, n, x2, bs, n2, x3, bs, n3, ex, C, status, st); },
                 "normalize_pow2");
  }

  // ------------------------------------------------------ boundary MPS (App. B)
  const Sketch& sketch_for(const std::vector<int>& vb, const std::vector<int>& p, cudaError_t& e) {
    std::string key;
    for (int v : vb) key += std::to_string(v) + ",";
    key += "|";
    for (int v : p) key += std::to_string(v) + ",";
    auto it = sketches.find(key);
    e = cudaSuccess;
    if (it != sketches.end()) return it->second;
    Sketch sk;
    const int L = (int)p.size();
    std::vector<float> host;
    for (int m = 0; m < L; ++m) {
      sk.off.push_back((long long)host.size());
      for (int a = 0; a < vb[m]; ++a)
        for (int d = 0; d < p[m]; ++d)
          for (int b = 0; b < vb[m + 1]; ++b)
            host.push_back((float)sketch_host[(((size_t)m * chi_x + a) * D + d) * chi_x + b]);
    }
    if ((e = alloc(&sk.dev, host.size())) != cudaSuccess) return sketches[key];
    if ((e = cp(sk.dev, host.data(), host.size() * sizeof(float), cudaMemcpyHostToDevice)) != cudaSuccess)
      return sketches[key];
    // right-orthonormal rows for sites m >= 1: QR of the transposed site, Q^T written back
    for (int m = 1; m < L; ++m) {
      const int rows = p[m] * vb[m + 1], cols = vb[m];
      float* s = sk.dev + sk.off[m];
      if ((e = qr(s, 0, 1, rows, s, 0, 1, rows, rows, cols, 1)) != cudaSuccess) return sketches[key];
    }
    e = sync();
    return sketches[key] = sk;
  }

  // V = fit(M_k |Tin>) into store row `slot`, bonds recorded as store.bond[row].
  cudaError_t compress(int o, int k, const View& Tin, Store& out, int row, int slot) {
    const Orient& Ob = O[o];
    const int L = Ob.Lx;
    const std::vector<int>& tb = *Tin.bond;
    std::vector<int> p(L), chiX(L > 1 ? L - 1 : 0);
    std::vector<SiteOp> a(L);
    for (int m = 0; m < L; ++m) {
      a[m] = site(o, k, m);
      p[m] = a[m].Dd;
      if (m < L - 1) chiX[m] = tb[m + 1] * a[m].Dr;
    }
    const std::vector<int> r = bond_caps(chiX, p, chi);
    std::vector<int> vb(L + 1, 1);
    for (int m = 0; m < L - 1; ++m) vb[m + 1] = r[m];
    out.bond[row] = vb;
    cudaError_t e;
    const Sketch& W = sketch_for(vb, p, e);
    PV_CUDA(e);
    float* Vb = out.row_ptr(slot, C, S);
    const long long vss = (long long)C * S;
    double* log_out = out.logs + (size_t)slot * C;
    auto envLp = [&](int m) { return envL + (long long)m * C * S; };
    auto envRp = [&](int m) { return envR + (long long)m * C * S; };
    // right environments of the starting guess
    for (int m = L - 1; m >= 1; --m) {
      const bool edge = (m == L - 1);
      PV_CUDA(right3(edge ? ones : envRp(m + 1), edge ? 1 : S, tb[m + 1], vb[m + 1], Tin.site(m),
                     Tin.chain_stride, tb[m], a[m], 0, W.dev + W.off[m], 0, vb[m], envRp(m), S));
      PV_CUDA(norm2(envRp(m), S, tb[m] * a[m].Dl * vb[m]));
    }
    for (int sw = 0; sw < nfit; ++sw) {
      if (sw % 2 == 0) {
        PV_CUDA(ms(exps, 0, C * sizeof(int)));
        for (int m = 0; m < L; ++m) {
          const float* Lin = m == 0 ? ones : envLp(m);
          const long long bsL = m == 0 ? 1 : S;
          const float* Rin = m == L - 1 ? ones : envRp(m + 1);
          const long long bsR = m == L - 1 ? 1 : S;
          float* Vs = Vb + m * vss;
          // fused: the optimal site in one kernel, then the new left environment as a full
          // three-line step with the fitted site as the bottom MPS (its first two products
          // are not kept on chip between the two kernels)
          const bool fz = proj_fused_ok(tb[m], vb[m], tb[m + 1], vb[m + 1], a[m]);
          if (fz)
            PV_CUDA(fused_proj3(Lin, bsL, tb[m], vb[m], Tin.site(m), Tin.chain_stride, tb[m + 1], a[m], Rin, bsR,
                                vb[m + 1], Vs, S));
          else
            PV_CUDA(proj3(Lin, bsL, tb[m], vb[m], Tin.site(m), Tin.chain_stride, tb[m + 1], a[m], Rin, bsR,
                          vb[m + 1], Vs, S));
          if (m < L - 1) {
            PV_CUDA(qr(Vs, S, vb[m + 1], 1, Vs, S, vb[m + 1], 1, vb[m] * p[m], vb[m + 1], C));
            if (fz)
              PV_CUDA(left3(Lin, bsL, tb[m], vb[m], Tin.site(m), Tin.chain_stride, tb[m + 1], a[m], 0, Vs, S,
                            vb[m + 1], envLp(m + 1), S));
            else
              PV_CUDA(left3_tail_after_proj(a[m], vb[m], tb[m + 1], Vs, S, vb[m + 1], envLp(m + 1), S));
            PV_CUDA(norm2(envLp(m + 1), S, tb[m + 1] * a[m].Dr * vb[m + 1], nullptr, 0, nullptr, 0, exps));
          }
        }
      } else {
        for (int m = L - 1; m >= 0; --m) {
          const float* Lin = m == 0 ? ones : envLp(m);
          const long long bsL = m == 0 ? 1 : S;
          const float* Rin = m == L - 1 ? ones : envRp(m + 1);
          const long long bsR = m == L - 1 ? 1 : S;
          float* Vs = Vb + m * vss;
          const bool fz = proj_fused_ok(tb[m], vb[m], tb[m + 1], vb[m + 1], a[m]);
          if (fz)
            PV_CUDA(fused_proj3(Lin, bsL, tb[m], vb[m], Tin.site(m), Tin.chain_stride, tb[m + 1], a[m], Rin, bsR,
                                vb[m + 1], Vs, S));
          else
            PV_CUDA(proj3_right(Lin, bsL, tb[m], vb[m], Tin.site(m), Tin.chain_stride, tb[m + 1], a[m], Rin,
                                bsR, vb[m + 1], Vs, S));
          if (m > 0) {
            const int rows = p[m] * vb[m + 1];
            PV_CUDA(qr(Vs, S, 1, rows, Vs, S, 1, rows, rows, vb[m], C));
            if (fz)
              PV_CUDA(right3(Rin, bsR, tb[m + 1], vb[m + 1], Tin.site(m), Tin.chain_stride, tb[m], a[m], 0, Vs, S,
                             vb[m], envRp(m), S));
            else
              PV_CUDA(right3_tail(a[m], tb[m], vb[m + 1], Vs, S, vb[m], envRp(m), S));
            PV_CUDA(norm2(envRp(m), S, tb[m] * a[m].Dl * vb[m]));
          }
        }
      }
    }
    float* center = Vb + (long long)(L - 1) * vss;
    if (!chains(center, S, vb[L - 1] * p[L - 1], 4, "mps centre") || !chains(log_out, 1, 1, 8, "mps log") ||
        !chains(Tin.logs, 1, 1, 8, "mps log in"))
      return cudaErrorInvalidValue;
    ++launches;
    return timed(2, [&] { return k_mps_normalize(center, S, vb[L - 1] * p[L - 1], exps, Tin.logs, log_out, C,
                                                 status, st); }, "mps_normalize");
  }

  // All top environments of orientation o (rows 1..Ly_o-1 into store, one slot per row).
  cudaError_t top_down_all(int o, Store& s) {
    for (int k = 0; k + 1 < O[o].Ly; ++k) PV_CUDA(compress(o, k, view(s, k, k), s, k + 1, k + 1));
    return cudaSuccess;
  }

  // ------------------------ spin-inversion symmetrised sampling (end of Sec. II B)
  // Chains p and p + pairs hold S and S-bar.  At the start of each phase w of every
  // chain is taken afresh from the two amplitudes closed at row 0 of the phase's lattice
  // (trivial top, the phase's bottom environment of row 0 at the sampler's cutoff), then
  // carried through the phase by k_phi_decide.
  bool sym = false;
  int pairs = 0;
  double *phi_rho = nullptr, *phi_w = nullptr, *phi_wm = nullptr, *eloc_phi = nullptr, *phi_wt = nullptr;
  double* phi_lp = nullptr;
  int8_t* phi_sg = nullptr;
  int* phi_exps = nullptr;
  cudaError_t phase_weight(int o, Store& top, Store& bot) {
    const Orient& Ob = O[o];
    const View T = view(top, 0, 0);
    const View B = view(bot, Ob.Ly - 1, Ob.Ly - 1);
    const std::vector<int>& tb = *T.bond;
    const std::vector<int>& bb = *B.bond;
    PV_CUDA(ms(phi_exps, 0, C * sizeof(int)));
    const float* Lin = ones;
    long long bsL = 1;
    for (int m = 0; m < Ob.Lx; ++m) {
      const SiteOp a = site(o, 0, m);
      float* cur = l3[(m + 1) % 2];
      PV_CUDA(left3(Lin, bsL, tb[m], bb[m], T.site(m), T.chain_stride, tb[m + 1], a, 0, B.site(m),
                    B.chain_stride, bb[m + 1], cur, S));
      if (m + 1 < Ob.Lx) {
        PV_CUDA(norm2(cur, S, tb[m + 1] * a.Dr * bb[m + 1], nullptr, 0, nullptr, 0, phi_exps));
      } else {
        if (!chains(cur, S, 1, 4, "phase amplitude") || !chains(T.logs, 1, 1, 8, "logT") ||
            !chains(B.logs, 1, 1, 8, "logB"))
          return cudaErrorInvalidValue;
        launches += 2;
        PV_CUDA(k_logpsi(cur, S, phi_exps, T.logs, B.logs, phi_lp, phi_sg, C, status, st));
        PV_CUDA(k_phi_combine(phi_lp, phi_sg, nullptr, C, pairs, phi_w, nullptr, nullptr, status, st));
      }
      Lin = cur;
      bsL = S;
    }
    return cudaSuccess;
  }

  // --------------------------------------------- sequential sweep (Sec. II A, Eq. (9))
  // Horizontal bonds of every row of orientation o.  `top` receives T_k (slot = row, or
  // row % 2 when `pingpong`), `bot` must hold the top environments of the upside-down
  // orientation for the configuration at the start of the phase.
  cudaError_t row_phase(int o, Store& top, bool pingpong, Store& bot, int bond_base) {
    const Orient& Ob = O[o];
    const int Lyo = Ob.Ly, Lxo = Ob.Lx;
    auto slot_of = [&](int row) { return pingpong ? (row % 2) : row; };
    auto envRp = [&](int m) { return envR + (long long)m * C * S; };
    auto envRfp = [&](int m) { return envRf + (long long)m * C * S; };
    if (sym) PV_CUDA(phase_weight(o, top, bot));
    for (int k = 0; k < Lyo; ++k) {
      const View T = view(top, k, slot_of(k));
      const int kb = Lyo - 1 - k;
      const View B = view(bot, kb, kb);
      const std::vector<int>& tb = *T.bond;
      const std::vector<int>& bb = *B.bond;
      std::vector<SiteOp> a(Lxo);
      for (int m = 0; m < Lxo; ++m) a[m] = site(o, k, m);
      for (int m = Lxo - 1; m >= 1; --m) {
        const bool edge = (m == Lxo - 1);
        const float* Ein = edge ? ones : envRp(m + 1);
        const long long bsE = edge ? 1 : S;
        PV_CUDA(right3_pair(Ein, bsE, tb[m + 1], bb[m + 1], T.site(m), T.chain_stride, tb[m], a[m], B.site(m),
                            B.chain_stride, bb[m], envRp(m), envRfp(m), S));
        const int n = tb[m] * a[m].Dl * bb[m];
        PV_CUDA(norm2(envRp(m), S, n, envRfp(m), n));
      }
      const float* Lin = ones;
      long long bsL = 1;
      for (int m = 0; m + 1 < Lxo; ++m) {
        PV_CUDA(left3_pair(Lin, bsL, tb[m], bb[m], T.site(m), T.chain_stride, tb[m + 1], a[m], B.site(m),
                           B.chain_stride, bb[m + 1], l3[1], fl, S));
        MetropolisArgs ma{};
        ma.cur = l3[1]; ma.bs_cur = S;
        ma.Rcur = envRp(m + 1); ma.bs_Rcur = S;
        ma.flip = fl; ma.bs_flip = S;
        ma.Rflip = envRfp(m + 1); ma.bs_Rflip = S;
        ma.n = tb[m + 1] * a[m].Dr * bb[m + 1];
        ma.spins = spins; ma.spin_stride = (long long)Ly * Lx;
        ma.site_a = a[m].spin; ma.site_b = a[m + 1].spin;
        ma.key = cfg.seed; ma.sweep = d_sweep; ma.chain_base = chain_base;
        ma.bond = bond_base + k * (Lxo - 1) + m;
        ma.out = l3[0]; ma.bs_out = S;
        ma.trace_ratio = trace_on ? trace_ratio : nullptr;
        ma.trace_dec = trace_on ? trace_dec : nullptr;
        ma.trace_stride = nbonds();
        ma.counters = counters; ma.status = status;
        if (!chains(ma.cur, S, ma.n, 4, "metropolis cur") || !chains(ma.Rcur, S, ma.n, 4, "metropolis R") ||
            !chains(ma.flip, S, ma.n, 4, "metropolis flip") || !chains(ma.Rflip, S, ma.n, 4, "metropolis Rf") ||
            !chains(ma.out, S, ma.n, 4, "metropolis out") ||
            !chains(spins, ma.spin_stride, std::max(ma.site_a, ma.site_b) + 1, 1, "metropolis spins") ||
            (ma.trace_ratio && !chains(ma.trace_ratio, nbonds(), ma.bond + 1, 8, "trace")))
          return cudaErrorInvalidValue;
        if (sym) {
          ma.rho_out = phi_rho;
          ma.phi_w = phi_w;
          ma.pairs = pairs;
          launches += 2;
          PV_CUDA(timed(2, [&] { return k_metropolis(ma, C, st); }, "metropolis"));
          PV_CUDA(timed(2, [&] { return k_phi_decide(ma, C, st); }, "phi_decide"));
        } else {
          ++launches;
          PV_CUDA(timed(2, [&] { return k_metropolis(ma, C, st); }, "metropolis"));
        }
        Lin = l3[0];
        bsL = S;
      }
      if (k + 1 < Lyo) PV_CUDA(compress(o, k, T, top, k + 1, slot_of(k + 1)));
    }
    return cudaSuccess;
  }

  cudaError_t sweep_once() {
    // vertical bonds: columns of the transposed lattice (O2), bottom environments from O3
    PV_CUDA(top_down_all(3, st_colbot));
    PV_CUDA(row_phase(2, st_coltop, true, st_colbot, 0));
    // horizontal bonds: rows (O0), bottom environments from O1
    PV_CUDA(top_down_all(1, st_bot));
    PV_CUDA(row_phase(0, st_top, false, st_bot, Lx * (Ly - 1)));
    top_valid = true;
    return cudaSuccess;
  }

  // Publish the host's sweep counter to the device for the next sweep.
  cudaError_t set_sweep() {
    ++launches;
    return k_set_u64(d_sweep, sweep_counter, st);
  }

  // ------------------------------------------------------ one sample step as a graph
  // Sweep, fresh environments, E_loc, G and the float64 sums of every chain: the same
  // launches every time (all per-chain choices are device data), so after one eager
  // pass (which also runs the autotuner and builds the sketches) the whole sequence is
  // captured once into a CUDA graph on the context's own non-blocking stream and
  // replayed, ordered against the caller's stream by events.
  bool use_graphs = true;
  cudaStream_t gst = nullptr;
  cudaGraphExec_t step_exec = nullptr;
  cudaEvent_t g_in = nullptr, g_out = nullptr;
  int eager_steps = 0;

  cudaError_t sample_step_body() {
    PV_CUDA(sweep_once());
    if (proposal_mode == 1) PV_CUDA(learned_sweep());
    PV_CUDA(measure_dev());
    launches += 2;
    // symmetrised: one sample per pair, E^Phi for both chains, G weighted into G^Phi
    PV_CUDA(k_energy_accum(sym ? eloc_phi : eloc, sym ? pairs : C, sums, st));
    return k_grad_accum(G, Ph, Ph, elem_site, d_site_half_off, d_site_full_off, d_site_size, d_site_spin, spins,
                        (long long)Ly * Lx, sym ? eloc_phi : eloc, C, sumG, sumGE, st, sym ? phi_wt : nullptr);
  }
  void drop_graph() {
    if (step_exec) cudaGraphExecDestroy(step_exec);
    step_exec = nullptr;
  }
  cudaError_t sample_step() {
    PV_CUDA(set_sweep());
    const bool graphable = use_graphs && !dry && !prof && !trace_on;
    if (!graphable || eager_steps < 1) {
      ++eager_steps;
      return sample_step_body();
    }
    if (!gst) {
      PV_CUDA(cudaStreamCreateWithFlags(&gst, cudaStreamNonBlocking));
      PV_CUDA(cudaEventCreateWithFlags(&g_in, cudaEventDisableTiming));
      PV_CUDA(cudaEventCreateWithFlags(&g_out, cudaEventDisableTiming));
    }
    PV_CUDA(cudaEventRecord(g_in, st));
    PV_CUDA(cudaStreamWaitEvent(gst, g_in, 0));
    if (!step_exec) {
      cudaStream_t user = st;
      st = gst;
      capturing = true;
      const long long l0 = launches;
      cudaError_t e = cudaStreamBeginCapture(gst, cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) e = sample_step_body();
      cudaGraph_t graph = nullptr;
      cudaError_t e2 = cudaStreamEndCapture(gst, &graph);
      capturing = false;
      st = user;
      graph_launches = launches - l0;
      launches = l0;
      if (e == cudaSuccess) e = e2;
      if (e == cudaSuccess) e = cudaGraphInstantiate(&step_exec, graph, 0);
      if (graph) cudaGraphDestroy(graph);
      if (e != cudaSuccess) {
        drop_graph();
        return e;
      }
    }
    launches += graph_launches;
    PV_CUDA(cudaGraphLaunch(step_exec, gst));
    PV_CUDA(cudaEventRecord(g_out, gst));
    return cudaStreamWaitEvent(st, g_out, 0);
  }
  long long graph_launches = 0;

  // ------------------------------------------------ measurement (Eqs. (3)-(7), App. C)
  cudaError_t measure_dev() {
    if (chi_m != chi_s) {
      // the measurement's own cutoff: fresh top environments at chi_m; the sampler's
      // are no longer in st_top afterwards
      chi = chi_m;
      top_valid = false;
      const cudaError_t e = measure_at_cutoff();
      chi = chi_s;
      PV_CUDA(e);
    } else {
      PV_CUDA(measure_at_cutoff());
    }
    if (!sym) return cudaSuccess;
    ++launches;
    return k_phi_combine(logpsi, sign, eloc, C, pairs, phi_wm, eloc_phi, phi_wt, status, st);
  }
  cudaError_t measure_at_cutoff() {
    if (!top_valid) {
      PV_CUDA(top_down_all(0, st_top));
      top_valid = chi == chi_s;
    }
    PV_CUDA(top_down_all(1, st_bot));
    ++launches;
    PV_CUDA(k_eloc_diag(spins, Ly, Lx, cfg.J1, cfg.J2, eloc, C, st));
    auto envRp = [&](int m) { return envR + (long long)m * C * S; };
    auto envRfp = [&](int m) { return envRf + (long long)m * C * S; };
    const int kstar = Ly / 2;
    for (int k = 0; k < Ly; ++k) {
      const View T = view(st_top, k, k);
      const View B = view(st_bot, Ly - 1 - k, Ly - 1 - k);
      const std::vector<int>& tb = *T.bond;
      const std::vector<int>& bb = *B.bond;
      std::vector<SiteOp> a(Lx);
      for (int m = 0; m < Lx; ++m) a[m] = site(0, k, m);
      for (int m = Lx - 1; m >= 1; --m) {
        const bool edge = (m == Lx - 1);
        const float* Ein = edge ? ones : envRp(m + 1);
        const long long bsE = edge ? 1 : S;
        PV_CUDA(right3_pair(Ein, bsE, tb[m + 1], bb[m + 1], T.site(m), T.chain_stride, tb[m], a[m], B.site(m),
                            B.chain_stride, bb[m], envRp(m), envRfp(m), S));
        const int n = tb[m] * a[m].Dl * bb[m];
        PV_CUDA(norm2(envRp(m), S, n, envRfp(m), n));
      }
      if (k == kstar) PV_CUDA(ms(exps, 0, C * sizeof(int)));
      const float* Lin = ones;
      long long bsL = 1;
      for (int m = 0; m < Lx; ++m) {
        const bool edge = (m == Lx - 1);
        const float* Rin = edge ? ones : envRp(m + 1);
        const long long bsR = edge ? 1 : S;
        float* cur = l3[(m + 1) % 2];
        const int n = tb[m + 1] * a[m].Dr * bb[m + 1];
        PV_CUDA(left3_pair(Lin, bsL, tb[m], bb[m], T.site(m), T.chain_stride, tb[m + 1], a[m], B.site(m),
                           B.chain_stride, bb[m + 1], cur, edge ? nullptr : fl, S, true));
        PV_CUDA(dot(cur, S, Rin, bsR, n, den));
        if (!edge)
          PV_CUDA(ratio(fl, S, envRfp(m + 1), S, n, a[m].spin, a[m + 1].spin, 0.5 * cfg.J1, (long long)k * Lx + m));
        PV_CUDA(delta3_after_left3(bb[m], tb[m + 1], a[m], B.site(m), B.chain_stride, bb[m + 1], Rin, bsR, den,
                                   G + site_half_off[(size_t)k * Lx + m], Ph));
        if (!edge) {
          PV_CUDA(norm2(cur, S, n, nullptr, 0, nullptr, 0, k == kstar ? exps : nullptr));
        } else if (k == kstar) {
          PV_CUDA(logpsi_of(cur, S, T.logs, B.logs));
        }
        Lin = cur;
        bsL = S;
      }
    }
    for (int k = 0; k + 1 < Ly; ++k) PV_CUDA(pair_terms(k));
    have_measure = true;
    return cudaSuccess;
  }

  // Vertical NN terms and both NNN diagonals of rows (k, k+1) by four-line environments.
  cudaError_t pair_terms(int k) {
    const View T = view(st_top, k, k);
    const View B = view(st_bot, Ly - 2 - k, Ly - 2 - k);
    const std::vector<int>& tb = *T.bond;
    const std::vector<int>& bb = *B.bond;
    std::vector<SiteOp> a1(Lx), a2(Lx);
    for (int m = 0; m < Lx; ++m) {
      a1[m] = site(0, k, m);
      a2[m] = site(0, k + 1, m);
    }
    auto R4p = [&](int m) { return R4 + (long long)m * C * S4; };
    for (int m = Lx - 1; m >= 1; --m) {
      const bool edge = (m == Lx - 1);
      PV_CUDA(right4(edge ? ones : R4p(m + 1), edge ? 1 : S4, tb[m + 1], bb[m + 1], T.site(m), T.chain_stride,
                     tb[m], a1[m], 0, a2[m], 0, B.site(m), B.chain_stride, bb[m], R4p(m), S4));
      PV_CUDA(norm2(R4p(m), S4, tb[m] * a1[m].Dl * a2[m].Dl * bb[m]));
    }
    const float* Lin = ones;
    long long bsL = 1;
    const float *Pt = nullptr, *Pb = nullptr;
    for (int m = 0; m < Lx; ++m) {
      const bool edge = (m == Lx - 1);
      const float* Rin = edge ? ones : R4p(m + 1);
      const long long bsR = edge ? 1 : S4;
      const int n = tb[m + 1] * a1[m].Dr * a2[m].Dr * bb[m + 1];
      float* cur = l4[(m + 1) % 2];
      auto step = [&](const float* Ein, long long bsE, int f1, int f2, float* out) {
        return left4(Ein, bsE, tb[m], bb[m], T.site(m), T.chain_stride, tb[m + 1], a1[m], f1, a2[m], f2,
                     B.site(m), B.chain_stride, bb[m + 1], out, S4);
      };
      // the four variants of this column from Lin share X = Lin . T and Y(f1) = X . a1
      auto from_y = [&](const float* Y, int f2, float* out) {
        return left4_zw(Y, bb[m], tb[m + 1], a1[m], a2[m], f2, B.site(m), B.chain_stride, bb[m + 1], out, S4,
                        tmp1);
      };
      // with the fused kernel every variant is one launch from Lin; otherwise the four
      // variants share X = Lin . T and Y(f1) = X . a1
      // (and in FP32 one launch computes all variants with the intermediates in shared memory)
      const bool fz = four_bmajor();
      float *Ptn = nullptr, *Pbn = nullptr;
      if (cfg.J2 != 0.0 && !edge) {
        Ptn = ptop[(m + 1) % 2];
        Pbn = pbot[(m + 1) % 2];
      }
      const Env4Fused f4 = fused4_left(Lin, bsL, tb[m], bb[m], T.site(m), T.chain_stride, tb[m + 1], a1[m], 0, a2[m], 0,
                                       B.site(m), B.chain_stride, bb[m + 1], cur, S4);
      const Env4Outs o4{{cur, Pbn, Ptn, fl4}};
      const bool f32 = f32_fused() && env4_f32_takes(f4, o4, C);
      if (fz) {
        PV_CUDA(step(Lin, bsL, 0, 0, cur));
      } else if (f32) {
        PV_CUDA(step4_f32(f4, o4, false));
      } else {
        PV_CUDA(left4_x(Lin, bsL, tb[m], bb[m], T.site(m), T.chain_stride, tb[m + 1], a1[m], a2[m], tmp1));
        PV_CUDA(left4_y(tmp1, bb[m], tb[m + 1], a1[m], 0, a2[m], tmp3));
        PV_CUDA(left4_y(tmp1, bb[m], tb[m + 1], a1[m], 1, a2[m], tmp4));
        PV_CUDA(from_y(tmp3, 0, cur));
      }
      PV_CUDA(dot(cur, S4, Rin, bsR, n, den));
      if (!f32) PV_CUDA(fz ? step(Lin, bsL, 1, 1, fl4) : from_y(tmp4, 1, fl4));
      PV_CUDA(ratio(fl4, S4, Rin, bsR, n, a1[m].spin, a2[m].spin, 0.5 * cfg.J1, (long long)Ly * Lx + k * Lx + m));
      if (cfg.J2 != 0.0) {
        if (!edge && !f32) {
          PV_CUDA(fz ? step(Lin, bsL, 1, 0, Ptn) : from_y(tmp4, 0, Ptn));
          PV_CUDA(fz ? step(Lin, bsL, 0, 1, Pbn) : from_y(tmp3, 1, Pbn));
        }
        if (m >= 1) {
          PV_CUDA(step(Pt, S4, 0, 1, fl4));
          PV_CUDA(ratio(fl4, S4, Rin, bsR, n, a1[m - 1].spin, a2[m].spin, 0.5 * cfg.J2));
          PV_CUDA(step(Pb, S4, 1, 0, fl4));
          PV_CUDA(ratio(fl4, S4, Rin, bsR, n, a2[m - 1].spin, a1[m].spin, 0.5 * cfg.J2));
        }
      }
      if (!edge) PV_CUDA(norm2(cur, S4, n, Ptn, Ptn ? n : 0, Pbn, Pbn ? n : 0));
      Lin = cur;
      bsL = S4;
      Pt = Ptn;
      Pb = Pbn;
    }
    return cudaSuccess;
  }

  // ------------------------------------------------------------ learned proposal
  // One exact MH move per row band (k, k+1), bands top-down k = 0..Ly-2; T_k is
  // rebuilt after the band above it moved, B_{k+1} comes from the start of the sweep.
  int proposal_mode = 0;
  bool net_ready = false;
  float *net = nullptr, *net_g = nullptr, *net_m = nullptr, *net_v = nullptr;
  float *h1 = nullptr, *h2 = nullptr, *logits = nullptr, *logits2 = nullptr;
  int8_t* prop = nullptr;
  int* move = nullptr;
  double *lq_fwd = nullptr, *lq_rev = nullptr, *net_acc = nullptr;
  int *ex_den = nullptr, *ex_num = nullptr;
  unsigned long long* lcount = nullptr;
  double *ltr_rho = nullptr, *ltr_dlq = nullptr;
  int8_t* ltr_dec = nullptr;
  int adam_t = 0;
  // training set collected from the plain sampler: spins and the measured NN ratios
  int8_t* ds_spins = nullptr;
  float* ds_rho = nullptr;
  long long ds_cap = 0, ds_n = 0;
  int8_t* spins_saved = nullptr;  // chain spins kept aside while pepsvmc_train_proposal measures
  float *tr_h1 = nullptr, *tr_h2 = nullptr, *tr_out = nullptr, *tr_d1 = nullptr, *tr_d2 = nullptr;
  int tr_batch = 0;

  cudaError_t net_alloc() {
    if (net) return cudaSuccess;
    const long long N = (long long)Ly * Lx;
    PV_CUDA(alloc(&net, kNetParams));
    PV_CUDA(alloc(&net_g, kNetParams));
    PV_CUDA(alloc(&net_m, kNetParams));
    PV_CUDA(alloc(&net_v, kNetParams));
    PV_CUDA(alloc(&h1, (size_t)C * kNetC * N));
    PV_CUDA(alloc(&h2, (size_t)C * kNetC * N));
    PV_CUDA(alloc(&logits, (size_t)C * 2 * N));
    PV_CUDA(alloc(&logits2, (size_t)C * 2 * N));
    PV_CUDA(alloc(&prop, (size_t)C * N));
    PV_CUDA(alloc(&move, (size_t)C * 4));
    PV_CUDA(alloc(&lq_fwd, C));
    PV_CUDA(alloc(&lq_rev, C));
    PV_CUDA(alloc(&net_acc, 2));
    PV_CUDA(alloc(&ex_den, C));
    PV_CUDA(alloc(&ex_num, C));
    PV_CUDA(alloc(&lcount, 2));
    PV_CUDA(alloc(&ltr_rho, (size_t)C * (Ly - 1)));
    PV_CUDA(alloc(&ltr_dlq, (size_t)C * (Ly - 1)));
    PV_CUDA(alloc(&ltr_dec, (size_t)C * (Ly - 1)));
    PV_CUDA(ms(net_m, 0, kNetParams * sizeof(float)));
    PV_CUDA(ms(net_v, 0, kNetParams * sizeof(float)));
    PV_CUDA(ms(lcount, 0, 2 * sizeof(unsigned long long)));
    return cudaSuccess;
  }

  // Four-line closure of band k for spin array sp: out points at the final scalar.
  cudaError_t band_closure(int k, const View& T, const View& B, const int8_t* sp, float* ba, float* bb, int* ex,
                           float** out) {
    const std::vector<int>& tb = *T.bond;
    const std::vector<int>& bbd = *B.bond;
    PV_CUDA(ms(ex, 0, C * sizeof(int)));
    sel_base = sp;
    const float* Lin = ones;
    long long bsL = 1;
    float* cur = ba;
    for (int m = 0; m < Lx; ++m) {
      const SiteOp a1 = site(0, k, m), a2 = site(0, k + 1, m);
      cur = (m % 2 == 0) ? ba : bb;
      cudaError_t e = left4(Lin, bsL, tb[m], bbd[m], T.site(m), T.chain_stride, tb[m + 1], a1, 0, a2, 0, B.site(m),
                            B.chain_stride, bbd[m + 1], cur, S4);
      if (e == cudaSuccess && m + 1 < Lx)
        e = norm2(cur, S4, tb[m + 1] * a1.Dr * a2.Dr * bbd[m + 1], nullptr, 0, nullptr, 0, ex);
      if (e != cudaSuccess) {
        sel_base = nullptr;
        return e;
      }
      Lin = cur;
      bsL = S4;
    }
    sel_base = nullptr;
    *out = cur;
    return cudaSuccess;
  }

  cudaError_t learned_sweep() {
    PV_CUDA(top_down_all(1, st_bot));
    const long long N = (long long)Ly * Lx;
    const NetParams w = NetParams::at(net);
    for (int k = 0; k + 1 < Ly; ++k) {
      const View T = view(st_top, k, k);
      const View B = view(st_bot, Ly - 2 - k, Ly - 2 - k);
      launches += 8;
      PV_CUDA(net_forward(w, spins, C, Ly, Lx, h1, h2, logits, st));
      PV_CUDA(propose_moves(logits, spins, prop, C, Ly, Lx, k, cfg.seed, d_sweep, move, lq_fwd, chain_base, st));
      PV_CUDA(net_forward(w, prop, C, Ly, Lx, h1, h2, logits2, st));
      PV_CUDA(reverse_logq(logits2, prop, C, Ly, Lx, k, move, lq_rev, st));
      float *den_p = nullptr, *num_p = nullptr;
      PV_CUDA(band_closure(k, T, B, spins, l4[0], l4[1], ex_den, &den_p));
      PV_CUDA(band_closure(k, T, B, prop, fl4, ptop[0], ex_num, &num_p));
      ++launches;
      PV_CUDA(accept_moves(spins, prop, C, (int)N, move, den_p, num_p, S4, ex_den, ex_num, lq_fwd, lq_rev, cfg.seed,
                           d_sweep, k, Ly - 1, trace_on ? ltr_rho : nullptr, ltr_dlq, trace_on ? ltr_dec : nullptr,
                           lcount, status, chain_base, st));
      PV_CUDA(compress(0, k, T, st_top, k + 1, k + 1));
    }
    top_valid = true;
    return cudaSuccess;
  }

  cudaError_t train_epochs(int epochs, int batch, float lr, double* loss) {
    const long long N = (long long)Ly * Lx;
    if (batch != tr_batch) {
      PV_CUDA(alloc(&tr_h1, (size_t)batch * kNetC * N));
      PV_CUDA(alloc(&tr_h2, (size_t)batch * kNetC * N));
      PV_CUDA(alloc(&tr_d1, (size_t)batch * kNetC * N));
      PV_CUDA(alloc(&tr_d2, (size_t)batch * kNetC * N));
      PV_CUDA(alloc(&tr_out, (size_t)batch * 2 * N));
      tr_batch = batch;
    }
    const NetParams w = NetParams::at(net), g = NetParams::at(net_g);
    double sse = 0.0, cnt = 0.0;
    for (int ep = 0; ep < epochs; ++ep) {
      sse = cnt = 0.0;
      for (long long off = 0; off + batch <= ds_n; off += batch) {
        ++adam_t;
        launches += 12;
        PV_CUDA(net_train_step(w, g, net_m, net_v, kNetParams, adam_t, lr, ds_spins + off * N, ds_rho + off * 2 * N,
                               batch, Ly, Lx, tr_h1, tr_h2, tr_out, tr_d2, tr_d1, net_acc, st));
        double a[2] = {0, 0};
        PV_CUDA(cps(a, net_acc, sizeof(a), cudaMemcpyDeviceToHost));
        sse += a[0];
        cnt += a[1];
      }
    }
    if (loss) *loss = cnt > 0 ? sse / cnt : 0.0;
    return cudaSuccess;
  }

  // Psi of the current configuration contracted at row `row` (fresh environments).
  cudaError_t amplitude_dev(int row) {
    PV_CUDA(top_down_all(0, st_top));
    top_valid = true;
    PV_CUDA(top_down_all(1, st_bot));
    const View T = view(st_top, row, row);
    const View B = view(st_bot, Ly - 1 - row, Ly - 1 - row);
    const std::vector<int>& tb = *T.bond;
    const std::vector<int>& bb = *B.bond;
    PV_CUDA(ms(exps, 0, C * sizeof(int)));
    const float* Lin = ones;
    long long bsL = 1;
    for (int m = 0; m < Lx; ++m) {
      const SiteOp a = site(0, row, m);
      float* cur = l3[(m + 1) % 2];
      PV_CUDA(left3(Lin, bsL, tb[m], bb[m], T.site(m), T.chain_stride, tb[m + 1], a, 0, B.site(m),
                    B.chain_stride, bb[m + 1], cur, S));
      if (m + 1 < Lx) {
        PV_CUDA(norm2(cur, S, tb[m + 1] * a.Dr * bb[m + 1], nullptr, 0, nullptr, 0, exps));
      } else {
        PV_CUDA(logpsi_of(cur, S, T.logs, B.logs));
      }
      Lin = cur;
      bsL = S;
    }
    return cudaSuccess;
  }

  // ------------------------------------------ random-NNASP sweep (Sec. II A, Eq. (prob_r))
  // N attempts; each proposes one uniformly chosen antiparallel NN pair per chain and
  // needs Psi of every chain's trial configuration: a full boundary-MPS contraction
  // (closed at row Ly/2, as the measurement's amplitude) with the site tensors selected
  // by the trial spins.  Psi of the current configurations is kept across attempts.
  int8_t *r_prop = nullptr, *r_sg = nullptr, *r_tr_dec = nullptr;
  int *r_Ka = nullptr, *r_Kb = nullptr, *r_bond = nullptr, *r_tr_bond = nullptr;
  double *r_lp = nullptr, *r_tr_ratio = nullptr;
  cudaError_t random_alloc() {
    if (r_prop) return cudaSuccess;
    const long long N = (long long)Ly * Lx;
    PV_CUDA(alloc(&r_prop, C * N));
    PV_CUDA(alloc(&r_sg, C));
    PV_CUDA(alloc(&r_Ka, C));
    PV_CUDA(alloc(&r_Kb, C));
    PV_CUDA(alloc(&r_bond, C));
    PV_CUDA(alloc(&r_lp, C));
    PV_CUDA(alloc(&r_tr_bond, C * N));
    PV_CUDA(alloc(&r_tr_ratio, C * N));
    PV_CUDA(alloc(&r_tr_dec, C * N));
    return cudaSuccess;
  }
  cudaError_t random_sweep() {
    PV_CUDA(random_alloc());
    const int kstar = Ly / 2;
    const long long N = (long long)Ly * Lx;
    PV_CUDA(amplitude_dev(kstar));
    PV_CUDA(cp(r_lp, logpsi, C * sizeof(double), cudaMemcpyDeviceToDevice));
    PV_CUDA(cp(r_sg, sign, C, cudaMemcpyDeviceToDevice));
    RandomArgs ra{};
    ra.spins = spins; ra.prop = r_prop; ra.C = C; ra.Ly = Ly; ra.Lx = Lx;
    ra.key = cfg.seed; ra.sweep = d_sweep; ra.chain_base = chain_base;
    ra.Ka = r_Ka; ra.Kb = r_Kb; ra.bond = r_bond;
    ra.lp_cur = r_lp; ra.sg_cur = r_sg; ra.lp_new = logpsi; ra.sg_new = sign;
    ra.tr_bond = trace_on ? r_tr_bond : nullptr; ra.tr_ratio = r_tr_ratio; ra.tr_dec = r_tr_dec; ra.tr_stride = N;
    ra.counters = counters; ra.status = status;
    for (int t = 0; t < N; ++t) {
      ra.attempt = t;
      launches += 2;
      PV_CUDA(k_random_propose(ra, st));
      sel_base = r_prop;
      const cudaError_t e = amplitude_dev(kstar);
      sel_base = nullptr;
      PV_CUDA(e);
      PV_CUDA(k_random_accept(ra, st));
    }
    top_valid = false;
    return cudaSuccess;
  }

  cudaError_t refresh_perms() {
    for (int o = 0; o < 4; ++o)
      for (int t = 0; t < 2; ++t) {
        ++launches;
        PV_CUDA(k_gather_f32(perm[o][t], master, perm_map[o][t], P, st));
      }
    return cudaSuccess;
  }

  int check_status() {
    unsigned h = 0;
    cudaError_t e = cp(&h, status, sizeof(unsigned), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = sync();
    if (e != cudaSuccess) return fail_cuda(e);
    if (h) {
      ms(status, 0, sizeof(unsigned));
      // the environments of a failed call are not valid; the root cause comes first (a
      // timed-out product leaves garbage behind, a zero amplitude leads to 0/0 later)
      top_valid = false;
      if (h & ST_TIMEOUT) return fail(PEPSVMC_ETIMEOUT, "device wait budget exhausted");
      if (h & ST_ZEROPSI) return fail(PEPSVMC_EZEROPSI, "a configuration with Psi(S) = 0 was met");
      if (h & ST_NONFINITE) return fail(PEPSVMC_ENONFINITE, "non-finite amplitude ratio or environment");
    }
    return PEPSVMC_OK;
  }

  int fail(int code, const std::string& m) {
    err = m;
    return code;
  }
  int fail_cuda(cudaError_t e) {
    if (e == cudaErrorInvalidValue && err.rfind("bounds check", 0) == 0) return PEPSVMC_EINVAL;
    if (e == cudaErrorInvalidValue && err.rfind("contraction layout", 0) == 0) return PEPSVMC_EINVAL;
    err = std::string("CUDA error: ") + cudaGetErrorString(e);
    return PEPSVMC_ECUDA;
  }
};

// ============================================================================= C ABI
namespace {

int validate(const pepsvmc_config* c, std::string& why) {
  if (!c) { why = "null config"; return PEPSVMC_EINVAL; }
  if (c->Ly < 1 || c->Lx < 1 || c->Ly > 64 || c->Lx > 64) { why = "Ly, Lx must be in 1..64"; return PEPSVMC_EINVAL; }
  if ((c->Ly * c->Lx) % 2) { why = "Ly*Lx must be even (S^z = 0 sector)"; return PEPSVMC_EINVAL; }
  if (c->D < 1 || c->D > 16) { why = "D must be in 1..16"; return PEPSVMC_EINVAL; }
  if (c->chi < 1 || c->chi > 64) { why = "chi must be in 1..64"; return PEPSVMC_EINVAL; }
  if (c->chi_measure < 0 || c->chi_measure > 64) { why = "chi_measure must be in 0..64"; return PEPSVMC_EINVAL; }
  const long long cx = std::max(c->chi, c->chi_measure);
  if (cx * cx * c->D * 2 * 4 > 200 * 1024) { why = "chi*chi*D too large for the QR kernel"; return PEPSVMC_EINVAL; }
  if (c->n_chains < 1 || c->n_chains > (1 << 20)) { why = "n_chains must be >= 1"; return PEPSVMC_EINVAL; }
  if (c->n_fit < 1 || c->n_fit % 2 == 0) { why = "n_fit must be odd and >= 1"; return PEPSVMC_EINVAL; }
  if (c->precision != PEPSVMC_FP32 && c->precision != PEPSVMC_MIXED_BF16 && c->precision != PEPSVMC_MIXED_TF32 &&
      c->precision != PEPSVMC_MIXED_BF16X3) {
    why = "unknown precision";
    return PEPSVMC_EINVAL;
  }
  if (c->chain_offset < 0) { why = "chain_offset must be >= 0"; return PEPSVMC_EINVAL; }
  if (c->wait_budget_cycles > (uint64_t)1 << 62) { why = "wait_budget_cycles too large"; return PEPSVMC_EINVAL; }
  if (c->symmetrize != 0 && c->symmetrize != 1) { why = "symmetrize must be 0 or 1"; return PEPSVMC_EINVAL; }
  if (c->symmetrize && c->n_chains % 2) { why = "symmetrize needs an even n_chains (S, S-bar pairs)"; return PEPSVMC_EINVAL; }
  for (int i = 0; i < 2; ++i)
    if (c->reserved[i]) { why = "reserved fields must be zero"; return PEPSVMC_EINVAL; }
  return PEPSVMC_OK;
}

int setup(pepsvmc_ctx* x, const double* tensors, const double* sketch) {
  const int Ly = x->Ly, Lx = x->Lx, D = x->D, C = x->C;
  x->O[0] = {Ly, Lx, false, false};
  x->O[1] = {Ly, Lx, false, true};
  x->O[2] = {Lx, Ly, true, false};
  x->O[3] = {Lx, Ly, true, true};
  x->Lmax = std::max(Ly, Lx);
  const long long X = x->chi_x;
  x->S = X * D * X;
  x->S4 = X * D * D * X;
  x->SI = std::max((long long)D * D * D * X * X, std::max(x->S, (long long)D * D * X * X));
  x->trivial_bond.assign(x->Lmax + 1, 1);
  // original site offsets
  long long off = 0, hoff = 0;
  for (int k = 0; k < Ly; ++k)
    for (int m = 0; m < Lx; ++m) {
      const int sz = (m == 0 ? 1 : D) * (m == Lx - 1 ? 1 : D) * (k == 0 ? 1 : D) * (k == Ly - 1 ? 1 : D);
      x->site_off.push_back(off);
      x->site_half_off.push_back(hoff);
      x->site_size.push_back(sz);
      off += 2LL * sz;
      hoff += sz;
    }
  x->P = off;
  x->Ph = hoff;
  x->sketch_host.assign(sketch, sketch + (size_t)x->Lmax * x->chi_x * D * x->chi_x);

  cudaError_t e;
#define ALLOC(p, n) if ((e = x->alloc(&(p), (size_t)(n))) != cudaSuccess) return x->fail(PEPSVMC_ENOMEM, std::string("cudaMalloc failed: ") + cudaGetErrorString(e))
  ALLOC(x->master, x->P);
  ALLOC(x->grad, x->P);
  ALLOC(x->sumG, x->P);
  ALLOC(x->sumGE, x->P);
  ALLOC(x->sums, 4);
  ALLOC(x->spins, (long long)C * Ly * Lx);
  ALLOC(x->ones, std::max(C, 1) + 1);
  ALLOC(x->zeros_d, C);
  for (int o = 0; o < 4; ++o) {
    // permuted copies and their gather maps
    const Orient& Ob = x->O[o];
    std::vector<int> map_lurd(x->P), map_urld(x->P);
    long long po = 0;
    x->perm_site_off[o].clear();
    for (int kp = 0; kp < Ob.Ly; ++kp)
      for (int mp = 0; mp < Ob.Lx; ++mp) {
        const int Dlp = mp == 0 ? 1 : D, Drp = mp == Ob.Lx - 1 ? 1 : D, Dup = kp == 0 ? 1 : D,
                  Ddp = kp == Ob.Ly - 1 ? 1 : D;
        int k, m;
        x->orig(o, kp, mp, k, m);
        const int Dl = m == 0 ? 1 : D, Dr = m == Lx - 1 ? 1 : D, Du = k == 0 ? 1 : D, Dd = k == Ly - 1 ? 1 : D;
        const long long sz = (long long)Dlp * Drp * Dup * Ddp;
        x->perm_site_off[o].push_back(po);
        for (int s = 0; s < 2; ++s)
          for (int lp = 0; lp < Dlp; ++lp)
            for (int rp = 0; rp < Drp; ++rp)
              for (int up = 0; up < Dup; ++up)
                for (int dp = 0; dp < Ddp; ++dp) {
                  int l, r, u, d;
                  if (o == 0) { l = lp; r = rp; u = up; d = dp; }
                  else if (o == 1) { l = lp; r = rp; u = dp; d = up; }
                  else if (o == 2) { l = up; r = dp; u = lp; d = rp; }
                  else { l = dp; r = up; u = lp; d = rp; }
                  const long long src = x->site_off[(size_t)k * Lx + m] + s * sz + (((long long)l * Dr + r) * Du + u) * Dd + d;
                  const long long i_lurd = po + s * sz + (((long long)lp * Dup + up) * Drp + rp) * Ddp + dp;
                  const long long i_urld = po + s * sz + (((long long)up * Drp + rp) * Dlp + lp) * Ddp + dp;
                  map_lurd[i_lurd] = (int)src;
                  map_urld[i_urld] = (int)src;
                }
        po += 2 * sz;
      }
    for (int t = 0; t < 2; ++t) {
      ALLOC(x->perm[o][t], x->P);
      ALLOC(x->perm_map[o][t], x->P);
      const std::vector<int>& mp = t == 0 ? map_lurd : map_urld;
      if ((e = x->cps(x->perm_map[o][t], mp.data(), x->P * sizeof(int), cudaMemcpyHostToDevice)) != cudaSuccess)
        return x->fail_cuda(e);
    }
  }
  auto mkstore = [&](Store& s, int rows, int L, int nslots) -> int {
    s.rows = rows;
    s.L = L;
    s.bond.assign(rows, std::vector<int>(L + 1, 1));
    cudaError_t ee;
    if ((ee = x->alloc(&s.base, (size_t)nslots * L * C * x->S)) != cudaSuccess)
      return x->fail(PEPSVMC_ENOMEM, std::string("cudaMalloc failed (boundary MPS store): ") + cudaGetErrorString(ee));
    if ((ee = x->alloc(&s.logs, (size_t)nslots * C)) != cudaSuccess) return x->fail(PEPSVMC_ENOMEM, "cudaMalloc failed");
    return PEPSVMC_OK;
  };
  int rc;
  if ((rc = mkstore(x->st_top, Ly, Lx, Ly)) != 0) return rc;
  if ((rc = mkstore(x->st_bot, Ly, Lx, Ly)) != 0) return rc;
  if ((rc = mkstore(x->st_colbot, Lx, Ly, Lx)) != 0) return rc;
  if ((rc = mkstore(x->st_coltop, Lx, Ly, 2)) != 0) return rc;
  const long long L1 = x->Lmax + 1;
  ALLOC(x->envL, L1 * C * x->S);
  ALLOC(x->envR, L1 * C * x->S);
  ALLOC(x->envRf, L1 * C * x->S);
  ALLOC(x->l3[0], C * x->S);
  ALLOC(x->l3[1], C * x->S);
  ALLOC(x->fl, C * x->S);
  ALLOC(x->tmp1, C * x->SI);
  ALLOC(x->tmp2, C * x->SI);
  ALLOC(x->tmp3, C * x->SI);
  ALLOC(x->tmp4, C * x->SI);
  ALLOC(x->R4, (long long)(Lx + 1) * C * x->S4);
  ALLOC(x->l4[0], C * x->S4);
  ALLOC(x->l4[1], C * x->S4);
  ALLOC(x->fl4, C * x->S4);
  for (int i = 0; i < 2; ++i) {
    ALLOC(x->ptop[i], C * x->S4);
    ALLOC(x->pbot[i], C * x->S4);
  }
  ALLOC(x->G, C * x->Ph);
  ALLOC(x->eloc, C);
  ALLOC(x->den, C);
  ALLOC(x->logpsi, C);
  ALLOC(x->sign, C);
  ALLOC(x->exps, C);
  ALLOC(x->status, 1);
  ALLOC(x->counters, 2);
  ALLOC(x->d_sweep, 1);
  if (x->sym) {
    ALLOC(x->phi_rho, C);
    ALLOC(x->phi_w, C);
    ALLOC(x->phi_wm, C);
    ALLOC(x->eloc_phi, C);
    ALLOC(x->phi_wt, C);
    ALLOC(x->phi_lp, C);
    ALLOC(x->phi_sg, C);
    ALLOC(x->phi_exps, C);
  }
  // site tables for the gradient accumulation
  {
    std::vector<int> es(x->Ph), sp(Ly * Lx);
    std::vector<long long> full(Ly * Lx);
    for (int j = 0; j < Ly * Lx; ++j) {
      for (int i = 0; i < x->site_size[j]; ++i) es[x->site_half_off[j] + i] = j;
      sp[j] = j;
      full[j] = x->site_off[j];
    }
    ALLOC(x->elem_site, x->Ph);
    ALLOC(x->d_site_half_off, Ly * Lx);
    ALLOC(x->d_site_full_off, Ly * Lx);
    ALLOC(x->d_site_size, Ly * Lx);
    ALLOC(x->d_site_spin, Ly * Lx);
    if ((e = x->cps(x->elem_site, es.data(), es.size() * sizeof(int), cudaMemcpyHostToDevice)) ||
        (e = x->cps(x->d_site_half_off, x->site_half_off.data(), Ly * Lx * sizeof(long long), cudaMemcpyHostToDevice)) ||
        (e = x->cps(x->d_site_full_off, full.data(), Ly * Lx * sizeof(long long), cudaMemcpyHostToDevice)) ||
        (e = x->cps(x->d_site_size, x->site_size.data(), Ly * Lx * sizeof(int), cudaMemcpyHostToDevice)) ||
        (e = x->cps(x->d_site_spin, sp.data(), Ly * Lx * sizeof(int), cudaMemcpyHostToDevice)))
      return x->fail_cuda(e);
  }
#undef ALLOC
  if ((e = x->cps(x->master, tensors, x->P * sizeof(double), cudaMemcpyHostToDevice)) != cudaSuccess)
    return x->fail_cuda(e);
  if ((e = k_fill(x->ones, C + 1, 1.f, x->st)) != cudaSuccess) return x->fail_cuda(e);
  if ((e = k_fill_d(x->zeros_d, C, 0.0, x->st)) != cudaSuccess) return x->fail_cuda(e);
  if ((e = x->ms(x->status, 0, sizeof(unsigned))) != cudaSuccess) return x->fail_cuda(e);
  if ((e = x->ms(x->counters, 0, 2 * sizeof(unsigned long long))) != cudaSuccess) return x->fail_cuda(e);
  if ((e = x->refresh_perms()) != cudaSuccess) return x->fail_cuda(e);
  // Neel start
  std::vector<int8_t> neel((size_t)C * Ly * Lx);
  for (int c = 0; c < C; ++c)
    for (int k = 0; k < Ly; ++k)
      for (int m = 0; m < Lx; ++m)
        neel[((size_t)c * Ly + k) * Lx + m] = (((k + m) % 2 == 0) != (x->sym && c >= x->pairs)) ? 1 : -1;
  if ((e = x->cps(x->spins, neel.data(), neel.size(), cudaMemcpyHostToDevice)) != cudaSuccess) return x->fail_cuda(e);
  if ((e = x->sync()) != cudaSuccess) return x->fail_cuda(e);
  return PEPSVMC_OK;
}

}  // namespace

extern "C" {

int pepsvmc_init(const pepsvmc_config* cfg, const double* tensors, const double* sketch, void* stream,
                 pepsvmc_ctx** out) {
  if (!out) return PEPSVMC_EINVAL;
  *out = nullptr;
  std::string why;
  int rc = validate(cfg, why);
  pepsvmc_ctx* x = new (std::nothrow) pepsvmc_ctx();
  if (!x) return PEPSVMC_ENOMEM;
  *out = x;
  if (rc != PEPSVMC_OK) return x->fail(rc, why);
  if (!tensors || !sketch) return x->fail(PEPSVMC_EINVAL, "tensors and sketch must not be null");
  x->cfg = *cfg;
  x->st = (cudaStream_t)stream;
  // PEPSVMC_DRY_RUN=1 (read once per process): no device is touched; every launch of
  // the orchestration is bounds-checked on the host and skipped.  Validation tooling only.
  static const bool dry_env = [] {
    const char* v = getenv("PEPSVMC_DRY_RUN");
    return v && v[0] == '1';
  }();
  g_dry_run = dry_env;
  x->dry = dry_env;
  x->C = cfg->n_chains;
  x->Ly = cfg->Ly;
  x->Lx = cfg->Lx;
  x->D = cfg->D;
  x->chi = x->chi_s = cfg->chi;
  x->chi_m = cfg->chi_measure ? cfg->chi_measure : cfg->chi;
  x->chi_x = std::max(x->chi_s, x->chi_m);
  x->nfit = cfg->n_fit;
  x->wait_budget = (long long)cfg->wait_budget_cycles;
  x->chain_base = (unsigned)cfg->chain_offset;
  x->sym = cfg->symmetrize != 0;
  x->pairs = x->sym ? x->C / 2 : 0;
  return setup(x, tensors, sketch);
}

void pepsvmc_destroy(pepsvmc_ctx* x) {
  if (!x) return;
  if (!x->allocs.empty()) {
    if (x->st) cudaStreamSynchronize(x->st);
    else cudaDeviceSynchronize();  // NOLINT
  }
  x->collect();
  x->drop_graph();
  if (x->gst) cudaStreamDestroy(x->gst);
  if (x->g_in) cudaEventDestroy(x->g_in);
  if (x->g_out) cudaEventDestroy(x->g_out);
  for (cudaEvent_t e : x->ev_pool) cudaEventDestroy(e);
  for (void* p : x->allocs) cudaFree(p);
  delete x;
}

const char* pepsvmc_last_error(const pepsvmc_ctx* x) { return x ? x->err.c_str() : "null context"; }
int64_t pepsvmc_n_params(const pepsvmc_ctx* x) { return x ? x->P : 0; }
int64_t pepsvmc_n_grad_entries(const pepsvmc_ctx* x) { return x ? x->Ph : 0; }
int64_t pepsvmc_launch_count(const pepsvmc_ctx* x) { return x ? x->launches : 0; }

int pepsvmc_env3_left(pepsvmc_ctx* x, const float* E, const float* T, const float* A, const int8_t* spins,
                      const float* B, float* out, int32_t n_chains, int32_t cT, int32_t cB, int32_t cT2, int32_t cB2,
                      int32_t Dl, int32_t Dr, int32_t Du, int32_t Dd) {
  if (!x) return PEPSVMC_EINVAL;
  const Env3Dims d{cT, cB, cT2, cB2, Dl, Dr, Du, Dd};
  if (!E || !T || !A || !B || !out || n_chains < 1 || !env3_dims_ok(d))
    return x->fail(PEPSVMC_EINVAL, "env3_left: null pointer or non-positive size");
  if (n_chains > x->C || env3_scratch(d) > x->SI)
    return x->fail(PEPSVMC_EINVAL, "env3_left: more chains or larger bonds than the context was created for");
  SiteOp op;
  op.Dl = Dl; op.Dr = Dr; op.Du = Du; op.Dd = Dd;
  op.size = (long long)Dl * Dr * Du * Dd;
  op.lurd = A;
  op.spin = 0;
  if (x->fused_ok(cT, cB, cT2, cB2, op)) {
    Env3Fused f = x->fused_left(E, (long long)cT * Dl * cB, cT, cB, T, (long long)cT * Du * cT2, cT2, op, 0, B,
                                (long long)cB * Dd * cB2, cB2, out, (long long)cT2 * Dr * cB2);
    f.sel = spins;
    f.sel_stride = 1;
    cudaError_t e = x->fused3(f, n_chains, true);
    return e == cudaSuccess ? PEPSVMC_OK : x->fail_cuda(e);
  }
  if (x->f32_fused()) {
    Env3Fused f = x->fused_left(E, (long long)cT * Dl * cB, cT, cB, T, (long long)cT * Du * cT2, cT2, op, 0, B,
                                (long long)cB * Dd * cB2, cB2, out, (long long)cT2 * Dr * cB2);
    f.sel = spins;
    f.sel_stride = 1;
    const long long no = n_chains * f.bsO;
    if (env3_f32_fits(f) && !overlaps(out, no, E, n_chains * f.bsE) && !overlaps(out, no, T, n_chains * f.bsT) &&
        !overlaps(out, no, A, 2 * f.ssA) && !overlaps(out, no, B, n_chains * f.bsB) &&
        !overlaps(out, no, spins, n_chains)) {
      cudaError_t e = x->step3_f32(f, nullptr, false, n_chains, true);
      return e == cudaSuccess ? PEPSVMC_OK : x->fail_cuda(e);
    }
  }
  GemmDesc g[3];
  env3_left_descs(g, d, E, (long long)cT * Dl * cB, T, (long long)cT * Du * cT2, A, (long long)Dl * Dr * Du * Dd,
                  spins, 1, 0, B, (long long)cB * Dd * cB2, out, (long long)cT2 * Dr * cB2, x->tmp1, x->tmp2, x->SI);
  for (int i = 0; i < 3; ++i) {
    g[i].batch = n_chains;
    ++x->launches;
    cudaError_t e = x->launch_gemm(g[i]);
    if (e != cudaSuccess) return x->fail_cuda(e);
  }
  return PEPSVMC_OK;
}

int pepsvmc_env4_left(pepsvmc_ctx* x, const float* E, const float* T, const float* A1, const int8_t* spins1,
                      const float* A2, const int8_t* spins2, const float* B, float* out, int32_t n_chains, int32_t cT,
                      int32_t cB, int32_t cT2, int32_t cB2, int32_t D1l, int32_t D1r, int32_t Du1, int32_t Dd1,
                      int32_t D2l, int32_t D2r, int32_t Dd2, int32_t bmajor) {
  if (!x) return PEPSVMC_EINVAL;
  if (bmajor != 0 && bmajor != 1) return x->fail(PEPSVMC_EINVAL, "env4_left: bmajor must be 0 or 1");
  const int dims[11] = {cT, cB, cT2, cB2, D1l, D1r, Du1, Dd1, D2l, D2r, Dd2};
  if (!E || !T || !A1 || !A2 || !B || !out || n_chains < 1)
    return x->fail(PEPSVMC_EINVAL, "env4_left: null pointer or no chains");
  for (int v : dims)
    if (v < 1) return x->fail(PEPSVMC_EINVAL, "env4_left: non-positive size");
  const long long X = (long long)D2l * cB * cT2 * std::max(D1l * Du1, D1r * Dd1);
  const long long Z = (long long)cB * cT2 * D1r * std::max(D2l * Dd1, D2r * Dd2);
  if (n_chains > x->C || std::max(X, Z) > x->SI)
    return x->fail(PEPSVMC_EINVAL, "env4_left: more chains or larger bonds than the context was created for");
  const long long s1 = (long long)D1l * Du1 * D1r * Dd1, s2 = (long long)D2l * Dd1 * D2r * Dd2;
  Env4Fused f;
  f.cT = cT; f.cB = cB; f.cT2 = cT2; f.cB2 = cB2;
  f.D1l = D1l; f.D1r = D1r; f.Du1 = Du1; f.Dd1 = Dd1; f.D2l = D2l; f.D2r = D2r; f.Dd2 = Dd2;
  f.batch = n_chains;
  f.wait_cycles = x->wait_budget;
  f.E = E; f.bsE = (long long)cT * D1l * D2l * cB;
  if (bmajor) {
    f.sEb = (long long)cT * D1l * D2l; f.sEa = (long long)D1l * D2l; f.sEl1 = D2l; f.sEl2 = 1;
  } else {
    f.sEa = (long long)D1l * D2l * cB; f.sEl1 = (long long)D2l * cB; f.sEl2 = cB; f.sEb = 1;
  }
  f.T = T; f.bsT = (long long)cT * Du1 * cT2; f.sTa = (long long)Du1 * cT2; f.sTu = cT2; f.sTa2 = 1;
  f.A1 = A1; f.ss1 = s1; f.s1l = (long long)Du1 * D1r * Dd1; f.s1u = (long long)D1r * Dd1; f.s1r = Dd1; f.s1d = 1;
  f.A2 = A2; f.ss2 = s2; f.s2l = (long long)Dd1 * D2r * Dd2; f.s2u = (long long)D2r * Dd2; f.s2r = Dd2; f.s2d = 1;
  f.sel1 = spins1; f.sel2 = spins2; f.sel_stride = 1;
  f.B = B; f.bsB = (long long)cB * Dd2 * cB2; f.sBb = (long long)Dd2 * cB2; f.sBd = cB2; f.sBb2 = 1;
  f.out = out; f.bsO = (long long)cT2 * D1r * D2r * cB2;
  if (bmajor) {
    f.sOb2 = (long long)cT2 * D1r * D2r; f.sOa2 = (long long)D1r * D2r; f.sOr1 = D2r; f.sOr2 = 1;
  } else {
    f.sOa2 = (long long)D1r * D2r * cB2; f.sOr1 = (long long)D2r * cB2; f.sOr2 = cB2; f.sOb2 = 1;
  }
  if (x->fused4_ok(f)) {
    ++x->launches;
    cudaError_t e = env4_fused(f, x->tc_mode() == 3, x->status, x->st);
    return e == cudaSuccess ? PEPSVMC_OK : x->fail_cuda(e);
  }
  if (bmajor) return x->fail(PEPSVMC_EINVAL, "env4_left: the b-major layout needs the fused kernel");
  const Env4Outs outs{{out}};
  const long long no = n_chains * f.bsO;
  if (x->f32_fused() && env4_f32_takes(f, outs, n_chains) && !overlaps(out, no, E, n_chains * f.bsE) &&
      !overlaps(out, no, T, n_chains * f.bsT) && !overlaps(out, no, A1, 2 * s1) && !overlaps(out, no, A2, 2 * s2) &&
      !overlaps(out, no, B, n_chains * f.bsB) && !overlaps(out, no, spins1, n_chains) &&
      !overlaps(out, no, spins2, n_chains)) {
    ++x->launches;
    cudaError_t e = env4_f32(f, outs, false, x->st);
    return e == cudaSuccess ? PEPSVMC_OK : x->fail_cuda(e);
  }
  // four separate products, as left4_x / left4_y / left4_zw with the caller's spins
  GemmDesc g[4];
  float* t1 = x->tmp1;
  float* t2 = x->tmp2;
  g[0].M = D1l * D2l * cB; g[0].N = Du1 * cT2; g[0].K = cT;
  g[0].A = E; g[0].sAm = 1; g[0].sAk = (long long)D1l * D2l * cB; g[0].bsA = (long long)cT * D1l * D2l * cB;
  g[0].B = T; g[0].sBk = (long long)Du1 * cT2; g[0].sBn = 1; g[0].bsB = (long long)cT * Du1 * cT2;
  g[0].C = t1; g[0].bsC = x->SI;
  g[0].cm2 = D2l * cB; g[0].sCm1 = Du1; g[0].sCm2 = (long long)cT2 * D1l * Du1;
  g[0].cn2 = cT2; g[0].sCn1 = 1; g[0].sCn2 = (long long)D1l * Du1;
  g[1].M = D2l * cB * cT2; g[1].N = D1r * Dd1; g[1].K = D1l * Du1;
  g[1].A = t1; g[1].sAm = (long long)D1l * Du1; g[1].sAk = 1; g[1].bsA = x->SI;
  g[1].B = A1; g[1].ssB = s1; g[1].sel = spins1; g[1].sel_stride = 1; g[1].sBk = (long long)D1r * Dd1; g[1].sBn = 1;
  g[1].C = t2; g[1].bsC = x->SI;
  g[1].cm2 = cB * cT2; g[1].sCm1 = Dd1; g[1].sCm2 = (long long)D1r * D2l * Dd1;
  g[1].cn2 = Dd1; g[1].sCn1 = (long long)D2l * Dd1; g[1].sCn2 = 1;
  g[2].M = cB * cT2 * D1r; g[2].N = D2r * Dd2; g[2].K = D2l * Dd1;
  g[2].A = t2; g[2].sAm = (long long)D2l * Dd1; g[2].sAk = 1; g[2].bsA = x->SI;
  g[2].B = A2; g[2].ssB = s2; g[2].sel = spins2; g[2].sel_stride = 1; g[2].sBk = (long long)D2r * Dd2; g[2].sBn = 1;
  g[2].C = t1; g[2].bsC = x->SI;
  g[2].cm2 = cT2 * D1r; g[2].sCm1 = Dd2; g[2].sCm2 = (long long)D2r * cB * Dd2;
  g[2].cn2 = Dd2; g[2].sCn1 = (long long)cB * Dd2; g[2].sCn2 = 1;
  g[3].M = cT2 * D1r * D2r; g[3].N = cB2; g[3].K = cB * Dd2;
  g[3].A = t1; g[3].sAm = (long long)cB * Dd2; g[3].sAk = 1; g[3].bsA = x->SI;
  g[3].B = B; g[3].sBk = cB2; g[3].sBn = 1; g[3].bsB = (long long)cB * Dd2 * cB2;
  g[3].C = out; g[3].bsC = (long long)cT2 * D1r * D2r * cB2; g[3].sCm1 = cB2; g[3].sCn1 = 1;
  for (int i = 0; i < 4; ++i) {
    g[i].batch = n_chains;
    ++x->launches;
    cudaError_t e = x->launch_gemm(g[i]);
    if (e != cudaSuccess) return x->fail_cuda(e);
  }
  return PEPSVMC_OK;
}

int pepsvmc_set_profiling(pepsvmc_ctx* x, int32_t on) {
  if (!x) return PEPSVMC_EINVAL;
  cudaError_t e = x->collect();
  if (e != cudaSuccess) return x->fail_cuda(e);
  for (double& v : x->prof_acc) v = 0.0;
  x->shape_stats.clear();
  x->prof = on != 0;
  return PEPSVMC_OK;
}

int pepsvmc_get_profile_shapes(pepsvmc_ctx* x, char* buf, int64_t len) {
  if (!x || !buf || len < 2) return PEPSVMC_EINVAL;
  cudaError_t e = x->collect();
  if (e != cudaSuccess) return x->fail_cuda(e);
  std::string js = "[";
  for (const auto& kv : x->shape_stats) {
    char row[256];
    snprintf(row, sizeof(row), "%s{\"shape\":\"%s\",\"launches\":%lld,\"flops\":%.6g,\"ms\":%.6g}",
             js.size() > 1 ? "," : "", kv.first.c_str(), kv.second.n, kv.second.flops, kv.second.ms);
    js += row;
  }
  js += "]";
  if ((int64_t)js.size() + 1 > len) return x->fail(PEPSVMC_EINVAL, "profile text longer than the buffer");
  memcpy(buf, js.c_str(), js.size() + 1);
  return PEPSVMC_OK;
}

int pepsvmc_set_proposal_params(pepsvmc_ctx* x, const double* params) {
  if (!x || !params) return PEPSVMC_EINVAL;
  cudaError_t e = x->net_alloc();
  if (e != cudaSuccess) return x->fail(PEPSVMC_ENOMEM, "proposal network allocation failed");
  std::vector<float> h(params, params + kNetParams);
  if ((e = x->cps(x->net, h.data(), h.size() * sizeof(float), cudaMemcpyHostToDevice))) return x->fail_cuda(e);
  x->net_ready = true;
  x->drop_graph();
  x->eager_steps = 0;
  return PEPSVMC_OK;
}

int pepsvmc_get_proposal_params(pepsvmc_ctx* x, double* out) {
  if (!x || !out) return PEPSVMC_EINVAL;
  if (!x->net_ready) return x->fail(PEPSVMC_ESTATE, "no proposal network: call pepsvmc_set_proposal_params");
  std::vector<float> h(kNetParams);
  cudaError_t e = x->cps(h.data(), x->net, h.size() * sizeof(float), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return x->fail_cuda(e);
  for (int i = 0; i < kNetParams; ++i) out[i] = h[i];
  return PEPSVMC_OK;
}

int pepsvmc_proposal_logits(pepsvmc_ctx* x, double* out) {
  if (!x || !out) return PEPSVMC_EINVAL;
  if (!x->net_ready) return x->fail(PEPSVMC_ESTATE, "no proposal network: call pepsvmc_set_proposal_params");
  const long long n = (long long)x->C * 2 * x->Ly * x->Lx;
  cudaError_t e = net_forward(NetParams::at(x->net), x->spins, x->C, x->Ly, x->Lx, x->h1, x->h2, x->logits, x->st);
  std::vector<float> h(n);
  if (e == cudaSuccess) e = x->cps(h.data(), x->logits, n * sizeof(float), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return x->fail_cuda(e);
  for (long long i = 0; i < n; ++i) out[i] = h[i];
  return PEPSVMC_OK;
}

int pepsvmc_proposal_collect(pepsvmc_ctx* x, int32_t n_sweeps) {
  if (!x || n_sweeps < 1) return PEPSVMC_EINVAL;
  const long long N = (long long)x->Ly * x->Lx, need = x->ds_n + (long long)n_sweeps * x->C;
  cudaError_t e = cudaSuccess;
  if (need > x->ds_cap) {
    int8_t* s2 = nullptr;
    float* r2 = nullptr;
    if ((e = x->alloc(&s2, (size_t)need * N)) || (e = x->alloc(&r2, (size_t)need * 2 * N)))
      return x->fail(PEPSVMC_ENOMEM, "training set allocation failed");
    if (x->ds_n && ((e = x->cp(s2, x->ds_spins, x->ds_n * N, cudaMemcpyDeviceToDevice)) ||
                    (e = x->cp(r2, x->ds_rho, x->ds_n * 2 * N * sizeof(float), cudaMemcpyDeviceToDevice))))
      return x->fail_cuda(e);
    x->ds_spins = s2;
    x->ds_rho = r2;
    x->ds_cap = need;
  }
  for (int t = 0; t < n_sweeps; ++t) {
    if ((e = x->set_sweep()) || (e = x->sweep_once())) return x->fail_cuda(e);
    x->rho_export = x->ds_rho + x->ds_n * 2 * N;
    e = x->measure_dev();
    x->rho_export = nullptr;
    if (e || (e = x->cp(x->ds_spins + x->ds_n * N, x->spins, (size_t)x->C * N, cudaMemcpyDeviceToDevice)))
      return x->fail_cuda(e);
    x->ds_n += x->C;
    ++x->sweep_counter;
  }
  return x->check_status();
}

int64_t pepsvmc_proposal_dataset_size(const pepsvmc_ctx* x) { return x ? x->ds_n : 0; }

int pepsvmc_train_proposal(pepsvmc_ctx* x, const int8_t* configs, int64_t n, int32_t epochs, double lr,
                           double* final_loss_out) {
  if (!x || !configs || n < 1 || epochs < 1 || !(lr > 0.0)) return PEPSVMC_EINVAL;
  if (!x->net_ready) return x->fail(PEPSVMC_ESTATE, "no proposal network: call pepsvmc_set_proposal_params");
  const long long N = (long long)x->Ly * x->Lx;
  for (long long i = 0; i < n * N; ++i)
    if (configs[i] != 1 && configs[i] != -1) return x->fail(PEPSVMC_EINVAL, "configurations must be +1 or -1");
  cudaError_t e = cudaSuccess;
  // the training set is replaced; a measurement exports the ratios of all C chains, so
  // the last (partial) batch needs room for C entries
  const long long need = n + x->C;
  if (need > x->ds_cap) {
    int8_t* s2 = nullptr;
    float* r2 = nullptr;
    if ((e = x->alloc(&s2, (size_t)need * N)) || (e = x->alloc(&r2, (size_t)need * 2 * N)))
      return x->fail(PEPSVMC_ENOMEM, "training set allocation failed");
    x->ds_spins = s2;
    x->ds_rho = r2;
    x->ds_cap = need;
  }
  if (!x->spins_saved && (e = x->alloc(&x->spins_saved, (size_t)x->C * N)))
    return x->fail(PEPSVMC_ENOMEM, "allocation failed");
  if ((e = x->cp(x->spins_saved, x->spins, (size_t)x->C * N, cudaMemcpyDeviceToDevice))) return x->fail_cuda(e);
  x->ds_n = 0;
  std::vector<int8_t> batch((size_t)x->C * N);
  for (long long b0 = 0; b0 < n; b0 += x->C) {
    const long long cnt = std::min<long long>(x->C, n - b0);
    for (long long c = 0; c < x->C; ++c)
      memcpy(&batch[(size_t)(c * N)], configs + (b0 + (c < cnt ? c : 0)) * N, (size_t)N);
    if ((e = x->cps(x->spins, batch.data(), batch.size(), cudaMemcpyHostToDevice))) return x->fail_cuda(e);
    x->top_valid = false;
    x->rho_export = x->ds_rho + x->ds_n * 2 * N;
    e = x->measure_dev();
    x->rho_export = nullptr;
    if (e || (e = x->cp(x->ds_spins + x->ds_n * N, x->spins, (size_t)cnt * N, cudaMemcpyDeviceToDevice)))
      return x->fail_cuda(e);
    x->ds_n += cnt;
    const int rc = x->check_status();
    if (rc) return rc;
  }
  if ((e = x->cp(x->spins, x->spins_saved, (size_t)x->C * N, cudaMemcpyDeviceToDevice))) return x->fail_cuda(e);
  x->top_valid = false;
  x->have_measure = false;
  e = x->train_epochs(epochs, (int)std::min<long long>(256, x->ds_n), (float)lr, final_loss_out);
  if (e != cudaSuccess) return x->fail_cuda(e);
  x->drop_graph();
  x->eager_steps = 0;
  return x->check_status();
}

int pepsvmc_proposal_load(pepsvmc_ctx* x, const int8_t* spins, const double* rho, int64_t n) {
  if (!x || !spins || !rho || n < 1) return PEPSVMC_EINVAL;
  const long long N = (long long)x->Ly * x->Lx;
  cudaError_t e;
  if (n > x->ds_cap) {
    if ((e = x->alloc(&x->ds_spins, (size_t)n * N)) || (e = x->alloc(&x->ds_rho, (size_t)n * 2 * N)))
      return x->fail(PEPSVMC_ENOMEM, "training set allocation failed");
    x->ds_cap = n;
  }
  std::vector<float> r(rho, rho + n * 2 * N);
  if ((e = x->cps(x->ds_spins, spins, (size_t)n * N, cudaMemcpyHostToDevice)) ||
      (e = x->cps(x->ds_rho, r.data(), r.size() * sizeof(float), cudaMemcpyHostToDevice)))
    return x->fail_cuda(e);
  x->ds_n = n;
  return PEPSVMC_OK;
}

int pepsvmc_proposal_train(pepsvmc_ctx* x, int32_t epochs, int32_t batch, double lr, double* loss_out) {
  if (!x || epochs < 1 || batch < 1) return PEPSVMC_EINVAL;
  if (!x->net_ready) return x->fail(PEPSVMC_ESTATE, "no proposal network: call pepsvmc_set_proposal_params");
  if (x->ds_n < batch) return x->fail(PEPSVMC_ESTATE, "training set smaller than one batch");
  cudaError_t e = x->train_epochs(epochs, batch, (float)lr, loss_out);
  if (e != cudaSuccess) return x->fail_cuda(e);
  x->drop_graph();
  x->eager_steps = 0;
  return x->check_status();
}

int pepsvmc_set_proposal(pepsvmc_ctx* x, int32_t mode) {
  if (!x || mode < 0 || mode > 1) return PEPSVMC_EINVAL;
  if (mode == 1 && x->sym) return x->fail(PEPSVMC_EINVAL, "symmetrize: only the sequential sweep samples |Phi|^2");
  if (mode == 1 && !x->net_ready) return x->fail(PEPSVMC_ESTATE, "no proposal network: call pepsvmc_set_proposal_params");
  x->proposal_mode = mode;
  x->drop_graph();
  x->eager_steps = 0;
  return PEPSVMC_OK;
}

int pepsvmc_learned_sweep(pepsvmc_ctx* x, int32_t n, double* rate) {
  if (!x || n < 0) return PEPSVMC_EINVAL;
  if (x->sym) return x->fail(PEPSVMC_EINVAL, "symmetrize: only the sequential sweep samples |Phi|^2");
  if (!x->net_ready) return x->fail(PEPSVMC_ESTATE, "no proposal network: call pepsvmc_set_proposal_params");
  cudaError_t e = x->ms(x->lcount, 0, 2 * sizeof(unsigned long long));
  for (int i = 0; i < n && e == cudaSuccess; ++i) {
    e = x->set_sweep();
    if (e == cudaSuccess) e = x->learned_sweep();
    ++x->sweep_counter;
  }
  if (e != cudaSuccess) return x->fail_cuda(e);
  int rc = x->check_status();
  if (rc) return rc;
  if (rate) {
    unsigned long long h[2] = {0, 0};
    if ((e = x->cps(h, x->lcount, sizeof(h), cudaMemcpyDeviceToHost))) return x->fail_cuda(e);
    *rate = h[0] ? (double)h[1] / (double)h[0] : 0.0;
  }
  return PEPSVMC_OK;
}

int pepsvmc_get_learned_trace(pepsvmc_ctx* x, double* rho, double* dlq, int8_t* dec) {
  if (!x) return PEPSVMC_EINVAL;
  if (!x->net || !x->trace_on) return x->fail(PEPSVMC_ESTATE, "learned trace needs a network and tracing on");
  const size_t n = (size_t)x->C * (x->Ly - 1);
  cudaError_t e = cudaSuccess;
  if (rho) e = x->cp(rho, x->ltr_rho, n * sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && dlq) e = x->cp(dlq, x->ltr_dlq, n * sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && dec) e = x->cp(dec, x->ltr_dec, n, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = x->sync();
  return e == cudaSuccess ? PEPSVMC_OK : x->fail_cuda(e);
}

int pepsvmc_set_graphs(pepsvmc_ctx* x, int32_t on) {
  if (!x) return PEPSVMC_EINVAL;
  x->use_graphs = on != 0;
  x->drop_graph();
  x->eager_steps = 0;
  return PEPSVMC_OK;
}

int pepsvmc_set_autotune(pepsvmc_ctx* x, int32_t on) {
  if (!x) return PEPSVMC_EINVAL;
  x->autotune = on != 0;
  if (!on) x->tuned.clear();
  x->drop_graph();
  x->eager_steps = 0;
  return PEPSVMC_OK;
}

int pepsvmc_set_contraction_kernel(pepsvmc_ctx* x, int32_t kind, int32_t tile) {
  if (!x) return PEPSVMC_EINVAL;
  int choice = -1;
  if (kind == 1 && tile >= 0 && tile < gemm_f32_num_configs()) choice = tile;
  if (kind == 2 && x->tc_mode() && (tile == 32 || tile == 64 || tile == 128 || tile == 256)) choice = 100 + tile;
  if (kind == 3 && x->tc_mode() == 3 && (tile == 32 || tile == 64)) choice = 1000 + tile;
  if (kind != 0 && choice < 0) return x->fail(PEPSVMC_EINVAL, "no such contraction kernel for this precision");
  x->forced = choice;
  x->drop_graph();
  x->eager_steps = 0;
  return PEPSVMC_OK;
}

int pepsvmc_get_tuning(pepsvmc_ctx* x, char* buf, int64_t len) {
  if (!x || !buf || len < 2) return PEPSVMC_EINVAL;
  std::string js = "[";
  for (const auto& kv : x->tuned) {
    const int c = kv.second;
    std::string times;
    for (float t : x->tune_ms[kv.first]) times += (times.empty() ? "" : ",") + std::to_string(t);
    char row[512];
    snprintf(row, sizeof(row), "%s{\"shape\":\"%s\",\"choice\":\"%s%d\",\"candidate_ms\":[%s]}",
             js.size() > 1 ? "," : "", kv.first.c_str(), c >= 1000 ? "tc2_bn" : c >= 100 ? "tc_bn" : "f32_cfg",
             c >= 1000 ? c - 1000 : c >= 100 ? c - 100 : c,
             times.c_str());
    js += row;
  }
  js += "]";
  if ((int64_t)js.size() + 1 > len) return x->fail(PEPSVMC_EINVAL, "tuning text longer than the buffer");
  memcpy(buf, js.c_str(), js.size() + 1);
  return PEPSVMC_OK;
}

int pepsvmc_get_profile(pepsvmc_ctx* x, double* out) {
  if (!x || !out) return PEPSVMC_EINVAL;
  cudaError_t e = x->collect();
  if (e != cudaSuccess) return x->fail_cuda(e);
  for (int i = 0; i < 6; ++i) out[i] = x->prof_acc[i];
  return PEPSVMC_OK;
}

int pepsvmc_set_spins(pepsvmc_ctx* x, const int8_t* s) {
  if (!x || !s) return PEPSVMC_EINVAL;
  const size_t n = (size_t)x->C * x->Ly * x->Lx;
  for (size_t i = 0; i < n; ++i)
    if (s[i] != 1 && s[i] != -1) return x->fail(PEPSVMC_EINVAL, "spins must be +1 or -1");
  if (x->sym) {
    const size_t half = n / 2;
    for (size_t i = 0; i < half; ++i)
      if (s[half + i] != -s[i])
        return x->fail(PEPSVMC_EINVAL, "symmetrize: chain p + n_chains/2 must be the inversion of chain p");
  }
  cudaError_t e = x->cp(x->spins, s, n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = x->sync();
  if (e != cudaSuccess) return x->fail_cuda(e);
  x->top_valid = false;
  return PEPSVMC_OK;
}

int pepsvmc_get_spins(pepsvmc_ctx* x, int8_t* s) {
  if (!x || !s) return PEPSVMC_EINVAL;
  cudaError_t e = x->cp(s, x->spins, (size_t)x->C * x->Ly * x->Lx, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = x->sync();
  return e == cudaSuccess ? PEPSVMC_OK : x->fail_cuda(e);
}

int pepsvmc_set_tensors(pepsvmc_ctx* x, const double* t) {
  if (!x || !t) return PEPSVMC_EINVAL;
  cudaError_t e = x->cp(x->master, t, x->P * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = x->refresh_perms();
  if (e == cudaSuccess) e = x->sync();
  if (e != cudaSuccess) return x->fail_cuda(e);
  x->top_valid = false;
  return PEPSVMC_OK;
}

int pepsvmc_get_tensors(pepsvmc_ctx* x, double* t) {
  if (!x || !t) return PEPSVMC_EINVAL;
  cudaError_t e = x->cp(t, x->master, x->P * sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = x->sync();
  return e == cudaSuccess ? PEPSVMC_OK : x->fail_cuda(e);
}

int pepsvmc_set_sweep_counter(pepsvmc_ctx* x, uint64_t s) {
  if (!x) return PEPSVMC_EINVAL;
  x->sweep_counter = s;
  return PEPSVMC_OK;
}
uint64_t pepsvmc_get_sweep_counter(const pepsvmc_ctx* x) { return x ? x->sweep_counter : 0; }

int pepsvmc_enable_trace(pepsvmc_ctx* x, int32_t on) {
  if (!x) return PEPSVMC_EINVAL;
  if (on && !x->trace_ratio) {
    cudaError_t e;
    if ((e = x->alloc(&x->trace_ratio, (size_t)x->C * x->nbonds())) != cudaSuccess ||
        (e = x->alloc(&x->trace_dec, (size_t)x->C * x->nbonds())) != cudaSuccess)
      return x->fail(PEPSVMC_ENOMEM, "trace allocation failed");
  }
  x->trace_on = on ? 1 : 0;
  return PEPSVMC_OK;
}

int pepsvmc_get_trace(pepsvmc_ctx* x, double* ratio, int8_t* decision) {
  if (!x) return PEPSVMC_EINVAL;
  if (!x->trace_ratio) return x->fail(PEPSVMC_ESTATE, "trace not enabled");
  const size_t n = (size_t)x->C * x->nbonds();
  cudaError_t e = cudaSuccess;
  if (ratio) e = x->cp(ratio, x->trace_ratio, n * sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && decision) e = x->cp(decision, x->trace_dec, n, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = x->sync();
  return e == cudaSuccess ? PEPSVMC_OK : x->fail_cuda(e);
}

int pepsvmc_sample_sweep(pepsvmc_ctx* x, int32_t n, double* rate) {
  if (!x || n < 0) return PEPSVMC_EINVAL;
  cudaError_t e = x->ms(x->counters, 0, 2 * sizeof(unsigned long long));
  for (int i = 0; i < n && e == cudaSuccess; ++i) {
    e = x->set_sweep();
    if (e == cudaSuccess) e = x->sweep_once();
    ++x->sweep_counter;
  }
  if (e != cudaSuccess) return x->fail_cuda(e);
  int rc = x->check_status();
  if (rc) return rc;
  if (rate) {
    unsigned long long h[2];
    e = x->cps(h, x->counters, sizeof(h), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return x->fail_cuda(e);
    *rate = h[0] ? (double)h[1] / (double)h[0] : 0.0;
  }
  return PEPSVMC_OK;
}

int pepsvmc_measure(pepsvmc_ctx* x, double* eloc, double* logpsi, int8_t* sign) {
  if (!x) return PEPSVMC_EINVAL;
  cudaError_t e = x->measure_dev();
  if (e != cudaSuccess) return x->fail_cuda(e);
  int rc = x->check_status();
  if (rc) return rc;
  if (eloc && (e = x->cps(eloc, x->eloc, x->C * sizeof(double), cudaMemcpyDeviceToHost))) return x->fail_cuda(e);
  if (logpsi && (e = x->cps(logpsi, x->logpsi, x->C * sizeof(double), cudaMemcpyDeviceToHost))) return x->fail_cuda(e);
  if (sign && (e = x->cps(sign, x->sign, x->C, cudaMemcpyDeviceToHost))) return x->fail_cuda(e);
  return PEPSVMC_OK;
}

int pepsvmc_get_phi(pepsvmc_ctx* x, double* eloc_phi, double* w) {
  if (!x) return PEPSVMC_EINVAL;
  if (!x->sym) return x->fail(PEPSVMC_ESTATE, "get_phi: the context was created without symmetrize");
  if (!x->have_measure) return x->fail(PEPSVMC_ESTATE, "no measurement yet");
  cudaError_t e = cudaSuccess;
  if (eloc_phi) e = x->cp(eloc_phi, x->eloc_phi, x->pairs * sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && w) e = x->cp(w, x->phi_wm, x->pairs * sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = x->sync();
  return e == cudaSuccess ? PEPSVMC_OK : x->fail_cuda(e);
}

int pepsvmc_get_chain_grad(pepsvmc_ctx* x, int32_t chain, double* out) {
  if (!x || !out || chain < 0 || chain >= x->C) return PEPSVMC_EINVAL;
  if (!x->have_measure) return x->fail(PEPSVMC_ESTATE, "no measurement yet");
  std::vector<float> h(x->Ph);
  cudaError_t e = x->cps(h.data(), x->G + (long long)chain * x->Ph, x->Ph * sizeof(float), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return x->fail_cuda(e);
  for (long long i = 0; i < x->Ph; ++i) out[i] = h[i];
  return PEPSVMC_OK;
}

int pepsvmc_amplitude(pepsvmc_ctx* x, int32_t row, double* logpsi, int8_t* sign) {
  if (!x || row < 0 || row >= x->Ly) return PEPSVMC_EINVAL;
  cudaError_t e = x->amplitude_dev(row);
  if (e != cudaSuccess) return x->fail_cuda(e);
  int rc = x->check_status();
  if (rc) return rc;
  if (logpsi && (e = x->cps(logpsi, x->logpsi, x->C * sizeof(double), cudaMemcpyDeviceToHost))) return x->fail_cuda(e);
  if (sign && (e = x->cps(sign, x->sign, x->C, cudaMemcpyDeviceToHost))) return x->fail_cuda(e);
  return PEPSVMC_OK;
}

int pepsvmc_energy_and_grad(pepsvmc_ctx* x, int32_t n, double* E_mean, double* E_var, double* eloc,
                            double* logpsi, int8_t* sign, double* grad) {
  if (!x || n < 1) return PEPSVMC_EINVAL;
  cudaError_t e = cudaSuccess;
  if ((e = x->ms(x->sumG, 0, x->P * sizeof(double))) ||
      (e = x->ms(x->sumGE, 0, x->P * sizeof(double))) ||
      (e = x->ms(x->sums, 0, 4 * sizeof(double))) ||
      (e = x->ms(x->counters, 0, 2 * sizeof(unsigned long long))))
    return x->fail_cuda(e);
  for (int t = 0; t < n; ++t) {
    if ((e = x->sample_step())) return x->fail_cuda(e);
    ++x->sweep_counter;
    x->top_valid = true;
    x->have_measure = true;
    if (eloc && (e = x->cp(eloc + (size_t)t * x->C, x->sym ? x->eloc_phi : x->eloc, x->C * sizeof(double),
                           cudaMemcpyDeviceToHost)))
      return x->fail_cuda(e);
    if (logpsi && (e = x->cp(logpsi + (size_t)t * x->C, x->logpsi, x->C * sizeof(double), cudaMemcpyDeviceToHost)))
      return x->fail_cuda(e);
    if (sign && (e = x->cp(sign + (size_t)t * x->C, x->sign, x->C, cudaMemcpyDeviceToHost)))
      return x->fail_cuda(e);
  }
  ++x->launches;
  if ((e = k_grad_final(x->sumG, x->sumGE, x->sums, x->P, x->grad, x->st))) return x->fail_cuda(e);
  int rc = x->check_status();
  if (rc) return rc;
  x->have_grad = true;
  double s[4];
  if ((e = x->cps(s, x->sums, sizeof(s), cudaMemcpyDeviceToHost))) return x->fail_cuda(e);
  const double mean = s[0] / s[2];
  if (E_mean) *E_mean = mean;
  if (E_var) *E_var = s[1] / s[2] - mean * mean;
  if (grad && (e = x->cps(grad, x->grad, x->P * sizeof(double), cudaMemcpyDeviceToHost))) return x->fail_cuda(e);
  return PEPSVMC_OK;
}

int pepsvmc_random_sweep(pepsvmc_ctx* x, int32_t n, double* rate) {
  if (!x || n < 0) return PEPSVMC_EINVAL;
  if (x->sym) return x->fail(PEPSVMC_EINVAL, "symmetrize: only the sequential sweep samples |Phi|^2");
  cudaError_t e = x->ms(x->counters, 0, 2 * sizeof(unsigned long long));
  for (int i = 0; i < n && e == cudaSuccess; ++i) {
    e = x->set_sweep();
    if (e == cudaSuccess) e = x->random_sweep();
    ++x->sweep_counter;
  }
  if (e != cudaSuccess) return x->fail_cuda(e);
  int rc = x->check_status();
  if (rc) return rc;
  if (rate) {
    unsigned long long h[2];
    e = x->cps(h, x->counters, sizeof(h), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return x->fail_cuda(e);
    *rate = h[0] ? (double)h[1] / (double)h[0] : 0.0;
  }
  return PEPSVMC_OK;
}

int pepsvmc_get_random_trace(pepsvmc_ctx* x, int32_t* bond, double* ratio, int8_t* decision) {
  if (!x) return PEPSVMC_EINVAL;
  if (!x->r_tr_bond || !x->trace_on) return x->fail(PEPSVMC_ESTATE, "no traced random sweep");
  const size_t n = (size_t)x->C * x->Ly * x->Lx;
  cudaError_t e = cudaSuccess;
  if (bond) e = x->cp(bond, x->r_tr_bond, n * sizeof(int), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && ratio) e = x->cp(ratio, x->r_tr_ratio, n * sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && decision) e = x->cp(decision, x->r_tr_dec, n, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = x->sync();
  return e == cudaSuccess ? PEPSVMC_OK : x->fail_cuda(e);
}

int pepsvmc_set_fused(pepsvmc_ctx* x, int32_t on) {
  if (!x) return PEPSVMC_EINVAL;
  x->fused_on = on != 0;
  x->drop_graph();
  return PEPSVMC_OK;
}

int pepsvmc_set_wait_budget(pepsvmc_ctx* x, uint64_t cycles) {
  if (!x) return PEPSVMC_EINVAL;
  if (cycles > (uint64_t)1 << 62) return x->fail(PEPSVMC_EINVAL, "wait budget too large");
  x->wait_budget = (long long)cycles;
  x->drop_graph();  // a captured step carries the old budget in its launch arguments
  return PEPSVMC_OK;
}

int pepsvmc_get_sums(pepsvmc_ctx* x, double* scalars, double* sumGE, double* sumG) {
  if (!x || !scalars) return PEPSVMC_EINVAL;
  if (!x->have_grad) return x->fail(PEPSVMC_ESTATE, "no sums: call pepsvmc_energy_and_grad first");
  cudaError_t e = x->cp(scalars, x->sums, 3 * sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && sumGE) e = x->cp(sumGE, x->sumGE, x->P * sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && sumG) e = x->cp(sumG, x->sumG, x->P * sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = x->sync();
  return e == cudaSuccess ? PEPSVMC_OK : x->fail_cuda(e);
}

int pepsvmc_finalize_sums(pepsvmc_ctx* x) {
  if (!x) return PEPSVMC_EINVAL;
  double n = 0.0;
  cudaError_t e = x->cps(&n, x->sums + 2, sizeof(double), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return x->fail_cuda(e);
  if (!x->dry && !(n > 0.0)) return x->fail(PEPSVMC_EINVAL, "sums: the sample count must be positive");
  ++x->launches;
  if ((e = k_grad_final(x->sumG, x->sumGE, x->sums, x->P, x->grad, x->st)) != cudaSuccess) return x->fail_cuda(e);
  if ((e = x->sync()) != cudaSuccess) return x->fail_cuda(e);
  x->have_grad = true;
  return PEPSVMC_OK;
}

int pepsvmc_set_sums(pepsvmc_ctx* x, const double* scalars, const double* sumGE, const double* sumG) {
  if (!x || !scalars || !sumGE || !sumG) return PEPSVMC_EINVAL;
  if (!(scalars[2] > 0.0)) return x->fail(PEPSVMC_EINVAL, "sums: the sample count must be positive");
  cudaError_t e = x->cp(x->sums, scalars, 3 * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = x->cp(x->sumGE, sumGE, x->P * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = x->cp(x->sumG, sumG, x->P * sizeof(double), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return x->fail_cuda(e);
  return pepsvmc_finalize_sums(x);
}

int pepsvmc_sums_device(pepsvmc_ctx* x, double** scalars, double** sumGE, double** sumG) {
  if (!x || !scalars || !sumGE || !sumG) return PEPSVMC_EINVAL;
  *scalars = x->sums;
  *sumGE = x->sumGE;
  *sumG = x->sumG;
  return PEPSVMC_OK;
}

int pepsvmc_update(pepsvmc_ctx* x, double delta, uint64_t step) {
  if (!x) return PEPSVMC_EINVAL;
  if (!x->have_grad) return x->fail(PEPSVMC_ESTATE, "no gradient: call pepsvmc_energy_and_grad first");
  ++x->launches;
  cudaError_t e = k_sgd(x->master, x->grad, x->P, delta, x->cfg.seed, step, x->st);
  if (e == cudaSuccess) e = x->refresh_perms();
  if (e == cudaSuccess) e = x->sync();
  if (e != cudaSuccess) return x->fail_cuda(e);
  x->top_valid = false;
  return PEPSVMC_OK;
}

}  // extern "C"
