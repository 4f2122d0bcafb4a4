// The tick engine: a set of simulations advanced together by one captured
// CUDA graph of phase-gated kernels. One tick is
//   k_open, then iters_per_tick x (k_apply_dot, k_update),
// over device-side work lists of (simulation, operator tile) and
// (simulation, pointwise chunk) pairs. Each simulation carries its own phase,
// so simulations of different sizes, at different steps and iterations, share
// every launch; the host only replays the graph and polls a counter of
// unfinished simulations every few ticks (the paper's host reads the residual
// back after every iteration, §3.4.3).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "engine.h"
#include "loop_kernels.cuh"
#include "open_kernels.cuh"
#include "res_kernels.cuh"

namespace heat {

using TileFn = void (*)(const SimDev*, const int2*, const int*);

struct KernelSet {
  TileFn open, apply, update;
  int sx, sy;
  int open_threads, apply_threads;
  // warp-segment apply; when set it replaces `apply` (always on the FP64 path)
  TileFn apply_w;
  int wsx, wny, wwarps;
  int pw_chunk;  // nodes per pointwise (k_update) work item
  int seg_nodes[3];  // warp-segment tile size per mesh-size bucket
  int apply_w_smem;  // dynamic shared memory of apply_w per block
  bool fused;        // apply_w is k_cg_iter: one kernel per CG iteration, no update kernel
  // Chebyshev passes: block form, and the warp form matching apply_w (which
  // then replaces it, on the same work list)
  TileFn cheb, cheb_w;
  // step-start and refinement passes in the warp-segment march (replaces
  // `open` when set), on their own segment geometry and work list
  TileFn open_w = nullptr;
  int owsx = 0, owny = 0, owwarps = 0;
  int w_occ = 0, o_occ = 0;  // blocks of apply_w and open_w resident on an SM (0: unknown)
  // the CG iterations of a tick as one persistent kernel (replaces the
  // apply and update launches when set; FP32 paths, register-prefetch apply)
  LoopFn loop = nullptr;
  bool auto_seg = false;  // a default form: segment size kAutoSeg stands for the estimated best height
  bool dual = false;  // apply_w takes 16- and 32-lane segments, chosen per mesh (wsx for Chebyshev members)
  // the inner solve held on the chip: iterates the members whose mesh fits
  // (SimDev::res.g > 0); the others take apply and update
  ResFn res = nullptr;
  int res_blocks = 0, res_smem = 0;  // resident blocks, dynamic shared memory limit
};

// The warp-segment forms of k_open (tuning open_w): 32-lane segments of 2
// rows (shape 1) or 1 row (shape 2), 4 warps per block; double-float on the
// FP32 paths, FP64 on the FP64 path. Two rows hold twice the double-width
// values of a lane (254 registers, 2 blocks per SM); one row fits 168
// registers and 3 blocks per SM at the cost of more halo rows per output.
constexpr int kOpenSX = 32, kOpenWarps = 4;
static int open_w_rows(int shape) { return shape == 2 ? 1 : 2; }
static TileFn open_w_kernel(int prec, int shape) {
  if (shape == 2) {
    switch (prec) {
      case P_FP64: return k_open_w<P_FP64, kOpenSX, 1, kOpenWarps, 3>;
      case P_FP32_REFINED: return k_open_w<P_FP32_REFINED, kOpenSX, 1, kOpenWarps, 3>;
      default: return k_open_w<P_FP32_PLAIN, kOpenSX, 1, kOpenWarps, 3>;
    }
  }
  switch (prec) {
    case P_FP64: return k_open_w<P_FP64, kOpenSX, 2, kOpenWarps, 1>;
    case P_FP32_REFINED: return k_open_w<P_FP32_REFINED, kOpenSX, 2, kOpenWarps, 2>;
    default: return k_open_w<P_FP32_PLAIN, kOpenSX, 2, kOpenWarps, 2>;
  }
}

template <int P, int SX, int SY, int E = E_Q1>
static KernelSet make_set() {
  using T = typename std::conditional<P == P_FP64, double, float>::type;
  TileFn apply = nullptr, cheb = nullptr;  // FP64 has no block-tile form of these
  if constexpr (P != P_FP64) {
    apply = k_apply_dot<T, SX, SY, E>;
    cheb = k_cheb<T, SX, SY, E>;
  }
  return {k_open<P, SX, SY, E>, apply, k_update<T, P, sizeof(T) == 4 ? 4 : 2>, SX, SY, SX * SY,
          SX * SY, nullptr, 0, 0, 0, pw_chunk(sizeof(T) == 4 ? 4 : 2), {512, 512, 512}, 0, false,
          cheb, nullptr};
}

// Warp-segment apply variants the tuner chooses from: segment width, rows per
// lane, warps per block, cp.async stages (0: register prefetch); f64 is null
// where the FP64 registers or shared memory do not fit. Each kernel exists
// for both elements (the march differs, op_warp.cuh); index 0 trilinear
// boxes, 1 six-tetrahedra boxes.
struct WVariant {
  int sx, ny, warps, stages;
  TileFn f32[2], f64[2];
  int smem32, smem64;  // dynamic shared memory per block
  bool fused;          // FP32 only: the fused iteration kernel k_cg_iter
  TileFn cheb32[2], cheb64[2];  // Chebyshev passes of this segment shape (null: fused)
  bool res = false;    // FP32 only: meshes that fit iterate on the chip (k_cg_res)
};
// One register-prefetch Chebyshev pass kernel per segment shape and type,
// bounded like that shape's register-prefetch apply (FP64: one block per SM).
template <class T, int SX, int NY, int W, bool ON, int E>
static constexpr TileFn chebfn() {
  if constexpr (!ON) {
    return nullptr;
  } else if constexpr (sizeof(T) == 8) {
    return k_cheb_w<double, SX, NY, W, 1, E>;
  } else {
    constexpr int MINB = (SX == 16 && NY == 2) ? 2 : ((SX == 32 && NY == 2) ? 4 : 3);
    return k_cheb_w<float, SX, NY, W, MINB, E>;
  }
}
template <class T, int SX, int NY, int W, int S, int MINB, bool ON, int E>
static constexpr TileFn wfn() {
  if constexpr (ON) return k_apply_dot_w<T, SX, NY, W, S, MINB, E>;
  else return nullptr;
}
template <int SX, int NY, int W, int S, int MINB, int MINB64>
static constexpr WVariant wv() {
  return {SX,
          NY,
          W,
          S,
          {wfn<float, SX, NY, W, S, MINB, true, E_Q1>(), wfn<float, SX, NY, W, S, MINB, true, E_P1>()},
          {wfn<double, SX, NY, W, S, MINB64, (MINB64 > 0), E_Q1>(),
           wfn<double, SX, NY, W, S, MINB64, (MINB64 > 0), E_P1>()},
          S ? 32 * W * async_stage_bytes<float, NY, (S ? S : 2)>() : 0,
          S ? 32 * W * async_stage_bytes<double, NY, (S ? S : 2)>() : 0,
          false,
          {chebfn<float, SX, NY, W, true, E_Q1>(), chebfn<float, SX, NY, W, true, E_P1>()},
          {chebfn<double, SX, NY, W, (MINB64 > 0), E_Q1>(), chebfn<double, SX, NY, W, (MINB64 > 0), E_P1>()}};
}
template <int SX, int NY, int W, int MINB>
static constexpr WVariant wv_fused() {
  return {SX, NY, W, 0, {k_cg_iter<SX, NY, W, MINB, E_Q1>, k_cg_iter<SX, NY, W, MINB, E_P1>}, {nullptr, nullptr},
          0,  0,  true, {nullptr, nullptr}, {nullptr, nullptr}};
}
// the on-chip inner solve where the mesh fits, this streaming shape elsewhere
template <int SX, int NY, int W, int MINB>
static constexpr WVariant wv_res() {
  WVariant v = wv<SX, NY, W, 0, MINB, 0>();
  v.res = true;
  v.f32[0] = k_apply_dot_w2<float, NY, W, MINB, E_Q1>;
  v.f32[1] = k_apply_dot_w2<float, NY, W, MINB, E_P1>;
  return v;
}
// (segment width, rows, warps, stages, min blocks per SM for float / double,
// 0 = no double kernel)
static const WVariant kVariants[] = {
    wv_res<16, 4, 4, 3>(), wv<32, 4, 4, 0, 3, 0>(), wv<16, 2, 8, 0, 2, 1>(), wv<32, 2, 4, 0, 4, 1>(),
    wv<16, 4, 4, 3, 4, 0>(), wv<32, 4, 4, 3, 4, 0>(), wv<16, 2, 8, 3, 2, 1>(), wv<32, 4, 4, 3, 3, 0>(),
    wv<32, 4, 4, 4, 3, 0>(),     wv_fused<16, 4, 4, 2>(), wv_fused<32, 4, 4, 2>(), wv_fused<16, 4, 4, 3>(),
    wv_fused<32, 4, 4, 3>(),     wv_fused<16, 2, 8, 2>(), wv_fused<32, 2, 4, 4>(), wv<16, 4, 4, 0, 3, 0>(),
};
constexpr int kNumVariants = (int)(sizeof(kVariants) / sizeof(kVariants[0]));

// Process-wide tuning table, read when an engine is created: the warp apply
// variant per precision (-1: FP32 the block-tile apply, FP64 the default form)
// and the segment tile size per mesh-size bucket. Both are fixed per simulation size, so results stay
// bitwise identical alone and in batches built under the same table.
constexpr int kAutoSeg = 512;  // the default segment size: under the default variants, levels per tile from pick_levels
static Tuning g_tuning = {{-1, 0, 0}, {kAutoSeg, kAutoSeg, kAutoSeg}, {2, 4, 4}, {2, 2, 2}, {0, 0, 0}};
static std::mutex g_tuning_mu;

int num_variants() { return kNumVariants; }

bool variant_info(int v, int info[6]) {
  if (v < 0 || v >= kNumVariants) return false;
  info[0] = kVariants[v].sx;
  info[1] = kVariants[v].ny;
  info[2] = kVariants[v].warps;
  info[3] = kVariants[v].f64[0] != nullptr;
  info[4] = kVariants[v].res ? -1 : kVariants[v].stages;
  info[5] = kVariants[v].fused;
  return true;
}

int size_bucket(long long nn) { return nn < 200000 ? 0 : (nn < 4000000 ? 1 : 2); }

Tuning tuning_get() {
  std::lock_guard<std::mutex> lock(g_tuning_mu);
  return g_tuning;
}

heat_status tuning_set(const Tuning& t) {
  for (int p = 0; p < 3; ++p) {
    const int v = t.variant[p];
    if (v < -1 || v >= kNumVariants || (v >= 0 && p == P_FP64 && !kVariants[v].f64[0]))
      return set_error(HEAT_ERR_ARG, "tuning: bad variant %d for precision %d", v, p);
  }
  for (int p = 0; p < 3; ++p)
    if (t.pw_quads[p] != 1 && t.pw_quads[p] != 2 && t.pw_quads[p] != 4)
      return set_error(HEAT_ERR_ARG, "tuning: pointwise groups %d not 1, 2 or 4", t.pw_quads[p]);
  for (int p = 0; p < 3; ++p)
    if (t.open_w[p] < 0 || t.open_w[p] > 2)
      return set_error(HEAT_ERR_ARG, "tuning: open_w[%d] = %d not 0, 1 or 2", p, t.open_w[p]);
  for (int p = 0; p < 3; ++p)
    if (t.loop[p] < 0 || t.loop[p] > 1 || (p == P_FP64 && t.loop[p] != 0))
      return set_error(HEAT_ERR_ARG, "tuning: loop[%d] = %d not 0 or 1 (0 for FP64)", p, t.loop[p]);
  for (int b = 0; b < 3; ++b)
    if (t.seg_nodes[b] < 32 || t.seg_nodes[b] > (1 << 20))
      return set_error(HEAT_ERR_ARG, "tuning: segment size %d out of range", t.seg_nodes[b]);
  std::lock_guard<std::mutex> lock(g_tuning_mu);
  g_tuning = t;
  return HEAT_OK;
}

template <class T, int P>
static TileFn update_for(int qpt) {
  return qpt == 1 ? k_update<T, P, 1> : (qpt == 2 ? k_update<T, P, 2> : k_update<T, P, 4>);
}
static TileFn update_kernel(int prec, int qpt) {
  switch (prec) {
    case P_FP64: return update_for<double, P_FP64>(qpt);
    case P_FP32_REFINED: return update_for<float, P_FP32_REFINED>(qpt);
    default: return update_for<float, P_FP32_PLAIN>(qpt);
  }
}

static int sm_count();

// ------------------------------------------------- the on-chip inner solve

// k_cg_res of this precision and element, when the device can run it: one
// block per SM, all resident at once (a cooperative launch).
static void res_kernel_set(KernelSet& k, bool fp64, int elem) {
  int dev = 0, coop = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  k.res = nullptr;
  if (!coop || optin < 96 * 1024) {
    cudaGetLastError();
    return;
  }
  ResFn fn = res_kernel(fp64, elem);
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, (const void*)fn) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  const int smem = (optin - (int)fa.sharedSizeBytes) & ~15;
  if (cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  k.res = fn;
  k.res_smem = smem;
  k.res_blocks = sm_count();
}

static int res_nodes(const ResGeo& r) { return r.bx * r.by * r.bz; }

// Estimated cycles of one iteration on boxes r, fitted to clock readings in
// the kernel (boxes of 16^3 to 105^3 meshes): a march layer takes a warp 850
// cycles alone on its scheduler and 690 beside others, a pointwise group of
// 4 nodes per thread 640 over the passes, an all-sum about 4,000 with its
// block barriers.
static double res_cycles(const ResGeo& r, bool fp64) {
  const double sums = r.g > 1 ? 7600.0 + 5.0 * r.g : 2100.0;
  if (fp64) {
    // a warp's FP64 instruction takes its scheduler 64 cycles; 27 + 6 of them per node and iteration
    const int warps = (res_nodes(r) + 31) / 32;
    return ((warps + 3) / 4) * 33.0 * 64.0 + 3000.0 + sums;
  }
  const ResLayout l = res_layout(r, false);
  const int pairs = (l.nseg * l.nyt + 1) / 2, chunks = (r.bz + r.zc - 1) / r.zc;
  const int per_sched = (pairs * chunks + 3) / 4;
  const double march = (r.zc + 1.3) * (per_sched > 1 ? 690.0 * per_sched : 850.0);
  return march + res_groups(r) * 640.0 + 900.0 + sums;
}

// The boxes of one simulation (res.g = 0: it does not fit or gains nothing).
// FP32: the least time^2 x blocks, halfway between the fastest simulation
// alone (all SMs) and the most simulations side by side (fewest SMs each).
// FP64 runs at 1/58 of the FP32 rate, so its time is arithmetic spread over
// the SMs: the fastest alone is also the best in a batch. A function of the
// mesh and the GPU only, so results are the same alone and in a batch.
static ResGeo res_search(int X, int Y, int Z, int max_blocks, int smem, bool fp64) {
  ResGeo best{};
  double best_cost = 1e300;
  auto ceil_div = [](int a, int b) { return (a + b - 1) / b; };
  for (int gz = 1, last_z = 0; gz <= std::min(Z, max_blocks); ++gz) {
    const int bz = ceil_div(Z, gz);
    if (bz == last_z) continue;
    last_z = bz;
    for (int gy = 1, last_y = 0; gy <= Y && ceil_div(Z, bz) * gy <= max_blocks; ++gy) {
      const int by = ceil_div(Y, gy);
      if (by == last_y) continue;
      last_y = by;
      for (int gx = 1, last_x = 0; gx <= 8; ++gx) {
        int bx = ceil_div(X, gx);
        if (gx > 1) bx = (bx + 3) & ~3;  // exchanged groups of 4 start at multiples of 4
        if (bx == last_x) continue;
        last_x = bx;
        ResGeo r{};
        r.gx = ceil_div(X, bx);
        r.gy = ceil_div(Y, by);
        r.gz = ceil_div(Z, bz);
        r.g = r.gx * r.gy * r.gz;
        r.bx = bx;
        r.by = by;
        r.bz = bz;
        r.zc = bz;
        if (r.g > max_blocks) continue;
        if (fp64 ? res_nodes(r) > kResMaxN * kResThreads : res_groups(r) > kResMaxQ) continue;
        if (res_layout(r, fp64).bytes > smem) continue;
        for (int chunks = 1; chunks <= (fp64 ? 1 : std::min(8, bz)); ++chunks) {
          r.zc = ceil_div(bz, chunks);
          const double t = res_cycles(r, fp64), cost = fp64 ? t : t * t * r.g;
          if (cost < best_cost) {
            best_cost = cost;
            best = r;
          }
        }
      }
    }
  }
  return best;
}

static ResGeo res_plan(const SimDev& d, const KernelSet& ks, bool fp64) {
  if (!ks.res || d.cheb_m >= 2) return ResGeo{};  // Chebyshev passes run on the streaming kernels
  using Key = std::tuple<int, int, int, int, int, bool>;
  static std::mutex mu;
  static std::map<Key, ResGeo> plans;  // searched once per mesh size, bounded
  const Key key{d.nx, d.ny, d.nz, ks.res_blocks, ks.res_smem, fp64};
  std::lock_guard<std::mutex> lock(mu);
  auto it = plans.find(key);
  if (it != plans.end()) return it->second;
  const ResGeo r = res_search(d.nx + 1, d.ny + 1, d.nz + 1, ks.res_blocks, ks.res_smem, fp64);
  if (plans.size() >= 1024) plans.clear();
  plans[key] = r;
  return r;
}

// Bytes of a simulation's exchange area and where its parts start.
struct ResBytes {
  size_t z, x, slots, tag, total;
};
static ResBytes res_bytes(const SimDev& d, bool fp64) {
  ResBytes b{};
  if (d.res.g < 1) return b;
  auto up = [](size_t n) { return (n + 255) & ~(size_t)255; };
  b.z = 0;
  const size_t nz = d.res.g > 1 ? (size_t)((d.nx + 4) & ~3) * (d.ny + 1) * (d.nz + 1) * (fp64 ? 16 : 8) : 0;
  b.x = up(nz);
  b.slots = b.x + (fp64 ? 0 : (size_t)d.res.g * 2 * res_groups(d.res) * kResThreads * sizeof(float4));
  b.tag = b.slots + up(2 * (size_t)res_mail(d.res.g) * sizeof(ulonglong2));
  b.total = b.tag + 256;
  return b;
}

// Blocks of a kernel resident on an SM (0: unknown, as without a GPU).
static int occupancy(TileFn fn, int threads, int smem) {
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return occ;
}

// The register-prefetch variant with a separate update of variant v's shape
// (variant 0, which streams as one, where there is none).
static int plain_of(int v) {
  const WVariant& f = kVariants[v];
  for (int a = 0; a < kNumVariants; ++a)
    if (!kVariants[a].fused && !kVariants[a].res && kVariants[a].stages == 0 && kVariants[a].sx == f.sx &&
        kVariants[a].ny == f.ny && kVariants[a].warps == f.warps)
      return a;
  return 0;
}

// The kernels of precision prec under tuning table t. With Chebyshev passes
// (cheb) a fused variant is replaced by the register-prefetch variant of the
// same segment shape: the fused iteration has no place for the passes.
static KernelSet kernel_set(int prec, const Tuning& t, bool cheb = false, int elem = E_Q1) {
  const int ei = elem == E_P1 ? 1 : 0;
  int variant = t.variant[prec];
  // the persistent iteration: FP32 paths, trilinear boxes, no Chebyshev passes;
  // the on-chip form makes way for the plain one of its shape
  const bool loop = t.loop[prec] && prec != P_FP64 && elem == E_Q1 && !cheb;
  if (loop && variant >= 0 && variant < kNumVariants && kVariants[variant].res) variant = plain_of(variant);
  if (cheb && variant >= 0 && variant < kNumVariants && kVariants[variant].fused) variant = plain_of(variant);
  KernelSet k;
  if (elem == E_P1)
    k = prec == P_FP64 ? make_set<P_FP64, 16, 16, E_P1>()
                       : (prec == P_FP32_REFINED ? make_set<P_FP32_REFINED, 16, 16, E_P1>()
                                                  : make_set<P_FP32_PLAIN, 16, 16, E_P1>());
  else
    k = prec == P_FP64 ? make_set<P_FP64, 16, 16>()
                       : (prec == P_FP32_REFINED ? make_set<P_FP32_REFINED, 16, 16>()
                                                  : make_set<P_FP32_PLAIN, 16, 16>());
  if (variant >= 0 && variant < kNumVariants) {
    const WVariant& v = kVariants[variant];
    k.apply_w = prec == P_FP64 ? v.f64[ei] : v.f32[ei];
    if (k.apply_w) {
      k.wsx = v.sx;
      k.wny = v.ny;
      k.wwarps = v.warps;
      k.apply_w_smem = prec == P_FP64 ? v.smem64 : v.smem32;
      k.fused = v.fused;
      k.cheb_w = prec == P_FP64 ? v.cheb64[ei] : v.cheb32[ei];
      if (k.apply_w_smem > 0)
        cudaFuncSetAttribute(k.apply_w, cudaFuncAttributeMaxDynamicSharedMemorySize, k.apply_w_smem);
      if (loop && !v.fused && v.stages == 0)  // register prefetch, separate update
        k.loop = loop_kernel(v.sx, v.ny, v.warps, t.pw_quads[prec]);
      if (v.res) {
        res_kernel_set(k, false, elem);
        k.dual = true;
        k.auto_seg = true;
      }
    }
  }
  if (prec == P_FP64 && variant < 0) {
    // FP64 by default: on the chip where the mesh fits; else 16-lane segments
    // of 4 rows (the FP64 pipe bounds the apply, and 4 rows compute 5 rows'
    // elements where 2 compute 3)
    res_kernel_set(k, true, elem);
    k.auto_seg = true;
    // One block of 8 warps per SM: with two smaller ones, blocks that start
    // early (programmatic launch) pile up two to an SM while others stay empty
    // (100^3: 23.0 ms a step against 19.1 with the block tiles).
    k.apply_w = ei ? k_apply_dot_w<double, 16, 4, 8, 0, 1, E_P1> : k_apply_dot_w<double, 16, 4, 8, 0, 1, E_Q1>;
    k.wsx = 16;
    k.wny = 4;
    k.wwarps = 8;
    k.cheb_w = ei ? k_cheb_w<double, 16, 4, 8, 1, E_P1> : k_cheb_w<double, 16, 4, 8, 1, E_Q1>;
  }
  if (elem == E_Q1 && t.open_w[prec]) {
    k.open_w = open_w_kernel(prec, t.open_w[prec]);
    k.owsx = kOpenSX;
    k.owny = open_w_rows(t.open_w[prec]);
    k.owwarps = kOpenWarps;
    k.o_occ = occupancy(k.open_w, 32 * kOpenWarps, 0);
  }
  if (k.apply_w) k.w_occ = occupancy(k.apply_w, 32 * k.wwarps, k.apply_w_smem);
  for (int b = 0; b < 3; ++b) k.seg_nodes[b] = t.seg_nodes[b];
  const int qpt = t.pw_quads[prec];
  k.pw_chunk = pw_chunk(qpt);
  k.update = update_kernel(prec, qpt);
  return k;
}

// Number of simulations not yet DONE or FAILED.
__global__ void k_count_unfinished(const SimDev* __restrict__ sims, int nsims, int* out) {
  int c = 0;
  for (int i = threadIdx.x; i < nsims; i += blockDim.x) {
    const int ph = *(volatile const int*)&sims[i].sc->phase;
    c += (ph != PH_DONE && ph != PH_FAILED && ph != PH_IDLE) ? 1 : 0;
  }
  for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
  __shared__ int red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) t += red[w];
    *out = t;
  }
}

struct Engine {
  std::vector<heat_sim*> sims;
  int prec = 0;
  Tuning tuning{};  // the table the kernels come from, also when a preconditioner changes
  KernelSet ks{};
  cudaStream_t stream = nullptr;
  SimDev* d_sims = nullptr;
  int2* d_work_op = nullptr;
  int2* d_work_pw = nullptr;
  int2* d_work_aw = nullptr;  // warp-segment apply items
  long long cap_aw = 0;
  int grid_aw = 0;
  std::vector<int2> h_aw;
  int2* d_work_ow = nullptr;  // warp-segment open-pass items
  long long cap_ow = 0;
  int grid_ow = 0;
  std::vector<int2> h_ow;
  // [0] operator tiles, [1] pointwise chunks, [2] warp-apply items, [3] warp open-pass items
  int* d_nwork = nullptr;
  int* d_unfinished = nullptr;  // [2]: the two poll slots of engine_step_all
  int* h_unfinished = nullptr;  // [2], pinned
  cudaEvent_t poll_ev[2] = {nullptr, nullptr};
  double* d_partial = nullptr;
  long long cap_op = 0, cap_pw = 0, cap_partial = 0;
  int grid_op = 0, grid_pw = 0, iters_per_tick = 6;
  int elem = E_Q1;  // the members' finite element (one per engine)
  int ncheb = 0;    // Chebyshev passes per iteration in the tick: max over members of degree - 1
  int grid_ch = 0;  // grid of the pass kernel
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  // persistent iteration (ks.loop): its barrier state and grid
  GridSync* d_sync = nullptr;
  int* h_abort = nullptr;
  int grid_loop = 0;
  long long launches = 0;  // kernels launched by the last engine_step_all
  int* d_phases = nullptr;
  int* h_phases = nullptr;
  int phases_cap = 0;
  std::vector<SimDev> h_sims;
  std::vector<int2> h_op, h_pw;
  // on-chip solve (ks.res): exchange areas, each block's tasks
  unsigned char* d_res = nullptr;
  int* d_res_off = nullptr;
  int2* d_res_tasks = nullptr;
  size_t cap_res = 0;
  long long cap_tasks = 0;
  int grid_res = 0, smem_res = 0;
  bool has_res = false, has_stream = true;  // members on the chip / on the streaming kernels
  std::vector<int> h_res_off;
  std::vector<int2> h_res_tasks;
  long long cap_sims = 0;   // simulations the descriptor array holds
  bool grid_cap = false;    // grids sized by the capacities (members can change without a new graph)
};

// Host-side fault injection for tests of the server's recovery: the next
// g_fail_builds engine builds or membership updates return HEAT_ERR_NOMEM.
static std::atomic<int> g_fail_builds{0};
static bool injected_failure() {
  int n = g_fail_builds.load();
  while (n > 0)
    if (g_fail_builds.compare_exchange_weak(n, n - 1)) return true;
  return false;
}

// Kernels in one tick: k_open, then per iteration the Chebyshev passes and
// apply + update, or the fused kernel; or k_open and the persistent loop.
static int tick_launches(const Engine* e) {
  if (e->ks.loop) return 2;
  return 1 + (e->has_res ? 1 : 0) + (e->has_stream ? (e->ncheb + (e->ks.fused ? 1 : 2)) * e->iters_per_tick : 0);
}

// Rounds (CG iterations) one persistent launch runs at most: a solve's
// inner iterations normally end it first, at a phase change.
constexpr int kLoopRounds = 256;
constexpr int kPollDefault = 32;  // poll_period's default; larger values poll as often
constexpr int kResRounds = 4096;
// In a server's engine, whose members come and go between polls, a launch on the
// chip ends sooner: one long inner solve holds up neither the others' next phase
// nor an admission. 48 iterations carry most inner solves whole (a burst of 8
// mixed requests 35.2 ms with 48, 96 or 4,096, 39 with 24; six small requests
// beside two stiff ones 26.9 ms with 48, 31 with 96 or 4,096).
constexpr int kServeRounds = 48;

// Test hook (heat_debug_loop_wait): arrivals the barrier expects beyond the
// grid, and the bound of one wait in ns (0: the engine's own bound).
static std::atomic<unsigned int> g_loop_extra{0};
static std::atomic<unsigned long long> g_loop_limit_ns{0};

// Barrier state for a fresh launch. One wait is bounded by 1 s plus 50 ns
// per node of the members (a phase of the largest batches takes far less),
// or by the test hook's bound; a launch runs at most `rounds` iterations.
static heat_status loop_sync_reset(Engine* e, int rounds = 0) {
  if (!e->d_sync) return HEAT_OK;
  if (rounds == 0) rounds = e->ks.loop ? kLoopRounds : e->grid_cap ? kServeRounds : kResRounds;
  long long nodes = 0;
  for (const heat_sim* s : e->sims) nodes += s->nn;
  GridSync g{};
  g.extra = g_loop_extra.load();
  const unsigned long long hook = g_loop_limit_ns.load();
  g.limit_ns = hook ? hook : 1000000000ull + 50ull * (unsigned long long)nodes;
  g.rounds = rounds;
  CUDA_TRY(cudaMemcpyAsync(e->d_sync, &g, sizeof(g), cudaMemcpyHostToDevice, e->stream));
  CUDA_TRY(cudaStreamSynchronize(e->stream));
  return HEAT_OK;
}

// After a persistent launch gave up waiting (GridSync::abort): the members'
// iteration state is incomplete, so every member that has not finished
// fails with HEAT_ERR_TIMEOUT, and the barrier state is reset.
static heat_status loop_abort(Engine* e) {
  for (heat_sim* s : e->sims) {
    heat_status st = sim_read_scalars(s);
    if (st != HEAT_OK) return st;
    SimScalars* sc = s->h_sc;
    if (sc->phase != PH_DONE && sc->phase != PH_FAILED && sc->phase != PH_IDLE) {
      sc->status = HEAT_ERR_TIMEOUT;
      sc->phase = PH_FAILED;
    }
    sc->count = 0;
    st = sim_write_scalars(s);
    if (st != HEAT_OK) return st;
  }
  e->h_abort[0] = e->h_abort[1] = 0;
  if (e->d_res) CUDA_TRY(cudaMemsetAsync(e->d_res, 0, e->cap_res, e->stream));  // no tag of the broken launch stays
  return loop_sync_reset(e);
}

// Chebyshev passes the members need per iteration.
static int members_ncheb_of(heat_sim* const* sims, int nsims) {
  int n = 0;
  for (int i = 0; i < nsims; ++i) n = std::max(n, sims[i]->dev.cheb_m >= 2 ? sims[i]->dev.cheb_m - 1 : 0);
  return n;
}
static int members_ncheb(const Engine* e) { return members_ncheb_of(e->sims.data(), (int)e->sims.size()); }

// Operator tile geometry of one simulation: (SX-1) x (SY-1) node columns per
// tile, tz_len levels. tz_len trades z-halo work (3 extra levels per tile)
// against the number of tiles. It depends on the simulation's own mesh only
// (about kTileNodes output nodes per tile, at least 8 levels), so the tiles,
// and with them the order of every reduction, are the same whether the
// simulation runs alone or in a batch: its results are bitwise identical.
constexpr long long kTileNodes = 2048;

// Levels per segment tile for `cols` segment columns of `levels` node levels,
// spc tiles per block, at most hi levels. A block with tz levels takes
// tz + 2.5 level times (halo layers and start); an SM with b blocks takes
// ceil(b / occ) of those, or b * share where one block alone uses that share
// of the SM's throughput (1 where the FP64 pipe bounds the kernel: a second
// block then only waits for the first). The least time^weight * work wins:
// weight 1 for a launch whose time alone counts as much as the work it adds
// to a batch, less where the launch is a part of many batched ones. It
// depends on the mesh and the GPU only, so a simulation's tiles, and with
// them the order of its reductions, are the same alone and in a batch.
static int pick_levels(long long cols, int levels, int spc, int occ, double share, double weight, int hi) {
  const int sms = sm_count();
  double best = 1e300;
  int best_tz = std::min(levels, hi);
  for (int tz = std::min(levels, hi); tz >= 1; --tz) {
    const long long ntz = (levels + tz - 1) / tz, items = (cols * ntz + spc - 1) / spc, b = (items + sms - 1) / sms;
    const double t = (tz + 2.5) * std::max((double)((b + occ - 1) / occ), share * (double)b);
    const double cost = std::pow(t, weight) * (double)ntz * (tz + 2.5);
    if (cost < best * (1.0 - 1e-9)) {
      best = cost;
      best_tz = tz;
    }
  }
  return best_tz;
}

static void tile_geometry(SimDev& d, const KernelSet& ks, bool fp64) {
  d.res = res_plan(d, ks, fp64);
  d.ntx = (d.nx + 1 + ks.sx - 2) / (ks.sx - 1);
  d.nty = (d.ny + 1 + ks.sy - 2) / (ks.sy - 1);
  const int levels = d.nz + 1;
  const long long cols = (long long)d.ntx * d.nty;
  const long long want = std::max(1LL, d.nn / kTileNodes);
  int ntz = (int)std::max(1LL, std::min<long long>(levels, (want + cols - 1) / cols));
  ntz = std::min(ntz, std::max(1, levels / 8));
  d.tz_len = (levels + ntz - 1) / ntz;
  d.ntz = (levels + d.tz_len - 1) / d.tz_len;
  d.ntiles = d.ntx * d.nty * d.ntz;
  d.npw = (int)((d.nn + ks.pw_chunk - 1) / ks.pw_chunk);
  d.w_ntx = d.w_nty = d.w_ntz = d.w_tz = d.w_ntiles = d.w_items = 0;
  if (ks.apply_w) {
    // segment tiles of about seg output nodes, at least 4 levels (2 extra levels
    // per tile); under the default variants the default size stands for the
    // estimated best
    const int seg = ks.seg_nodes[size_bucket(d.nn)];
    // the narrower padded row; equal: whole lines
    const int pad16 = (d.nx + 1 + 13) / 14 * 14, pad32 = (d.nx + 1 + 29) / 30 * 30;
    d.w_sx = ks.dual && d.cheb_m < 2 ? (pad32 <= pad16 ? 32 : 16) : ks.wsx;
    d.w_ntx = (d.nx + 1 + d.w_sx - 3) / (d.w_sx - 2);
    d.w_nty = (d.ny + 1 + ks.wny - 1) / ks.wny;
    const int spc = ks.wwarps * (32 / d.w_sx);
    const int tz0 = ks.auto_seg && seg == kAutoSeg && ks.w_occ > 0
                        ? pick_levels((long long)d.w_ntx * d.w_nty, levels, spc, ks.w_occ, fp64 ? 1.0 : 0.34, 4.0, 96)
                        : std::max(4, std::min(levels, seg / ((d.w_sx - 2) * ks.wny)));
    d.w_ntz = (levels + tz0 - 1) / tz0;
    d.w_tz = (levels + d.w_ntz - 1) / d.w_ntz;
    d.w_ntiles = d.w_ntx * d.w_nty * d.w_ntz;
    d.w_items = (d.w_ntiles + spc - 1) / spc;
  }
  d.o_ntx = d.o_nty = d.o_ntz = d.o_tz = d.o_ntiles = d.o_items = 0;
  if (ks.open_w) {
    d.o_ntx = (d.nx + 1 + ks.owsx - 3) / (ks.owsx - 2);
    d.o_nty = (d.ny + 1 + ks.owny - 1) / ks.owny;
    const int spc = ks.owwarps * (32 / ks.owsx);
    // at most about 1,024 output nodes per segment tile
    const int hi = std::max(4, 1024 / ((ks.owsx - 2) * ks.owny));
    const int tz0 = ks.o_occ > 0 ? pick_levels((long long)d.o_ntx * d.o_nty, levels, spc, ks.o_occ, fp64 ? 1.0 : 0.34,
                                                 fp64 ? 1.0 : 0.25, hi)
                                 : std::min(levels, hi);
    d.o_ntz = (levels + tz0 - 1) / tz0;
    d.o_tz = (levels + d.o_ntz - 1) / d.o_ntz;
    d.o_ntiles = d.o_ntx * d.o_nty * d.o_ntz;
    d.o_items = (d.o_ntiles + spc - 1) / spc;
  }
}

static int sm_count() {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Deals the members on the chip to the blocks of k_cg_res. Every block runs
// its tasks in member order, so the first unfinished member's blocks are all
// at it and the launch always advances. Each member takes the blocks that
// are free first.
static heat_status res_schedule(Engine* e, bool has_res, bool has_stream, size_t res_used) {
  e->has_res = has_res;
  e->has_stream = has_stream;
  e->grid_res = e->smem_res = 0;
  if (!has_res) return HEAT_OK;
  const int nb = e->ks.res_blocks;
  const bool f64 = e->prec == P_FP64;
  std::vector<std::vector<int2>> list(nb);
  std::vector<double> load(nb, 0.0);
  std::vector<int> order(nb);
  int used = 0;
  long long ntasks = 0;
  for (size_t i = 0; i < e->h_sims.size(); ++i) {
    const ResGeo& r = e->h_sims[i].res;
    if (r.g == 0) continue;
    for (int b = 0; b < nb; ++b) order[b] = b;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return load[a] < load[b]; });
    const double end = load[order[r.g - 1]] + res_cycles(r, f64);
    for (int k = 0; k < r.g; ++k) {
      list[order[k]].push_back(make_int2((int)i, k));
      load[order[k]] = end;
      used = std::max(used, order[k] + 1);
    }
    ntasks += r.g;
    e->smem_res = std::max(e->smem_res, res_layout(r, f64).bytes);
  }
  if (ntasks > e->cap_tasks) return set_error(HEAT_ERR_ARG, "engine: on-chip tasks exceed their capacity");
  e->grid_res = e->grid_cap ? nb : used;
  if (e->grid_cap) e->smem_res = e->ks.res_smem;
  e->h_res_off.assign(1, 0);
  e->h_res_tasks.clear();
  for (int b = 0; b < nb; ++b) {
    e->h_res_tasks.insert(e->h_res_tasks.end(), list[b].begin(), list[b].end());
    e->h_res_off.push_back((int)e->h_res_tasks.size());
  }
  CUDA_TRY(cudaMemcpyAsync(e->d_res_off, e->h_res_off.data(), sizeof(int) * e->h_res_off.size(), cudaMemcpyHostToDevice,
                           e->stream));
  CUDA_TRY(cudaMemcpyAsync(e->d_res_tasks, e->h_res_tasks.data(), sizeof(int2) * e->h_res_tasks.size(),
                           cudaMemcpyHostToDevice, e->stream));
  CUDA_TRY(cudaMemsetAsync(e->d_res, 0, res_used, e->stream));  // tags start anew with the areas
  return HEAT_OK;
}

static heat_status engine_upload(Engine* e) {
  e->h_sims.clear();
  e->h_op.clear();
  e->h_pw.clear();
  e->h_aw.clear();
  e->h_ow.clear();
  const int sms = sm_count();
  long long item_base = 0;
  size_t res_base = 0;
  const bool f64 = e->prec == P_FP64;
  bool has_res = false, has_stream = false;
  for (size_t i = 0; i < e->sims.size(); ++i) {
    SimDev d = e->sims[i]->dev;
    tile_geometry(d, e->ks, e->prec == P_FP64);
    d.fused = e->ks.fused ? 1 : 0;
    d.partial = e->d_partial + 4 * item_base;
    item_base += std::max(std::max(std::max(d.ntiles, d.npw), d.w_items), d.o_items);
    const bool stream = d.res.g == 0;
    // the block tiles also carry k_open's passes
    if (stream || !e->ks.open_w)
      for (int t = 0; t < d.ntiles; ++t) e->h_op.push_back(make_int2((int)i, t));
    if (stream) {
      for (int t = 0; t < d.npw; ++t) e->h_pw.push_back(make_int2((int)i, t));
      for (int t = 0; t < d.w_items; ++t) e->h_aw.push_back(make_int2((int)i, t));
    }
    for (int t = 0; t < d.o_items; ++t) e->h_ow.push_back(make_int2((int)i, t));
    (stream ? has_stream : has_res) = true;
    if (!stream) {
      const ResBytes rb = res_bytes(d, f64);
      if (res_base + rb.total > e->cap_res) return set_error(HEAT_ERR_ARG, "engine: exchange areas exceed their capacity");
      unsigned char* p = e->d_res + res_base;
      d.res_z = p + rb.z;
      d.res_x = p + rb.x;
      d.res_slots = (ulonglong2*)(p + rb.slots);
      d.res_tag = (unsigned int*)(p + rb.tag);
      res_base += rb.total;
    }
    e->h_sims.push_back(d);
  }
  if ((long long)e->h_op.size() > e->cap_op || (long long)e->h_pw.size() > e->cap_pw ||
      (long long)e->h_aw.size() > e->cap_aw || (long long)e->h_ow.size() > e->cap_ow ||
      item_base > e->cap_partial)
    return set_error(HEAT_ERR_ARG, "engine: work lists exceed their capacity");
  heat_status rst = res_schedule(e, has_res, has_stream, res_base);
  if (rst != HEAT_OK) return rst;
  const int nwork[4] = {(int)e->h_op.size(), (int)e->h_pw.size(), (int)e->h_aw.size(), (int)e->h_ow.size()};
  CUDA_TRY(cudaMemcpyAsync(e->d_sims, e->h_sims.data(), sizeof(SimDev) * e->h_sims.size(), cudaMemcpyHostToDevice,
                           e->stream));
  if (!e->h_op.empty())
    CUDA_TRY(cudaMemcpyAsync(e->d_work_op, e->h_op.data(), sizeof(int2) * e->h_op.size(), cudaMemcpyHostToDevice,
                             e->stream));
  if (!e->h_pw.empty())
    CUDA_TRY(cudaMemcpyAsync(e->d_work_pw, e->h_pw.data(), sizeof(int2) * e->h_pw.size(), cudaMemcpyHostToDevice,
                             e->stream));
  if (!e->h_aw.empty())
    CUDA_TRY(cudaMemcpyAsync(e->d_work_aw, e->h_aw.data(), sizeof(int2) * e->h_aw.size(), cudaMemcpyHostToDevice,
                             e->stream));
  if (!e->h_ow.empty())
    CUDA_TRY(cudaMemcpyAsync(e->d_work_ow, e->h_ow.data(), sizeof(int2) * e->h_ow.size(), cudaMemcpyHostToDevice,
                             e->stream));
  CUDA_TRY(cudaMemcpyAsync(e->d_nwork, nwork, sizeof(nwork), cudaMemcpyHostToDevice, e->stream));
  CUDA_TRY(cudaStreamSynchronize(e->stream));
  int occ_op = 1, occ_pw = 1, occ_aw = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_op, e->ks.apply ? e->ks.apply : e->ks.open, e->ks.apply_threads, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_pw, e->ks.update, kPwThreads, 0);
  if (e->ks.apply_w)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_aw, e->ks.apply_w, 32 * e->ks.wwarps, e->ks.apply_w_smem);
  int occ_ch = 1;
  if (e->ks.cheb_w)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_ch, e->ks.cheb_w, 32 * e->ks.wwarps, 0);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_ch, e->ks.cheb, e->ks.apply_threads, 0);
  int occ_ow = 1;
  if (e->ks.open_w)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_ow, e->ks.open_w, 32 * e->ks.owwarps, 0);
  if (e->ks.loop) {
    // every block resident at once (the launch is cooperative)
    int occ_loop = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_loop, (const void*)e->ks.loop, 32 * e->ks.wwarps, 0);
    if (occ_loop < 1) return set_error(HEAT_ERR_CUDA, "engine: the persistent iteration kernel does not fit an SM");
    e->grid_loop = sms * occ_loop;
  }
  // With grid_cap the grids cover the capacities, so a later member set that
  // fits them runs under the same captured graph (surplus blocks find no item).
  const long long items[4] = {e->grid_cap ? e->cap_op : nwork[0], e->grid_cap ? e->cap_pw : nwork[1],
                              e->grid_cap ? e->cap_aw : nwork[2], e->grid_cap ? e->cap_ow : nwork[3]};
  e->grid_ow = (int)std::max(1LL, std::min<long long>(items[3], (long long)sms * std::max(1, occ_ow)));
  e->grid_op = (int)std::max(1LL, std::min<long long>(items[0], (long long)sms * std::max(1, occ_op)));
  e->grid_pw = (int)std::max(1LL, std::min<long long>(items[1], (long long)sms * std::max(1, occ_pw)));
  e->grid_aw = (int)std::max(1LL, std::min<long long>(items[2], (long long)sms * std::max(1, occ_aw)));
  e->grid_ch = (int)std::max(1LL, std::min<long long>(e->ks.cheb_w ? items[2] : items[0],
                                                      (long long)sms * std::max(1, occ_ch)));
  return HEAT_OK;
}

// The apply kernel of an iteration and its launch shape / work list.
static void apply_launch(const Engine* e, TileFn* fn, int* grid, int* threads, const int2** work,
                         const int** nwork, int* smem) {
  *smem = 0;
  if (e->ks.apply_w) {
    *smem = e->ks.apply_w_smem;
    *fn = e->ks.apply_w;
    *grid = e->grid_aw;
    *threads = 32 * e->ks.wwarps;
    *work = e->d_work_aw;
    *nwork = e->d_nwork + 2;
  } else {
    *fn = e->ks.apply;
    *grid = e->grid_op;
    *threads = e->ks.apply_threads;
    *work = e->d_work_op;
    *nwork = e->d_nwork;
  }
}

// One launch of the on-chip solve: cooperative, all blocks resident.
static cudaError_t res_launch(Engine* e, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(e->grid_res);
  cfg.blockDim = dim3(kResThreads);
  cfg.dynamicSmemBytes = (size_t)e->smem_res;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, e->ks.res, (const SimDev*)e->d_sims, (const int*)e->d_res_off,
                            (const int2*)e->d_res_tasks, e->d_sync);
}

static heat_status engine_capture(Engine* e) {
  if (e->gexec) {
    cudaGraphExecDestroy(e->gexec);
    e->gexec = nullptr;
  }
  if (e->graph) {
    cudaGraphDestroy(e->graph);
    e->graph = nullptr;
  }
  // Capture on a private stream (the legacy default stream cannot capture);
  // the instantiated graph is then launched on the engine's stream.
  cudaStream_t cap;
  CUDA_TRY(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
  // Each kernel may launch while its predecessor finishes (programmatic
  // dependent launch); the kernels wait for the predecessor's results with
  // cudaGridDependencySynchronize after their static prologue.
  auto launch = [&](TileFn fn, int grid, int block, const int2* work, const int* nwork, int smem) -> cudaError_t {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = cap;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, (const SimDev*)e->d_sims, work, nwork);
  };
  TileFn afn;
  int agrid, athreads, asmem;
  const int2* awork;
  const int* anwork;
  apply_launch(e, &afn, &agrid, &athreads, &awork, &anwork, &asmem);
  cudaError_t err = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
  if (err == cudaSuccess) {
    cudaError_t lerr = e->ks.open_w
                           ? launch(e->ks.open_w, e->grid_ow, 32 * e->ks.owwarps, e->d_work_ow, e->d_nwork + 3, 0)
                           : launch(e->ks.open, e->grid_op, e->ks.open_threads, e->d_work_op, e->d_nwork, 0);
    if (e->ks.loop && lerr == cudaSuccess) {
      // one persistent launch for the tick's iterations: cooperative (all
      // blocks resident, which its grid barriers need), no early start
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(e->grid_loop);
      cfg.blockDim = dim3(32 * e->ks.wwarps);
      cfg.dynamicSmemBytes = 0;
      cfg.stream = cap;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeCooperative;
      attr[0].val.cooperative = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      lerr = cudaLaunchKernelEx(&cfg, e->ks.loop, (const SimDev*)e->d_sims, (const int2*)e->d_work_aw,
                                (const int2*)e->d_work_pw, (const int*)e->d_nwork, e->d_sync);
    }
    if (e->has_res && lerr == cudaSuccess) lerr = res_launch(e, cap);
    for (int it = 0; it < (e->ks.loop || !e->has_stream ? 0 : e->iters_per_tick) && lerr == cudaSuccess; ++it) {
      for (int k = 0; k < e->ncheb && lerr == cudaSuccess; ++k) {
        if (e->ks.cheb_w) lerr = launch(e->ks.cheb_w, e->grid_ch, 32 * e->ks.wwarps, e->d_work_aw, e->d_nwork + 2, 0);
        else lerr = launch(e->ks.cheb, e->grid_ch, e->ks.apply_threads, e->d_work_op, e->d_nwork, 0);
      }
      if (lerr != cudaSuccess) break;
      lerr = launch(afn, agrid, athreads, awork, anwork, asmem);
      if (lerr == cudaSuccess && !e->ks.fused)
        lerr = launch(e->ks.update, e->grid_pw, kPwThreads, e->d_work_pw, e->d_nwork + 1, 0);
    }
    err = cudaStreamEndCapture(cap, &e->graph);
    if (err == cudaSuccess && lerr != cudaSuccess) err = lerr;
  }
  cudaStreamDestroy(cap);
  if (err != cudaSuccess) {
    cudaGetLastError();
    return set_error(HEAT_ERR_CUDA, "graph capture failed: %s", cudaGetErrorString(err));
  }
  CUDA_TRY(cudaGraphInstantiate(&e->gexec, e->graph, 0));
  return HEAT_OK;
}

heat_status engine_create(heat_sim* const* sims, int nsims, int precision, cudaStream_t stream, Engine** out,
                          const Tuning* tun, double headroom) {
  *out = nullptr;
  if (nsims < 1 || !sims) return set_error(HEAT_ERR_ARG, "engine: no simulations");
  if (injected_failure()) return set_error(HEAT_ERR_NOMEM, "engine: build failure injected by the test hook");
  if (!(headroom >= 1.0) || headroom > 64.0) return set_error(HEAT_ERR_ARG, "engine: headroom must be in [1, 64]");
  Engine* e = new Engine();
  e->sims.assign(sims, sims + nsims);
  e->prec = precision;
  e->elem = sims[0]->dev.elem;
  for (int i = 1; i < nsims; ++i)
    if (sims[i]->dev.elem != e->elem) {
      delete e;
      return set_error(HEAT_ERR_ARG, "engine: the simulations of one batch must share the element type");
    }
  e->ncheb = members_ncheb(e);
  e->tuning = tun ? *tun : tuning_get();
  e->stream = stream;
  // Capacities: the geometry is a function of each mesh and of whether the
  // member takes Chebyshev passes (they run on 16-lane segments where the plain
  // apply may take 32-lane ones or the chip), and a member may change that at
  // any time: each list holds the larger of the two forms.
  long long cap_op = 0, cap_pw = 0, cap_aw = 0, cap_ow = 0, cap_partial = 0, cap_tasks = 0;
  size_t cap_res = 0;
  const KernelSet sets[2] = {kernel_set(precision, e->tuning, false, e->elem),
                             kernel_set(precision, e->tuning, true, e->elem)};
  e->ks = sets[e->ncheb > 0 ? 1 : 0];
  const bool one_set = sets[0].apply_w == sets[1].apply_w && sets[0].dual == sets[1].dual && sets[0].res == sets[1].res;
  struct Need {
    int nx = 0, ny = 0, nz = 0;
    long long op = 0, pw = 0, aw = 0, ow = 0, tasks = 0;
    size_t res = 0;
  } n;
  for (heat_sim* s : e->sims) {
    if (n.nx != s->dev.nx || n.ny != s->dev.ny || n.nz != s->dev.nz) {  // members of one size need the same
      n = Need{s->dev.nx, s->dev.ny, s->dev.nz};
      for (int k = 0; k < (one_set ? 1 : 2); ++k)
        for (int cheb_m : {0, 2}) {
          SimDev d = s->dev;
          d.cheb_m = cheb_m;
          tile_geometry(d, sets[k], precision == P_FP64);
          n.op = std::max<long long>(n.op, d.ntiles);
          n.pw = std::max<long long>(n.pw, d.npw);
          n.aw = std::max<long long>(n.aw, d.w_items);
          n.ow = std::max<long long>(n.ow, d.o_items);
          n.res = std::max(n.res, res_bytes(d, precision == P_FP64).total);
          n.tasks = std::max<long long>(n.tasks, d.res.g);
        }
    }
    cap_op += n.op;
    cap_pw += n.pw;
    cap_aw += n.aw;
    cap_ow += n.ow;
    cap_partial += std::max(std::max(n.op, n.pw), std::max(n.aw, n.ow));
    cap_res += n.res;
    cap_tasks += n.tasks;
  }
  if (cap_op > (1LL << 30) || cap_pw > (1LL << 30) || cap_aw > (1LL << 30) || cap_ow > (1LL << 30)) {
    delete e;
    return set_error(HEAT_ERR_ARG, "engine: too many work items");
  }
  auto grow = [&](long long c) { return (long long)std::ceil((double)c * headroom); };
  e->cap_sims = grow(nsims);
  e->grid_cap = headroom > 1.0;
  cap_op = grow(cap_op);
  cap_pw = grow(cap_pw);
  cap_aw = grow(cap_aw);
  cap_ow = grow(cap_ow);
  cap_partial = grow(cap_partial);
  e->cap_op = cap_op;
  e->cap_pw = cap_pw;
  e->cap_aw = cap_aw;
  e->cap_ow = cap_ow;
  e->cap_partial = cap_partial;
  e->cap_res = (size_t)grow((long long)cap_res);
  e->cap_tasks = grow(cap_tasks);
  heat_status st = HEAT_OK;
  auto fail = [&](heat_status s) {
    engine_destroy(e);
    return s;
  };
  if (cudaMalloc(&e->d_sims, sizeof(SimDev) * e->cap_sims) != cudaSuccess ||
      cudaMalloc(&e->d_work_op, sizeof(int2) * cap_op) != cudaSuccess ||
      cudaMalloc(&e->d_work_pw, sizeof(int2) * cap_pw) != cudaSuccess ||
      cudaMalloc(&e->d_work_aw, sizeof(int2) * std::max(1LL, cap_aw)) != cudaSuccess ||
      cudaMalloc(&e->d_work_ow, sizeof(int2) * std::max(1LL, cap_ow)) != cudaSuccess ||
      cudaMalloc(&e->d_nwork, sizeof(int) * 4) != cudaSuccess ||
      cudaMalloc(&e->d_unfinished, 2 * sizeof(int)) != cudaSuccess ||
      cudaMalloc(&e->d_partial, sizeof(double) * 4 * cap_partial) != cudaSuccess ||
      cudaMallocHost(&e->h_unfinished, 2 * sizeof(int)) != cudaSuccess ||
      cudaMalloc(&e->d_sync, sizeof(GridSync)) != cudaSuccess ||
      cudaMallocHost(&e->h_abort, 2 * sizeof(int)) != cudaSuccess ||
      (e->cap_res > 0 && (cudaMalloc(&e->d_res, e->cap_res) != cudaSuccess ||
                          cudaMalloc(&e->d_res_off, sizeof(int) * (e->ks.res_blocks + 1)) != cudaSuccess ||
                          cudaMalloc(&e->d_res_tasks, sizeof(int2) * e->cap_tasks) != cudaSuccess)) ||
      cudaEventCreateWithFlags(&e->poll_ev[0], cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&e->poll_ev[1], cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    return fail(set_error(HEAT_ERR_NOMEM, "engine: device allocation failed"));
  }
  // the per-sim counters used by the last-block reductions start at zero
  for (heat_sim* s : e->sims) {
    st = sim_read_scalars(s);
    if (st != HEAT_OK) return fail(st);
    s->h_sc->count = 0;
    st = sim_write_scalars(s);
    if (st != HEAT_OK) return fail(st);
  }
  st = engine_upload(e);
  if (st != HEAT_OK) return fail(st);
  e->h_abort[0] = e->h_abort[1] = 0;
  st = loop_sync_reset(e);
  if (st != HEAT_OK) return fail(st);
  st = engine_capture(e);
  if (st != HEAT_OK) return fail(st);
  *out = e;
  return HEAT_OK;
}

void engine_destroy(Engine* e) {
  if (!e) return;
  cudaStreamSynchronize(e->stream);
  if (e->gexec) cudaGraphExecDestroy(e->gexec);
  if (e->graph) cudaGraphDestroy(e->graph);
  cudaFree(e->d_sims);
  cudaFree(e->d_work_op);
  cudaFree(e->d_work_pw);
  cudaFree(e->d_work_aw);
  cudaFree(e->d_work_ow);
  cudaFree(e->d_nwork);
  cudaFree(e->d_unfinished);
  cudaFree(e->d_partial);
  if (e->d_sync) cudaFree(e->d_sync);
  if (e->d_res) cudaFree(e->d_res);
  if (e->d_res_off) cudaFree(e->d_res_off);
  if (e->d_res_tasks) cudaFree(e->d_res_tasks);
  if (e->h_abort) cudaFreeHost(e->h_abort);
  if (e->h_unfinished) cudaFreeHost(e->h_unfinished);
  for (cudaEvent_t ev : e->poll_ev)
    if (ev) cudaEventDestroy(ev);
  if (e->d_phases) cudaFree(e->d_phases);
  if (e->h_phases) cudaFreeHost(e->h_phases);
  delete e;
}

heat_status engine_refresh(Engine* e) {
  const int g_op = e->grid_op, g_pw = e->grid_pw, g_aw = e->grid_aw, g_ch = e->grid_ch, g_ow = e->grid_ow;
  const int g_res = e->grid_res, sm_res = e->smem_res;
  const bool h_res = e->has_res, h_stream = e->has_stream;
  // a member's preconditioner may have changed: the passes per iteration, and
  // with them the kernel set (no fused iteration with passes) and the graph
  const int nch = members_ncheb(e);
  const bool recapture = nch != e->ncheb;
  for (const heat_sim* s : e->sims)
    if (s->dev.elem != e->elem) return set_error(HEAT_ERR_ARG, "engine: a member changed its element type");
  if ((nch > 0) != (e->ncheb > 0)) e->ks = kernel_set(e->prec, e->tuning, nch > 0, e->elem);
  e->ncheb = nch;
  heat_status st = engine_upload(e);
  if (st == HEAT_OK) st = loop_sync_reset(e);
  if (st != HEAT_OK) {  // the graph is no longer that of the members: captured anew by the next refresh
    if (e->gexec) cudaGraphExecDestroy(e->gexec);
    e->gexec = nullptr;
    return st;
  }
  if (recapture || !e->gexec || e->grid_op != g_op || e->grid_pw != g_pw || e->grid_aw != g_aw || e->grid_ch != g_ch ||
      e->grid_ow != g_ow || e->has_res != h_res || e->has_stream != h_stream || e->grid_res != g_res ||
      e->smem_res != sm_res)
    return engine_capture(e);
  return HEAT_OK;
}

heat_status engine_set_members(Engine* e, heat_sim* const* sims, int nsims) {
  if (injected_failure()) return set_error(HEAT_ERR_NOMEM, "engine: update failure injected by the test hook");
  if (nsims < 1 || !sims || nsims > e->cap_sims) return set_error(HEAT_ERR_ARG, "engine: member set exceeds capacity");
  long long op = 0, pw = 0, aw = 0, ow = 0, part = 0, tasks = 0;
  size_t res = 0;
  for (int i = 0; i < nsims; ++i) {
    const heat_sim* s = sims[i];
    if (s->prm.precision != e->prec || s->dev.elem != e->elem)
      return set_error(HEAT_ERR_ARG, "engine: a member's precision or element differs from the engine's");
    SimDev d = s->dev;
    tile_geometry(d, e->ks, e->prec == P_FP64);
    op += d.ntiles;
    pw += d.npw;
    aw += d.w_items;
    ow += d.o_items;
    part += std::max(std::max(std::max(d.ntiles, d.npw), d.w_items), d.o_items);
    res += res_bytes(d, e->prec == P_FP64).total;
    tasks += d.res.g;
  }
  if (op > e->cap_op || pw > e->cap_pw || aw > e->cap_aw || ow > e->cap_ow || part > e->cap_partial ||
      res > e->cap_res || tasks > e->cap_tasks)
    return set_error(HEAT_ERR_ARG, "engine: member set exceeds the work-list capacity");
  // the last-block counters of newly added members start at zero
  for (int i = 0; i < nsims; ++i) {
    heat_sim* s = sims[i];
    if (std::find(e->sims.begin(), e->sims.end(), s) != e->sims.end()) continue;
    heat_status st = sim_read_scalars(s);
    if (st != HEAT_OK) return st;
    s->h_sc->count = 0;
    st = sim_write_scalars(s);
    if (st != HEAT_OK) return st;
  }
  e->sims.assign(sims, sims + nsims);
  return engine_refresh(e);
}

__global__ void k_begin_steps(const SimDev* __restrict__ sims, int nsims, int nsteps, int reset_counters) {
  for (int i = threadIdx.x; i < nsims; i += blockDim.x) {
    SimScalars* sc = sims[i].sc;
    sc->target = sc->step + nsteps;
    sc->phase = PH_OPEN;
    sc->status = ST_OK;
    sc->count = 0;
    if (reset_counters) {
      sc->iters_total = 0;
      sc->outer_total = 0;
      sc->steps_total = 0;
      sc->max_iters_step = 0;
    }
  }
}

heat_status engine_step_all(Engine* e, int nsteps, heat_step_stats* stats, int reset_counters) {
  int max_iter = 1, max_outer = 1, poll = kPollDefault;
  const bool waits = e->ks.loop || e->has_res;  // kernels whose bounded waits can give up
  for (const heat_sim* s : e->sims) {
    max_iter = std::max(max_iter, s->prm.max_iter);
    max_outer = std::max(max_outer, s->prm.max_outer);
    poll = std::min(poll, s->prm.poll_period);
  }
  // Iterations and ticks between two polls. Streaming: poll_period iterations.
  // On the chip a launch carries a whole inner solve, and three ticks are a step
  // of the refined path; below the default poll_period a launch ends after that
  // many iterations and is polled after.
  const bool chip = e->has_res && !e->has_stream;
  const int rounds = !e->has_res || poll >= kPollDefault ? 0 : chip ? std::max(poll, e->iters_per_tick) : e->iters_per_tick;
  const int ticks_per_poll = !chip ? std::max(1, poll / e->iters_per_tick) : poll >= kPollDefault ? 3 : 1;
  if (waits) {  // the bound and the test hook as they are now
    heat_status st = loop_sync_reset(e, rounds);
    if (st != HEAT_OK) return st;
  }
  // the members' scalars are set on the device, all in one launch, after what
  // their own streams still hold (64 members: 1.8 ms of copies and waits when
  // each was read, changed and written from the host)
  for (size_t i = 0; i < e->sims.size(); ++i) {
    const cudaStream_t own = e->sims[i]->stream;
    if (own != e->stream && (i == 0 || own != e->sims[i - 1]->stream)) CUDA_TRY(cudaStreamSynchronize(own));
  }
  k_begin_steps<<<1, 256, 0, e->stream>>>(e->d_sims, (int)e->sims.size(), nsteps, reset_counters);
  CUDA_TRY(cudaGetLastError());
  // Every tick advances each unfinished simulation by at least one CG
  // iteration or one phase change, so this bound is never reached by a
  // healthy solve; it turns a logic error into HEAT_ERR_TIMEOUT.
  const long long max_ticks = (long long)nsteps * (max_iter + 2LL * max_outer + 4) + 64;
  long long ticks = 0;
  e->launches = 0;
  // Batch b of ticks_per_poll ticks ends with a count of the unfinished
  // members (and the persistent loop's abort flag) copied to slot b & 1 and
  // an event. The first batch is waited for at once (a short call leaves no
  // idle ticks behind); from then on batch b is queued before the host waits
  // for batch b - 1, so the GPU does not idle while the host polls. At most
  // one batch of idle ticks runs after the last member finishes.
  for (long long b = 0;; ++b) {
    const int slot = (int)(b & 1);
    for (int t = 0; t < ticks_per_poll; ++t) CUDA_TRY(cudaGraphLaunch(e->gexec, e->stream));
    ticks += ticks_per_poll;
    e->launches += (long long)ticks_per_poll * tick_launches(e) + 1;
    k_count_unfinished<<<1, 256, 0, e->stream>>>(e->d_sims, (int)e->sims.size(), e->d_unfinished + slot);
    CUDA_TRY(cudaGetLastError());
    CUDA_TRY(cudaMemcpyAsync(e->h_unfinished + slot, e->d_unfinished + slot, sizeof(int), cudaMemcpyDeviceToHost,
                             e->stream));
    if (waits)
      CUDA_TRY(cudaMemcpyAsync(e->h_abort + slot, &e->d_sync->abort, sizeof(int), cudaMemcpyDeviceToHost, e->stream));
    CUDA_TRY(cudaEventRecord(e->poll_ev[slot], e->stream));
    long long waited = -1;  // the batch whose counts are read now
    if (b == 0) waited = 0;
    else if (b >= 2) waited = b - 1;
    if (waited < 0) continue;  // batch 1 queued right after batch 0 was read
    const int ws = (int)(waited & 1);
    CUDA_TRY(cudaEventSynchronize(e->poll_ev[ws]));
    if (waits && e->h_abort[ws]) {
      CUDA_TRY(cudaStreamSynchronize(e->stream));
      heat_status st = loop_abort(e);
      if (st != HEAT_OK) return st;
      break;
    }
    if (e->h_unfinished[ws] == 0) break;
    if (ticks > max_ticks) {
      cudaStreamSynchronize(e->stream);
      return set_error(HEAT_ERR_TIMEOUT, "engine: solve did not finish within %lld ticks", ticks);
    }
  }
  heat_status first_bad = HEAT_OK;
  for (size_t i = 0; i < e->sims.size(); ++i) {
    heat_sim* s = e->sims[i];
    CUDA_TRY(cudaMemcpyAsync(s->h_sc, s->d_sc, sizeof(SimScalars), cudaMemcpyDeviceToHost, e->stream));
  }
  CUDA_TRY(cudaStreamSynchronize(e->stream));
  for (size_t i = 0; i < e->sims.size(); ++i) {
    const SimScalars* sc = e->sims[i]->h_sc;
    if (stats) {
      heat_step_stats& o = stats[i];
      o.steps = (int)sc->steps_total;
      o.status = sc->phase == PH_FAILED ? sc->status : HEAT_OK;
      o.iters = sc->iters_total;
      o.outer = sc->outer_total;
      o.max_iters_step = sc->max_iters_step;
      o.last_rel_residual = sc->rel_res;
      o.kernel_launches = e->launches;
    }
    if (sc->phase == PH_FAILED && first_bad == HEAT_OK) {
      first_bad = (heat_status)sc->status;
      set_error(first_bad, "simulation %zu failed at step %d: %s", i, sc->step + 1,
                heat_status_string((heat_status)sc->status));
    }
  }
  return first_bad;
}

__global__ void k_gather_phases(const SimDev* __restrict__ sims, int nsims, int* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nsims; i += gridDim.x * blockDim.x)
    out[i] = *(volatile const int*)&sims[i].sc->phase;
}

heat_status engine_launch_ticks(Engine* e, int nticks) {
  for (int t = 0; t < nticks; ++t) CUDA_TRY(cudaGraphLaunch(e->gexec, e->stream));
  e->launches += (long long)nticks * tick_launches(e);
  return HEAT_OK;
}

heat_status engine_read_phases(Engine* e, int* phases) {
  const int n = (int)e->sims.size();
  int* d = nullptr;
  if (!e->d_phases || e->phases_cap < n) {  // grown on first use
    if (e->d_phases) cudaFree(e->d_phases);
    if (e->h_phases) cudaFreeHost(e->h_phases);
    e->d_phases = nullptr;
    e->h_phases = nullptr;
    CUDA_TRY(cudaMalloc(&e->d_phases, sizeof(int) * n));
    CUDA_TRY(cudaMallocHost(&e->h_phases, sizeof(int) * n));
    e->phases_cap = n;
  }
  d = e->d_phases;
  if (e->ks.loop || e->has_res) {  // a persistent launch that gave up fails the unfinished members first
    CUDA_TRY(cudaMemcpyAsync(e->h_abort, &e->d_sync->abort, sizeof(int), cudaMemcpyDeviceToHost, e->stream));
    CUDA_TRY(cudaStreamSynchronize(e->stream));
    if (*e->h_abort) {
      heat_status st = loop_abort(e);
      if (st != HEAT_OK) return st;
    }
  }
  k_gather_phases<<<(n + 255) / 256, 256, 0, e->stream>>>(e->d_sims, n, d);
  CUDA_TRY(cudaGetLastError());
  e->launches += 1;
  CUDA_TRY(cudaMemcpyAsync(e->h_phases, d, sizeof(int) * n, cudaMemcpyDeviceToHost, e->stream));
  CUDA_TRY(cudaStreamSynchronize(e->stream));
  std::memcpy(phases, e->h_phases, sizeof(int) * n);
  return HEAT_OK;
}

bool engine_on_chip(const Engine* e) { return e->has_res; }

long long engine_launches(const Engine* e) { return e->launches; }

size_t engine_footprint(long long nn, long long nx, long long ny, long long nz) {
  // the largest work lists any precision's kernels need under the current table
  const Tuning t = tuning_get();
  long long op = 0, pw = 0, aw = 0, ow = 0;
  size_t res = 0;
  for (int p = 0; p < 3; ++p) {
    SimDev d{};
    d.nx = (int)nx;
    d.ny = (int)ny;
    d.nz = (int)nz;
    d.nn = nn;
    tile_geometry(d, kernel_set(p, t), p == P_FP64);
    res = std::max(res, res_bytes(d, p == P_FP64).total + sizeof(int2) * d.res.g);
    op = std::max<long long>(op, d.ntiles);
    pw = std::max<long long>(pw, d.npw);
    aw = std::max<long long>(aw, d.w_items);
    ow = std::max<long long>(ow, d.o_items);
  }
  return res + (size_t)(sizeof(int2) * (op + pw + aw + ow) +
                  sizeof(double) * 4 * std::max(std::max(std::max(op, pw), aw), ow) + sizeof(SimDev) + 64);
}

// Reads a buffer larger than L2 so the next kernel starts cold. Reading (not
// writing) leaves clean lines, so no write-back lands in the timed kernel.
__global__ void k_flush_read(const uint4* __restrict__ p, size_t n, unsigned int* sink) {
  unsigned int acc = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const uint4 v = __ldcg(p + i);
    acc ^= v.x ^ v.y ^ v.z ^ v.w;
  }
  if (acc == 0x9e3779b9u) *sink = acc;  // keeps the loads alive; practically never taken
}

// r[i] = a hash of i mapped to [-1, 1), zero on Dirichlet rows as in a solve
// (the on-chip forms count on it); *delta += sum r[i]^2 pinv[i].
template <class T>
__global__ void k_profile_seed(const SimDev* __restrict__ sp, T* __restrict__ r, const T* __restrict__ pinv,
                               double* delta) {
  const SimDev& s = *sp;
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < s.nn;
       i += (long long)gridDim.x * blockDim.x) {
    int a, b, c;
    node_of(s, i, a, b, c);
    unsigned int h = (unsigned int)i * 0x9E3779B1u;
    h ^= h >> 15;
    h *= 0x85EBCA77u;
    h ^= h >> 13;
    const T v = is_dirichlet(s, a, b, c) ? T(0) : (T)((double)(h >> 8) * (1.0 / 8388608.0) - 1.0);
    r[i] = v;
    acc += (double)v * (double)v * (double)pinv[i];
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(delta, acc);
}

// Puts every member into the middle of an inner solve that cannot converge:
// a seeded, well-scaled residual (pseudo-random entries in [-1, 1)) with
// delta = r^T P^-1 r computed for it, phase ITER, restart. Timed iterations
// are then ordinary CG iterations whatever state the members were left in
// (a converged step leaves a residual near underflow).
static heat_status profile_arm(Engine* e, double* d_delta, std::vector<double>& h_delta) {
  heat_status st = HEAT_OK;
  if (e->ncheb > 0)
    return set_error(HEAT_ERR_ARG, "profiling and tuning time the Jacobi iteration: set cheb_degree to 0 for them");
  if (cudaMemsetAsync(d_delta, 0, sizeof(double) * e->sims.size(), e->stream) != cudaSuccess)
    return set_error(HEAT_ERR_CUDA, "profile: memset failed");
  for (size_t i = 0; i < e->sims.size(); ++i) {
    heat_sim* s = e->sims[i];
    const int g = (int)std::min<long long>((s->nn + 255) / 256, 4LL * sm_count());
    if (e->prec == P_FP64) {
      k_profile_seed<double><<<g, 256, 0, e->stream>>>(s->d_dev, s->dev.r, s->dev.pinv, d_delta + i);
    } else {
      st = sim_read_scalars(s);
      if (st != HEAT_OK) return st;
      const int slot = e->ks.fused ? (s->h_sc->cgs & 1) : 0;
      k_profile_seed<float><<<g, 256, 0, e->stream>>>(s->d_dev, s->dev.rc32[slot], s->dev.pinv32, d_delta + i);
    }
  }
  if (cudaMemcpyAsync(h_delta.data(), d_delta, sizeof(double) * e->sims.size(), cudaMemcpyDeviceToHost,
                      e->stream) != cudaSuccess ||
      cudaStreamSynchronize(e->stream) != cudaSuccess)
    return set_error(HEAT_ERR_CUDA, "profile: residual seeding failed");
  for (size_t i = 0; i < e->sims.size(); ++i) {
    heat_sim* s = e->sims[i];
    st = sim_read_scalars(s);
    if (st != HEAT_OK) return st;
    SimScalars* sc = s->h_sc;
    sc->phase = PH_ITER;
    sc->iter = 1;
    sc->iter_step = 0;
    sc->restart = 1;
    sc->thresh = -1.0;
    sc->thresh_in = -1.0;
    sc->count = 0;
    sc->delta = h_delta[i] > 0.0 ? h_delta[i] : 1.0;
    st = sim_write_scalars(s);
    if (st != HEAT_OK) return st;
  }
  return HEAT_OK;
}

static heat_status profile_check(Engine* e) {
  if (e->ks.loop || e->has_res) {
    CUDA_TRY(cudaMemcpy(e->h_abort, &e->d_sync->abort, sizeof(int), cudaMemcpyDeviceToHost));
    if (*e->h_abort) {
      heat_status st = loop_abort(e);
      return st != HEAT_OK ? st : set_error(HEAT_ERR_TIMEOUT, "profile: a persistent iteration's wait ran out");
    }
  }
  for (heat_sim* s : e->sims) {
    heat_status st = sim_read_scalars(s);
    if (st != HEAT_OK) return st;
    if (s->h_sc->phase != PH_ITER)
      return set_error(HEAT_ERR_BREAKDOWN, "profile: the iteration left PH_ITER (status %d)", s->h_sc->status);
  }
  return HEAT_OK;
}

heat_status engine_profile(Engine* e, int reps, void* flush, size_t flush_bytes, double* ms_apply,
                           double* ms_update, double* bytes_apply, double* bytes_update) {
  const int chunk = 40;  // below the inner-solve cap and the true-residual period
  cudaEvent_t ev[4 * chunk];
  for (int i = 0; i < 4 * chunk; ++i) CUDA_TRY(cudaEventCreate(&ev[i]));
  double ta = 0.0, tu = 0.0;
  heat_status st = HEAT_OK;
  double* d_delta = nullptr;
  std::vector<double> h_delta(e->sims.size(), 0.0);
  if (cudaMalloc(&d_delta, sizeof(double) * e->sims.size()) != cudaSuccess) {
    cudaGetLastError();
    st = set_error(HEAT_ERR_NOMEM, "profile: no room for the residual norms");
  }
  const bool on_chip = e->has_res && !e->has_stream;
  for (int done = 0; done < reps && st == HEAT_OK && on_chip;) {
    // one launch runs a chunk of iterations; its time per iteration is reported as the apply's
    const int c = std::min(reps - done, chunk);
    st = loop_sync_reset(e, c);
    if (st == HEAT_OK) st = profile_arm(e, d_delta, h_delta);
    if (st != HEAT_OK) break;
    if (flush) k_flush_read<<<sm_count() * 4, 256, 0, e->stream>>>((const uint4*)flush, flush_bytes / 16, (unsigned int*)e->d_unfinished);
    cudaEventRecord(ev[0], e->stream);
    cudaError_t le = res_launch(e, e->stream);
    cudaEventRecord(ev[1], e->stream);
    if (le != cudaSuccess || cudaStreamSynchronize(e->stream) != cudaSuccess) {
      cudaGetLastError();
      st = set_error(HEAT_ERR_CUDA, "profile: launch failed");
      break;
    }
    float a = 0.f;
    cudaEventElapsedTime(&a, ev[0], ev[1]);
    ta += a;
    st = profile_check(e);
    done += c;
  }
  if (on_chip) {
    const heat_status st2 = loop_sync_reset(e);
    if (st == HEAT_OK) st = st2;
  }
  for (int done = 0; done < reps && st == HEAT_OK && !on_chip;) {
    const int c = std::min(reps - done, chunk);
    st = profile_arm(e, d_delta, h_delta);
    if (st != HEAT_OK) break;
    for (int i = 0; i < c; ++i) {
      if (flush) k_flush_read<<<sm_count() * 4, 256, 0, e->stream>>>((const uint4*)flush, flush_bytes / 16, (unsigned int*)e->d_unfinished);
      cudaEventRecord(ev[4 * i + 0], e->stream);
      {
        TileFn afn;
        int agrid, athreads, asmem;
        const int2* awork;
        const int* anwork;
        apply_launch(e, &afn, &agrid, &athreads, &awork, &anwork, &asmem);
        afn<<<agrid, athreads, asmem, e->stream>>>(e->d_sims, awork, anwork);
      }
      cudaEventRecord(ev[4 * i + 1], e->stream);
      if (flush && !e->ks.fused) k_flush_read<<<sm_count() * 4, 256, 0, e->stream>>>((const uint4*)flush, flush_bytes / 16, (unsigned int*)e->d_unfinished);
      cudaEventRecord(ev[4 * i + 2], e->stream);
      if (!e->ks.fused) e->ks.update<<<e->grid_pw, kPwThreads, 0, e->stream>>>(e->d_sims, e->d_work_pw, e->d_nwork + 1);
      cudaEventRecord(ev[4 * i + 3], e->stream);
    }
    if (cudaStreamSynchronize(e->stream) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
      st = set_error(HEAT_ERR_CUDA, "profile: launch failed");
      break;
    }
    for (int i = 0; i < c; ++i) {
      float a = 0.f, u = 0.f;
      cudaEventElapsedTime(&a, ev[4 * i + 0], ev[4 * i + 1]);
      if (!e->ks.fused) cudaEventElapsedTime(&u, ev[4 * i + 2], ev[4 * i + 3]);
      ta += a;
      tu += u;
    }
    st = profile_check(e);
    done += c;
  }
  for (int i = 0; i < 4 * chunk; ++i) cudaEventDestroy(ev[i]);
  cudaStreamSynchronize(e->stream);
  cudaFree(d_delta);
  if (st != HEAT_OK) return st;
  *ms_apply = ta / reps;
  *ms_update = tu / reps;
  // algorithmic bytes: every vector and coefficient touched once per launch, of
  // the members that the timed launches carry
  double ba = 0.0, bu = 0.0;
  for (size_t i = 0; i < e->sims.size(); ++i) {
    if (!on_chip && e->h_sims[i].res.g > 0) continue;
    const double n = (double)e->sims[i]->nn, ne = (double)e->sims[i]->ne;
    if (e->prec == P_FP64) {
      ba += n * (3 * 8 + 2 * 8) + ne * 16;    // r, P^-1, d_old in; d, q out; (rho_c, k)
      bu += n * (2 * 8 + 8 + 2 * 8 + 8 + 8);  // x in/out, d, r in/out, q, P^-1
    } else if (e->ks.fused) {
      ba += n * (6 * 4 + 5 * 4) + ne * 8;  // r, w, s, P^-1, p, e in; r', s', w', p, e out; (rho_c, k)
    } else {
      ba += n * (3 * 4 + 2 * 4) + ne * 8;
      bu += n * (2 * 4 + 4 + 2 * 4 + 4 + 4);
    }
  }
  // an iteration on the chip has no DRAM traffic of its own
  *bytes_apply = on_chip ? 0.0 : ba;
  *bytes_update = on_chip ? 0.0 : bu;
  return HEAT_OK;
}

heat_status prime_products(heat_sim* s, int nslots) {
  constexpr int SX = 16, SY = 16, TZ = 8;
  const SimDev& d = s->dev;
  const int ntx = (d.nx + 1 + SX - 2) / (SX - 1), nty = (d.ny + 1 + SY - 2) / (SY - 1);
  const int ntz = (d.nz + 1 + TZ - 1) / TZ;
  const long long grid = (long long)ntx * nty * ntz;
  if (grid > (1LL << 31) - 1) return set_error(HEAT_ERR_ARG, "prime_products: mesh too large");
  for (int v = 0; v < nslots; ++v) {
    if (d.elem == E_P1)
      k_product<SX, SY, E_P1><<<(unsigned)grid, SX * SY, 0, s->stream>>>(s->d_dev, d.vec64[v], d.yv[v], ntx, nty, TZ);
    else
      k_product<SX, SY><<<(unsigned)grid, SX * SY, 0, s->stream>>>(s->d_dev, d.vec64[v], d.yv[v], ntx, nty, TZ);
  }
  CUDA_TRY(cudaGetLastError());
  return HEAT_OK;
}

heat_status engine_time_iterations(Engine* e, int reps, double* ms_per_iter) {
  // 40 iterations per timed chunk: below the inner cap, and on small meshes
  // short of the point where a seeded residual has converged to rounding
  constexpr int kChunk = 40;
  const bool persistent = e->ks.loop || (e->has_res && !e->has_stream);
  const bool limited = e->ks.loop || e->has_res;  // launches that run several iterations
  const int per_tick = persistent ? kChunk : e->iters_per_tick;
  const int chunk_ticks = persistent ? 1 : std::max(1, kChunk / e->iters_per_tick);
  if (limited) {  // beside streaming members, one on the chip takes a tick's iterations too
    heat_status st = loop_sync_reset(e, per_tick);
    if (st != HEAT_OK) return st;
  }
  cudaEvent_t a, b;
  CUDA_TRY(cudaEventCreate(&a));
  if (cudaEventCreate(&b) != cudaSuccess) {
    cudaEventDestroy(a);
    return set_error(HEAT_ERR_CUDA, "timing: event creation failed");
  }
  heat_status st = HEAT_OK;
  double* d_delta = nullptr;
  std::vector<double> h_delta(e->sims.size(), 0.0);
  if (cudaMalloc(&d_delta, sizeof(double) * e->sims.size()) != cudaSuccess) {
    cudaGetLastError();
    st = set_error(HEAT_ERR_NOMEM, "timing: no room for the residual norms");
  }
  double ms = 0.0;
  long long iters = 0;
  for (int done = 0; done < reps && st == HEAT_OK;) {
    const int ticks = std::min(chunk_ticks, std::max(1, (reps - done + per_tick - 1) / per_tick));
    st = profile_arm(e, d_delta, h_delta);
    if (st != HEAT_OK) break;
    cudaEventRecord(a, e->stream);
    for (int t = 0; t < ticks && st == HEAT_OK; ++t)
      if (cudaGraphLaunch(e->gexec, e->stream) != cudaSuccess) st = set_error(HEAT_ERR_CUDA, "timing: graph launch failed");
    cudaEventRecord(b, e->stream);
    if (cudaEventSynchronize(b) != cudaSuccess) st = set_error(HEAT_ERR_CUDA, "timing: synchronisation failed");
    if (st != HEAT_OK) break;
    float t = 0.f;
    cudaEventElapsedTime(&t, a, b);
    ms += t;
    st = profile_check(e);
    if (st != HEAT_OK) break;
    // iterations actually run (profile_arm cleared iter_step; every member iterates alike)
    const long long n = e->sims[0]->h_sc->iter_step;
    iters += n;
    done += (int)std::max(1LL, n);
  }
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  cudaFree(d_delta);
  if (limited) {
    const heat_status st2 = loop_sync_reset(e);
    if (st == HEAT_OK) st = st2;
  }
  if (st != HEAT_OK) return st;
  *ms_per_iter = ms / (double)std::max(1LL, iters);
  return HEAT_OK;
}

// Segment sizes (output nodes per warp-segment tile) for table t's warp
// apply of precision prec on these simulations whose work items fill whole
// waves of resident blocks: for each count of waves, the largest levels per
// tile that keep the items within it, kept when the waves are at least 85%
// full; at most four, fewest waves first. Empty for the block-tile apply.
static std::vector<int> wave_segments(heat_sim* const* sims, int nsims, int prec, const Tuning& t, int bucket) {
  std::vector<int> out;
  const KernelSet ks = kernel_set(prec, t, members_ncheb_of(sims, nsims) > 0, sims[0]->dev.elem);
  if (!ks.apply_w) return out;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, ks.apply_w, 32 * ks.wwarps, ks.apply_w_smem) != cudaSuccess ||
      occ < 1) {
    cudaGetLastError();
    return out;
  }
  const long long cap = (long long)sm_count() * occ;
  const int per_level = (ks.wsx - 2) * ks.wny;
  const int levels = sims[0]->dev.nz + 1;
  long long best_items_for_waves[5] = {0, 0, 0, 0, 0};
  int best_seg_for_waves[5] = {0, 0, 0, 0, 0};
  for (int tz0 = levels; tz0 >= 4; --tz0) {
    const int seg = tz0 * per_level;
    if (seg > (1 << 20)) continue;
    KernelSet k2 = ks;
    k2.seg_nodes[bucket] = seg;
    long long items = 0;
    for (int i = 0; i < nsims; ++i) {
      SimDev d = sims[i]->dev;
      tile_geometry(d, k2, prec == P_FP64);
      items += d.w_items;
    }
    const long long waves = (items + cap - 1) / cap;
    if (waves < 1 || waves > 4) continue;
    if (items > best_items_for_waves[waves]) {  // the fullest last wave, largest tiles on ties
      best_items_for_waves[waves] = items;
      best_seg_for_waves[waves] = seg;
    }
  }
  for (int w = 1; w <= 4; ++w)
    if (best_seg_for_waves[w] && best_items_for_waves[w] >= (long long)(0.85 * (double)(w * cap)))
      out.push_back(best_seg_for_waves[w]);
  return out;
}

heat_status engine_autotune(heat_sim* const* sims, int nsims, int reps, int* best_variant, int* best_seg,
                            double* best_ms) {
  static const int kSegs[] = {256, 512, 1024, 2048};
  const int prec = sims[0]->prm.precision;
  const int bucket = size_bucket(sims[0]->nn);
  const Tuning base = tuning_get();
  Tuning best = base;
  double best_t = 1e300;
  heat_status st = HEAT_OK;
  // each warp variant's best time over the fixed segment sizes
  std::vector<double> vbest(kNumVariants, 1e300);
  for (int v = -1; v < kNumVariants && st == HEAT_OK; ++v) {
    if (v >= 0 && prec == P_FP64 && !kVariants[v].f64[0]) continue;
    // the on-chip solve does not depend on the segment size: it keeps the
    // table's, which the FP64 apply and the streaming meshes also follow
    for (int si = 0; si < (v < 0 || kVariants[v].res ? 1 : 4) && st == HEAT_OK; ++si) {
      Tuning t = base;
      t.variant[prec] = v;
      if (v >= 0 && !kVariants[v].res) t.seg_nodes[bucket] = kSegs[si];
      Engine* e = nullptr;
      st = engine_create(sims, nsims, prec, sims[0]->stream, &e, &t);
      if (st != HEAT_OK) break;
      // CG iterations as the solve runs them: the captured tick graph
      double ms = 0.0;
      st = engine_time_iterations(e, 8, &ms);  // warm-up
      if (st == HEAT_OK) st = engine_time_iterations(e, reps, &ms);
      engine_destroy(e);
      if (st == HEAT_OK && v >= 0) vbest[v] = std::min(vbest[v], ms);
      if (st == HEAT_OK && ms < best_t) {
        best_t = ms;
        best = t;
      }
    }
  }
  // then wave-aligned segment sizes for the two fastest warp applies: the levels
  // per segment tile whose total work items fill the resident blocks
  // (SMs x blocks per SM) best, a few waves at most (a launch whose last
  // wave is partly empty leaves SMs idle: on the 100^3 mesh 338 items on
  // 456 resident blocks run three blocks on some SMs and two on the others)
  int top[2] = {-1, -1};
  for (int v = 0; v < kNumVariants; ++v) {
    if (vbest[v] >= 1e300) continue;
    if (top[0] < 0 || vbest[v] < vbest[top[0]]) {
      top[1] = top[0];
      top[0] = v;
    } else if (top[1] < 0 || vbest[v] < vbest[top[1]]) {
      top[1] = v;
    }
  }
  for (int v : top) {
    if (v < 0 || kVariants[v].res || st != HEAT_OK) continue;
    Tuning tv = base;
    tv.variant[prec] = v;
    for (int seg : wave_segments(sims, nsims, prec, tv, bucket)) {
      if (st != HEAT_OK) break;
      bool tried = false;
      for (int k : kSegs) tried = tried || k == seg;
      if (tried) continue;
      Tuning t = tv;
      t.seg_nodes[bucket] = seg;
      Engine* e = nullptr;
      st = engine_create(sims, nsims, prec, sims[0]->stream, &e, &t);
      if (st != HEAT_OK) break;
      double ms = 0.0;
      st = engine_time_iterations(e, 8, &ms);
      if (st == HEAT_OK) st = engine_time_iterations(e, reps, &ms);
      engine_destroy(e);
      if (st == HEAT_OK && ms < best_t) {
        best_t = ms;
        best = t;
      }
    }
  }
  // then the pointwise kernel's item size with the chosen apply
  const Tuning chosen = best;
  for (int qpt : {1, 2, 4}) {
    if (st != HEAT_OK || qpt == chosen.pw_quads[prec]) continue;
    Tuning t = chosen;
    t.pw_quads[prec] = qpt;
    Engine* e = nullptr;
    st = engine_create(sims, nsims, prec, sims[0]->stream, &e, &t);
    if (st != HEAT_OK) break;
    double ms = 0.0;
    st = engine_time_iterations(e, 8, &ms);
    if (st == HEAT_OK) st = engine_time_iterations(e, reps, &ms);
    engine_destroy(e);
    if (st == HEAT_OK && ms < best_t) {
      best_t = ms;
      best = t;
    }
  }
  // then the persistent iteration with each item size (FP32 paths, where
  // the chosen apply has a persistent form)
  const Tuning chosen2 = best;
  for (int qpt : {1, 2, 4}) {
    if (st != HEAT_OK || prec == P_FP64) break;
    Tuning t = chosen2;
    t.loop[prec] = 1;
    t.pw_quads[prec] = qpt;
    if (!kernel_set(prec, t, members_ncheb_of(sims, nsims) > 0, sims[0]->dev.elem).loop) continue;
    Engine* e = nullptr;
    st = engine_create(sims, nsims, prec, sims[0]->stream, &e, &t);
    if (st != HEAT_OK) break;
    double ms = 0.0;
    st = engine_time_iterations(e, 8, &ms);
    if (st == HEAT_OK) st = engine_time_iterations(e, reps, &ms);
    engine_destroy(e);
    if (st == HEAT_OK && ms < best_t) {
      best_t = ms;
      best = t;
    }
  }
  if (st != HEAT_OK) return st;
  st = tuning_set(best);
  if (st != HEAT_OK) return st;
  *best_variant = best.variant[prec];
  *best_seg = best.seg_nodes[bucket];
  *best_ms = best_t;
  return HEAT_OK;
}

}  // namespace heat

extern "C" heat_status heat_debug_loop_wait(unsigned int extra_arrivals, double limit_s) {
  if (extra_arrivals > 1u || !(limit_s >= 0.0) || limit_s > 60.0)
    return heat::set_error(HEAT_ERR_ARG, "heat_debug_loop_wait: need extra_arrivals in {0, 1}, 0 <= limit_s <= 60");
  heat::g_loop_extra.store(extra_arrivals);
  heat::g_loop_limit_ns.store((unsigned long long)(limit_s * 1e9));
  return HEAT_OK;
}

extern "C" heat_status heat_debug_fail_engine_builds(int n) {
  if (n < 0) return heat::set_error(HEAT_ERR_ARG, "heat_debug_fail_engine_builds: n must be >= 0");
  heat::g_fail_builds.store(n);
  return HEAT_OK;
}
