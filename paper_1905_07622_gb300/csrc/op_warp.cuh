// The factorised operator (see op.cuh) with the y direction held in
// registers: a warp-segment tile.
//
// A segment of SX lanes (SX divides 32) owns node columns x = i0-1+lx; each
// thread holds NY+2 consecutive y rows of its column and marches up the z
// levels. Forward x and the final x-sum use segment shuffles; forward y,
// forward z, scaling, inverse z, the face sums and inverse y all stay in the
// thread's registers, so the level loop has no block barrier, and the NY rows
// are independent instruction streams. Outputs are lanes 1..SX-2 (the outer
// lanes only supply neighbours), rows 1..NY, levels [k0, k0+nzt):
// (SX-2) x NY x nzt nodes per segment.
//
// Where the loads come from is a policy (the Src argument):
//  - RegSrc: plain loads one level ahead into registers;
//  - AsyncSrc: each thread copies its own rows S-1 levels ahead into a
//    private ring of S stages in shared memory with cp.async (no registers held
//    for data in flight, no barrier: a thread reads back only what it copied,
//    after waiting for its own copy groups).
#pragma once

#include <type_traits>
#include <utility>

#include "op.cuh"

namespace heat {

// Pairs of values with element-wise arithmetic: packed FP32x2 instructions for
// float (two results per issued instruction on sm_100 and later), two scalar
// operations for double. fma(a, b, c) = a*b + c with one rounding per lane.
template <class T> struct Pair2;
template <> struct Pair2<float> {
  using t = float2;
  static __device__ __forceinline__ float2 make(float a, float b) { return make_float2(a, b); }
  static __device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
  static __device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
  static __device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
  // a - b, exact as a subtraction
  static __device__ __forceinline__ float2 sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
};
template <> struct Pair2<double> {
  using t = double2;
  static __device__ __forceinline__ double2 make(double a, double b) { return make_double2(a, b); }
  static __device__ __forceinline__ double2 add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
  static __device__ __forceinline__ double2 mul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
  static __device__ __forceinline__ double2 fma(double2 a, double2 b, double2 c) {
    return make_double2(::fma(a.x, b.x, c.x), ::fma(a.y, b.y, c.y));
  }
  static __device__ __forceinline__ double2 sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
};

// Double-float pairs (df.cuh): the refinement passes' arithmetic, about 48
// significant bits from FP32 instructions.
template <> struct Pair2<DF> {
  using t = DF2;
  static __device__ __forceinline__ DF2 make(DF a, DF b) { return DF2{a, b}; }
  static __device__ __forceinline__ DF2 add(DF2 a, DF2 b) { return DF2{a.x + b.x, a.y + b.y}; }
  static __device__ __forceinline__ DF2 mul(DF2 a, DF2 b) { return DF2{a.x * b.x, a.y * b.y}; }
  static __device__ __forceinline__ DF2 fma(DF2 a, DF2 b, DF2 c) { return DF2{a.x * b.x + c.x, a.y * b.y + c.y}; }
  static __device__ __forceinline__ DF2 sub(DF2 a, DF2 b) { return DF2{a.x - b.x, a.y - b.y}; }
};

// One element's precomputed Walsh-pair coefficients A_0..A_3, B_0..B_3 of the
// A operator (SimDev::acoef): FP64 pairs, or (hi, lo) float pairs for DF.
struct alignas(16) PreRec {
  float4 w[4];
};

// The march's per-element pair coefficients (A_q, B_q) for the pair halves
// h = 0 (q = 0, 1) and h = 1 (q = 2, 3): formed from the element's (rho_c,
// k) and the scaled eigenvalue sums AM, AK, BM, BK, or read from a PreRec.
template <class T, class C, class T2>
__device__ __forceinline__ void march_coeffs(const C& cf, const T2 (&AM)[2], const T2 (&AK)[2], const T2 (&BM)[2],
                                             const T2 (&BK)[2], T2 (&A)[2], T2 (&B)[2]) {
  using V = Pair2<T>;
  const T2 rc = V::make(cf.x, cf.x), kc = V::make(cf.y, cf.y);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    A[h] = V::fma(kc, AK[h], V::mul(rc, AM[h]));
    B[h] = V::fma(kc, BK[h], V::mul(rc, BM[h]));
  }
}
template <class T, class T2>
__device__ __forceinline__ void march_coeffs(const PreRec& cf, const T2 (&)[2], const T2 (&)[2], const T2 (&)[2],
                                             const T2 (&)[2], T2 (&A)[2], T2 (&B)[2]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if constexpr (sizeof(T) == 8 && !std::is_same<T, DF>::value) {
      A[h] = *reinterpret_cast<const T2*>(&cf.w[h]);
      B[h] = *reinterpret_cast<const T2*>(&cf.w[2 + h]);
    } else {
      A[h] = T2{T(cf.w[h].x, cf.w[h].y), T(cf.w[h].z, cf.w[h].w)};
      B[h] = T2{T(cf.w[2 + h].x, cf.w[2 + h].y), T(cf.w[2 + h].z, cf.w[2 + h].w)};
    }
  }
}

// Geometry of one lane of a segment tile: which of its rows exist, which are
// Dirichlet, where its column starts.
template <int NY>
struct LaneGeo {
  static constexpr int NR = NY + 2;  // staged rows
  static constexpr int NF = NY + 1;  // faces / element rows
  bool out_lane;
  unsigned rin, rdxy, ein, rstat;  // bit r: row inside / x-y Dirichlet / element row valid / loadable
  int nbase, ebase, estride, pxy, gnz, px, enx;
  bool dz0, dz1, mask;
  SimScalars* sc;      // where HEAT_CHECK builds count out-of-range indices
  long long nn, ne;    // node and element counts (the index bounds)

  __device__ __forceinline__ LaneGeo(const Geo& g, bool active, int lx, int SX, int i0, int j0, bool mask_,
                                     SimScalars* sc_ = nullptr) {
    sc = sc_;
    nn = (long long)g.px * (g.ny + 1) * (g.nz + 1);
    ne = (long long)g.nx * g.ny * g.nz;
    const int c = i0 - 1 + lx;
    const bool col_in = active && c >= 0 && c <= g.nx;
    out_lane = active && lx >= 1 && lx <= SX - 2 && c <= g.nx;
    const bool ecol = active && c >= 0 && c < g.nx;
    const bool dx = col_in && (((g.dir & 1u) && c == 0) || ((g.dir & 2u) && c == g.nx));
    rin = rdxy = ein = 0u;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int j = j0 - 1 + r;
      const bool in = col_in && j >= 0 && j <= g.ny;
      if (in) rin |= 1u << r;
      if (in && (dx || ((g.dir & 4u) && j == 0) || ((g.dir & 8u) && j == g.ny))) rdxy |= 1u << r;
      if (r < NF && ecol && j >= 0 && j < g.ny) ein |= 1u << r;
    }
    nbase = c + g.px * (j0 - 1);  // node index of row 0 at level 0 (rows step by px)
    ebase = c + g.nx * (j0 - 1);  // element index of element row 0 at level 0
    estride = g.nx * g.ny;
    pxy = g.pxy;
    gnz = g.nz;
    px = g.px;
    enx = g.nx;
    dz0 = (g.dir & 16u) != 0;
    dz1 = (g.dir & 32u) != 0;
    mask = mask_;
    rstat = rin & ~(mask ? rdxy : 0u);  // rows that can be live at any level
  }
  // rows of node level L that hold unknowns (bit r)
  __device__ __forceinline__ unsigned live_rows(int L) const {
    const bool lev = L >= 0 && L <= gnz && !(mask && ((dz0 && L == 0) || (dz1 && L == gnz)));
    return lev ? rstat : 0u;
  }
  // element rows of element layer E inside the mesh (bit r)
  __device__ __forceinline__ unsigned live_elems(int E) const { return (E >= 0 && E < gnz) ? ein : 0u; }
};

// *p where live, else zero: one predicated load, no branch around it (FP32;
// the FP64 kernels wait for the FP64 pipe instead). A time step on 200^3, which
// streams its vectors: 184.6 -> 180.0 ms.
__device__ __forceinline__ float ld_if(const float* p, bool live) {
  float v;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t@p ld.global.f32 %0, [%1];\n\t}"
               : "=f"(v) : "l"(p), "r"((int)live));
  return v;
}
__device__ __forceinline__ float2 ld_if(const float2* p, bool live) {
  float2 v;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.f32 %0, 0f00000000;\n\tmov.f32 %1, 0f00000000;\n\t"
               "@p ld.global.v2.f32 {%0, %1}, [%2];\n\t}"
               : "=f"(v.x), "=f"(v.y) : "l"(p), "r"((int)live));
  return v;
}
__device__ __forceinline__ double ld_if(const double* p, bool live) { return live ? *p : 0.0; }
__device__ __forceinline__ double2 ld_if(const double2* p, bool live) { return live ? *p : make_double2(0.0, 0.0); }

// Loads one level ahead into registers through caller-supplied functors:
// fetch(node, live) -> Raw, value(Raw) -> T.
template <class T, int NY, class Coef, class Fetch, class Value>
struct RegSrc {
  static constexpr int NR = NY + 2, NF = NY + 1;
  using Raw = decltype(std::declval<Fetch&>()(0, false));
  const Coef* __restrict__ coef;
  Fetch& fetch;
  Value& value;
  int k0;
  Raw raw[NR];
  Coef cf[NF];

  __device__ __forceinline__ RegSrc(const Coef* c, Fetch& f, Value& v, int k0_) : coef(c), fetch(f), value(v), k0(k0_) {}
  __device__ __forceinline__ void load_nodes(const LaneGeo<NY>& lg, int L) {
    const unsigned lv = lg.live_rows(L);
    const int off = lg.nbase + L * lg.pxy;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int m = off + r * lg.px;
      raw[r] = fetch(m, ((lv >> r) & 1u) && HEAT_INDEX_OK(lg.sc, m, lg.nn));
    }
  }
  __device__ __forceinline__ void load_coef(const LaneGeo<NY>& lg, int E) {
    const unsigned le = lg.live_elems(E);
#pragma unroll
    for (int r = 0; r < NF; ++r) {
      const int e = lg.ebase + r * lg.enx + E * lg.estride;
      cf[r] = ld_if(coef + e, ((le >> r) & 1u) && HEAT_INDEX_OK(lg.sc, e, lg.ne));
    }
  }
  // before the loop: node level k0-1, element layer k0-1 (used at t = 1)
  __device__ __forceinline__ void prologue(const LaneGeo<NY>& lg, int) {
    load_nodes(lg, k0 - 1);
    load_coef(lg, k0 - 1);
  }
  // values of node level L = k0-1+t, then the next level's loads
  __device__ __forceinline__ void level(const LaneGeo<NY>& lg, int t, int tzl, T v[NR]) {
#pragma unroll
    for (int r = 0; r < NR; ++r) v[r] = value(raw[r]);
    if (t <= tzl) load_nodes(lg, k0 + t);  // in flight during this level's arithmetic
  }
  // coefficients of element layer k0-2+t (valid for t >= 1)
  __device__ __forceinline__ Coef coef_row(int, int r) const { return cf[r]; }
  __device__ __forceinline__ void after_elements(const LaneGeo<NY>& lg, int t, int tzl) {
    if (t <= tzl) load_coef(lg, k0 - 1 + t);
  }
};

// RegSrc with each element row's coefficients read as a PreRec
// from SimDev::acoef: the warp-segment march of the A operator with its
// per-element coefficients precomputed.
// AHEAD: the coefficients too are loaded one layer ahead into registers; without
// it each row's are loaded where they are used (FP64: 16 registers per row
// saved, and the FP64 pipe hides the latency).
template <class T, int NY, class Fetch, class Value, bool AHEAD = true>
struct PreRegSrc {
  static constexpr int NR = NY + 2, NF = NY + 1;
  using Raw = decltype(std::declval<Fetch&>()(0, false));
  const float4* __restrict__ pre;
  Fetch& fetch;
  Value& value;
  int k0;
  Raw raw[NR];
  PreRec cf[AHEAD ? NF : 1];
  const LaneGeo<NY>* geo = nullptr;

  __device__ __forceinline__ PreRegSrc(const float4* p, Fetch& f, Value& v, int k0_)
      : pre(p), fetch(f), value(v), k0(k0_) {}
  __device__ __forceinline__ void load_nodes(const LaneGeo<NY>& lg, int L) {
    const unsigned lv = lg.live_rows(L);
    const int off = lg.nbase + L * lg.pxy;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int m = off + r * lg.px;
      raw[r] = fetch(m, ((lv >> r) & 1u) && HEAT_INDEX_OK(lg.sc, m, lg.nn));
    }
  }
  __device__ __forceinline__ PreRec load_row(const LaneGeo<NY>& lg, unsigned le, int E, int r) const {
    PreRec c;
    const int e = lg.ebase + r * lg.enx + E * lg.estride;
    if (((le >> r) & 1u) && HEAT_INDEX_OK(lg.sc, e, lg.ne)) {
      const float4* p = pre + 4 * (long long)e;
#pragma unroll
      for (int w = 0; w < 4; ++w) c.w[w] = __ldg(p + w);
    } else {
#pragma unroll
      for (int w = 0; w < 4; ++w) c.w[w] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    return c;
  }
  __device__ __forceinline__ void load_coef(const LaneGeo<NY>& lg, int E) {
    if constexpr (AHEAD) {
      const unsigned le = lg.live_elems(E);
#pragma unroll
      for (int r = 0; r < NF; ++r) cf[r] = load_row(lg, le, E, r);
    }
  }
  __device__ __forceinline__ void prologue(const LaneGeo<NY>& lg, int) {
    geo = &lg;
    load_nodes(lg, k0 - 1);
    load_coef(lg, k0 - 1);
  }
  __device__ __forceinline__ void level(const LaneGeo<NY>& lg, int t, int tzl, T v[NR]) {
#pragma unroll
    for (int r = 0; r < NR; ++r) v[r] = value(raw[r]);
    if (t <= tzl) load_nodes(lg, k0 + t);
  }
  // element layer k0-2+t
  __device__ __forceinline__ PreRec coef_row(int t, int r) const {
    if constexpr (AHEAD) return cf[r];
    else return load_row(*geo, geo->live_elems(k0 - 2 + t), k0 - 2 + t, r);
  }
  __device__ __forceinline__ void after_elements(const LaneGeo<NY>& lg, int t, int tzl) {
    if (t <= tzl) load_coef(lg, k0 - 1 + t);
  }
};

// cp.async of 4, 8 or 16 bytes into shared memory; live = false writes zeros
// and reads nothing (the source address must still be a valid pointer).
template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem, bool live) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  const int n = live ? BYTES : 0;
  if (BYTES == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sa), "l"(gmem), "r"(n) : "memory");
  else if (BYTES == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(sa), "l"(gmem), "r"(n) : "memory");
  else
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Shared-memory bytes one thread of AsyncSrc<T, NY, S> uses.
template <class T, int NY, int S>
__host__ __device__ constexpr int async_stage_bytes() {
  return S * ((NY + 2) * 3 * (int)sizeof(T) + (NY + 1) * 2 * (int)sizeof(T));
}

// The direction-fused apply's loads (P^-1, r, d_old per node; (rho_c, k) per
// element) staged through a per-thread ring of S stages; dold = nullptr is a
// restart. Stage t holds node level k0-1+t and element layer k0-2+t. Layout:
// planes of nt values (one per thread of the block), so a warp's accesses are
// conflict-free.
template <class T, int NY, int S, class Coef>
struct AsyncSrc {
  static constexpr int NR = NY + 2, NF = NY + 1;
  static_assert(S >= 2, "at least two stages");
  const T* __restrict__ pinv;
  const T* __restrict__ r;
  const T* __restrict__ dold;  // nullptr: restart, d_old = 0
  const Coef* __restrict__ coef;
  T beta;
  T* nodes;     // [S][NR][3][nt]
  Coef* elems;  // [S][NF][nt]
  int nt, tid, k0;

  __device__ __forceinline__ AsyncSrc(const T* p, const T* rr, const T* d, const Coef* c, T b, void* smem, int nthreads,
                                      int thread, int k0_)
      : pinv(p), r(rr), dold(d), coef(c), beta(b), nt(nthreads), tid(thread), k0(k0_) {
    nodes = reinterpret_cast<T*>(smem);
    elems = reinterpret_cast<Coef*>(nodes + S * NR * 3 * nt);
  }
  __device__ __forceinline__ T* node_slot(int st, int row, int comp) const {
    return nodes + ((st * NR + row) * 3 + comp) * nt + tid;
  }
  __device__ __forceinline__ Coef* elem_slot(int st, int row) const { return elems + (st * NF + row) * nt + tid; }

  // copies for stage t (node level k0-1+t, element layer k0-2+t) as one group
  __device__ __forceinline__ void issue(const LaneGeo<NY>& lg, int t) {
    const int st = t % S;
    const int L = k0 - 1 + t, E = L - 1;
    const unsigned lv = lg.live_rows(L);
    const int off = lg.nbase + L * lg.pxy;
#pragma unroll
    for (int row = 0; row < NR; ++row) {
      const bool live = ((lv >> row) & 1u) && HEAT_INDEX_OK(lg.sc, off + row * lg.px, lg.nn);
      const int m = live ? off + row * lg.px : 0;
      cp_async<sizeof(T)>(node_slot(st, row, 0), pinv + m, live);
      cp_async<sizeof(T)>(node_slot(st, row, 1), r + m, live);
      if (dold) cp_async<sizeof(T)>(node_slot(st, row, 2), dold + m, live);
    }
    const unsigned le = lg.live_elems(E);
#pragma unroll
    for (int row = 0; row < NF; ++row) {
      const bool live =
          ((le >> row) & 1u) && HEAT_INDEX_OK(lg.sc, lg.ebase + row * lg.enx + E * lg.estride, lg.ne);
      const int e = live ? lg.ebase + row * lg.enx + E * lg.estride : 0;
      cp_async<sizeof(Coef)>(elem_slot(st, row), coef + e, live);
    }
    cp_async_commit();
  }
  __device__ __forceinline__ void prologue(const LaneGeo<NY>& lg, int tzl) {
#pragma unroll
    for (int t = 0; t < S - 1; ++t) {
      if (t <= tzl + 1) issue(lg, t);
      else cp_async_commit();  // one group per stage keeps the wait count fixed
    }
  }
  __device__ __forceinline__ void level(const LaneGeo<NY>& lg, int t, int tzl, T v[NR]) {
    // stage t+S-1 reuses the slot of stage t-1, which the previous level consumed
    if (t + S - 1 <= tzl + 1) issue(lg, t + S - 1);
    else cp_async_commit();
    cp_async_wait<S - 1>();  // stage t has landed
    const int st = t % S;
#pragma unroll
    for (int row = 0; row < NR; ++row) {
      const T p = *node_slot(st, row, 0), rv = *node_slot(st, row, 1);
      const T d = dold ? *node_slot(st, row, 2) : T(0);
      v[row] = p * rv + beta * d;
    }
  }
  __device__ __forceinline__ Coef coef_row(int t, int row) const { return *elem_slot(t % S, row); }
  __device__ __forceinline__ void after_elements(const LaneGeo<NY>&, int, int) {}
};

// The march's constants for the operator (sa M + sb K): with lam_q and lam'_q
// = lam_{q+4} (the two z-Walsh indices of an xy index q), the face sum and the
// element's top half are
//   G_q = Tp_q + A_q Fp_q + B_q F_q,  Tn_q = B_q Fp_q + A_q F_q,
//   A_q = lam_q + lam'_q,  B_q = lam_q - lam'_q,
// and A_q, B_q are linear in (rho_c, k). The four xy indices are processed as
// two pairs, h = 0: q = (0, 1), h = 1: q = (2, 3).
//
// THIRD (float and double coefficients (rho_c, k)): the eigenvalues are
//   lam_w = m0 3^-|w| (sa rho_c + sb k sigma_w), sigma_w = sum of 12 / h_d^2 over w's differences,
// so with the factors 1/3 of x and y moved into the inverse butterflies (an
// addition becomes a multiply-add) the coefficients are A_q = R + k al_q,
// B_q = R / 2 + k be_q with R = (4/3) m0 sa rho_c, al_q = m0 sb (4 sigma_q + zeta) / 3,
// be_q = m0 sb (2 sigma_q - zeta) / 3, zeta = 12 / h_z^2: 8 multiply-adds and 2
// products per element instead of 16 and 8. The constants are rounded once, on
// the host, and k enters as it is: an FP64 product's error is then the plain
// form's (40^3, smooth x: 1.24e-15 both; with m0 sb k rounded before, 1.34e-15).
// Double-float has no
// multiply-add to hide the 1/3 in and keeps the plain form, as do coefficients
// that are precomputed (PreRec).
template <class T, bool THIRD>
struct MarchQ1T;
template <class T>
struct MarchQ1T<T, false> {
  using V = Pair2<T>;
  using T2 = typename V::t;
  T2 AM[2], AK[2], BM[2], BK[2];
  MarchQ1T() = default;
  __device__ __forceinline__ MarchQ1T(const SimDev& s, T sa, T sb) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int q0 = 2 * h, q1 = 2 * h + 1;
      AM[h] = V::make(sa * (lam_m<T>(s, q0) + lam_m<T>(s, q0 + 4)), sa * (lam_m<T>(s, q1) + lam_m<T>(s, q1 + 4)));
      AK[h] = V::make(sb * (lam_k<T>(s, q0) + lam_k<T>(s, q0 + 4)), sb * (lam_k<T>(s, q1) + lam_k<T>(s, q1 + 4)));
      BM[h] = V::make(sa * (lam_m<T>(s, q0) - lam_m<T>(s, q0 + 4)), sa * (lam_m<T>(s, q1) - lam_m<T>(s, q1 + 4)));
      BK[h] = V::make(sb * (lam_k<T>(s, q0) - lam_k<T>(s, q0 + 4)), sb * (lam_k<T>(s, q1) - lam_k<T>(s, q1 + 4)));
    }
  }
  template <class C>
  __device__ __forceinline__ void coeffs(const C& cf, T2 (&A)[2], T2 (&B)[2]) const {
    march_coeffs<T>(cf, AM, AK, BM, BK, A, B);
  }
};
template <class T>
struct MarchQ1T<T, true> {
  using V = Pair2<T>;
  using T2 = typename V::t;
  T2 al[2], be[2];
  T ra;
  MarchQ1T() = default;
  __device__ __forceinline__ MarchQ1T(const SimDev& s, T sa, T sb) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // (a conversion is an FP64 instruction: floats have their own copies)
      if constexpr (sizeof(T) == 8) {
        al[h] = V::make(sb * s.tal[2 * h], sb * s.tal[2 * h + 1]);
        be[h] = V::make(sb * s.tbe[2 * h], sb * s.tbe[2 * h + 1]);
        ra = s.m43 * sa;
      } else {
        al[h] = V::make(sb * s.tal_f[2 * h], sb * s.tal_f[2 * h + 1]);
        be[h] = V::make(sb * s.tbe_f[2 * h], sb * s.tbe_f[2 * h + 1]);
        ra = s.m43_f * sa;
      }
    }
  }
  template <class C>
  __device__ __forceinline__ void coeffs(const C& cf, T2 (&A)[2], T2 (&B)[2]) const {
    const T R = ra * cf.x, half = T(0.5);
    const T2 R2 = V::make(R, R), K2 = V::make(cf.y, cf.y);
    T2 H2;  // FP32: one packed product (200^3: 54.6 -> 53.8 us); FP64: one product for both
    if constexpr (sizeof(T) == 4) H2 = V::mul(R2, V::make(half, half));
    else H2 = V::make(half * R, half * R);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      A[h] = V::fma(K2, al[h], R2);
      B[h] = V::fma(K2, be[h], H2);
    }
  }
};
template <class T>
using MarchQ1 = MarchQ1T<T, !std::is_same<T, DF>::value>;
// with precomputed coefficients nothing is needed
template <class T>
struct MarchPre {
  using V = Pair2<T>;
  using T2 = typename V::t;
  __device__ __forceinline__ void coeffs(const PreRec& cf, T2 (&A)[2], T2 (&B)[2]) const {
    const T2 z[2] = {};
    march_coeffs<T>(cf, z, z, z, z, A, B);
  }
};
template <class MC> struct IsThird : std::false_type {};
template <class T> struct IsThird<MarchQ1T<T, true>> : std::true_type {};

// Every lane of the segment must call this with the same tzl (the trip count
// of the level loop): shuffles span the segment. Segments with no tile pass
// active = false (they load and store nothing). Levels beyond the mesh are
// zero; outputs are clipped to the mesh. out(node, dirichlet, y, v) receives
// the operator output y and the node's own input value v.
//
// pre(node, in) loads what out needs at a node (in false: nothing to load, no
// output); it runs before a level's arithmetic and out receives its result,
// so those loads are in flight meanwhile.
//
// lev(t) runs after a level's outputs (t = 2, 3, ..; the same t in every lane).
struct NoLev {
  __device__ __forceinline__ void operator()(int) const {}
};
template <class T, int SX, int NY, class MC, class Src, class Pre, class Out, class Lev = NoLev>
__device__ __forceinline__ void warp_tile_march_pre(const LaneGeo<NY>& lg, const MC& mc, Src& src, int tzl, Pre&& pre,
                                                    Out&& out, Lev&& lev = Lev{}) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int NR = NY + 2;  // staged rows
  constexpr int NF = NY + 1;  // faces / element rows
  using V = Pair2<T>;
  using T2 = typename V::t;
  constexpr bool THIRD = IsThird<MC>::value;
  src.prologue(lg, tzl);
  T2 Fp[NF][2], Tp[NF][2];
  T vprev[NY];
#pragma unroll
  for (int r = 0; r < NF; ++r)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      Fp[r][h] = V::make(T(0), T(0));
      Tp[r][h] = V::make(T(0), T(0));
    }
#pragma unroll
  for (int r = 0; r < NY; ++r) vprev[r] = T(0);

  const int k0 = src.k0;
  for (int t = 0; t <= tzl + 1; ++t) {
    const int L = k0 - 1 + t;
    T v[NR];
    src.level(lg, t, tzl, v);
    decltype(pre(0, false)) got[NY];
#pragma unroll
    for (int r = 1; r <= NY; ++r) {
      const int m = lg.nbase + r * lg.px + (L - 1) * lg.pxy;
      got[r - 1] = pre(m, t >= 2 && lg.out_lane && L - 1 <= lg.gnz && ((lg.rin >> r) & 1u) != 0u &&
                              HEAT_INDEX_OK(lg.sc, m, lg.nn));
    }
    // forward x (edges of each row, as the pair (sum, difference)) and
    // forward y (faces between rows): F[r][0] = (F_0, F_1), F[r][1] = (F_2, F_3)
    T2 E[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const T vr = __shfl_down_sync(FULL, v[r], 1, SX);
      E[r] = V::make(v[r] + vr, v[r] - vr);
    }
    T2 F[NF][2];
#pragma unroll
    for (int r = 0; r < NF; ++r) {
      F[r][0] = V::add(E[r], E[r + 1]);
      F[r][1] = V::sub(E[r], E[r + 1]);
    }
    if (t >= 1) {
      // elements (c, j0-1+r, L-1) between face levels L-1 and L
      T2 G[NF][2];
#pragma unroll
      for (int r = 0; r < NF; ++r) {
        T2 A[2], B[2];
        mc.coeffs(src.coef_row(t, r), A, B);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          G[r][h] = V::fma(B[h], F[r][h], V::fma(A[h], Fp[r][h], Tp[r][h]));
          Tp[r][h] = V::fma(A[h], F[r][h], V::mul(B[h], Fp[r][h]));
        }
      }
      src.after_elements(lg, t, tzl);
      if (t >= 2) {
        // node level L-1 is complete: inverse y, inverse x, x-sum
        const int lv = L - 1;
        const bool lvin = lv <= lg.gnz;
        const bool dzl = (lg.dz0 && lv == 0) || (lg.dz1 && lv == lg.gnz);
#pragma unroll
        for (int r = 1; r <= NY; ++r) {
          // (g0, g1) = (G_0 + G_2, G_1 + G_3) of row r + (G_0 - G_2, G_1 - G_3) of row r-1
          T2 g;
          T nl, nr;
          if constexpr (THIRD) {
            const T2 TH = V::make(T(1.0 / 3.0), T(1.0 / 3.0));
            // G_0 + G_2 / 3 of row r, G_0 - G_2 / 3 of row r - 1: the thirds of both in one product
            g = V::fma(V::sub(G[r][1], G[r - 1][1]), TH, V::add(G[r][0], G[r - 1][0]));
            nl = g.x + T(1.0 / 3.0) * g.y;
            nr = g.x - T(1.0 / 3.0) * g.y;
          } else {
            g = V::add(V::add(G[r][0], G[r][1]), V::sub(G[r - 1][0], G[r - 1][1]));
            nl = g.x + g.y;
            nr = g.x - g.y;
          }
          const T from_left = __shfl_up_sync(FULL, nr, 1, SX);
          const int m = lg.nbase + r * lg.px + lv * lg.pxy;
          if (lg.out_lane && lvin && ((lg.rin >> r) & 1u) && HEAT_INDEX_OK(lg.sc, m, lg.nn)) {
            const bool dir = ((lg.rdxy >> r) & 1u) || dzl;
            out(m, dir, nl + from_left, vprev[r - 1], got[r - 1]);
          }
        }
        lev(t);
      }
    }
#pragma unroll
    for (int r = 0; r < NY; ++r) vprev[r] = v[r + 1];
#pragma unroll
    for (int r = 0; r < NF; ++r)
#pragma unroll
      for (int h = 0; h < 2; ++h) Fp[r][h] = F[r][h];
  }
}

struct NoPre {};
template <class T, int SX, int NY, class MC, class Src, class Out, class Lev = NoLev>
__device__ __forceinline__ void warp_tile_march(const LaneGeo<NY>& lg, const MC& mc, Src& src, int tzl, Out&& out,
                                                Lev&& lev = Lev{}) {
  warp_tile_march_pre<T, SX, NY>(lg, mc, src, tzl, [](int, bool) { return NoPre{}; },
                                 [&](int m, bool dir, T y, T v, NoPre) { out(m, dir, y, v); }, lev);
}

// The same contract on six-tetrahedra boxes (heat.h HEAT_ELEM_P1). Each lane
// computes its box column's boxes row by row from the staged levels L-1 and
// L of its own column and of its right neighbour (one shuffle per row), with
// the split's structure instead of an 8x8 matrix:
//  - mass: each tetrahedron t adds V/20 (x_c + s_t) at its corners, s_t the
//    sum of its four values; a box corner c lies in n_c tetrahedra (6 for
//    corners 0 and 7, 2 for the others);
//  - stiffness: sum over the 12 box edges of w_e V/h_a^2 (x_i - x_j)^2, w_e
//    the number of tetrahedra that step along the edge: 2, 1, 1, 2 for the
//    edges of axis a leaving corners 0, the two one-axis corners and the
//    two-axis corner (the path gradients are axis-aligned).
// About 90 operations per box with every weight in registers. A node sums its
// <= 8 boxes' contributions in a fixed order: the upper corners of the layer
// below (carried in registers), then this layer's lower corners, the left
// neighbour's through one shuffle per row.
template <class T>
struct MarchP1 {
  T mw, kwx, kwy, kwz;  // sa V / 20 and sb V / h_a^2, V = hx hy hz / 6
  MarchP1() = default;
  __device__ __forceinline__ MarchP1(const SimDev& s, T sa, T sb)
      : mw(sa * p1_consts<T>(s)[0]),
        kwx(sb * p1_consts<T>(s)[1]),
        kwy(sb * p1_consts<T>(s)[2]),
        kwz(sb * p1_consts<T>(s)[3]) {}
};
template <class T, int SX, int NY, class Src, class Out, class Lev = NoLev>
__device__ __forceinline__ void warp_tile_march_p1(const LaneGeo<NY>& lg, const MarchP1<T>& mc, Src& src, int tzl,
                                                   Out&& out, Lev&& lev = Lev{}) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int NR = NY + 2;  // staged rows
  constexpr int NF = NY + 1;  // box rows
  const T mw = mc.mw, kwx = mc.kwx, kwy = mc.kwy, kwz = mc.kwz;
  src.prologue(lg, tzl);
  T prv[NR], prvR[NR], carry[NY];
#pragma unroll
  for (int r = 0; r < NR; ++r) prv[r] = prvR[r] = T(0);
#pragma unroll
  for (int r = 0; r < NY; ++r) carry[r] = T(0);
  const int k0 = src.k0;
  for (int t = 0; t <= tzl + 1; ++t) {
    const int L = k0 - 1 + t;
    T cur[NR], curR[NR];
    src.level(lg, t, tzl, cur);
#pragma unroll
    for (int r = 0; r < NR; ++r) curR[r] = __shfl_down_sync(FULL, cur[r], 1, SX);
    if (t >= 1) {
      // boxes (lane column, row r, layer L-1): lower corners to level L-1,
      // upper corners to level L; cx = 1 corners belong to the right lane
      T lo0[NF], lo2[NF], lo1[NF], lo3[NF], up4[NF], up6[NF], up5[NF], up7[NF];
#pragma unroll
      for (int r = 0; r < NF; ++r) {
        const auto cf = src.coef_row(t, r);
        const T x0 = prv[r], x1 = prvR[r], x2 = prv[r + 1], x3 = prvR[r + 1];
        const T x4 = cur[r], x5 = curR[r], x6 = cur[r + 1], x7 = curR[r + 1];
        const T s07 = x0 + x7;
        const T t1 = s07 + x1 + x3, t2 = s07 + x1 + x5, t3 = s07 + x2 + x3;
        const T t4 = s07 + x2 + x6, t5 = s07 + x4 + x5, t6 = s07 + x4 + x6;
        const T S6 = ((t1 + t2) + (t3 + t4)) + (t5 + t6);
        const T m = mw * cf.x;
        const T ax = kwx * cf.y, ay = kwy * cf.y, az = kwz * cf.y;
        const T e01 = T(2) * ax * (x0 - x1), e23 = ax * (x2 - x3), e45 = ax * (x4 - x5), e67 = T(2) * ax * (x6 - x7);
        const T e02 = T(2) * ay * (x0 - x2), e13 = ay * (x1 - x3), e46 = ay * (x4 - x6), e57 = T(2) * ay * (x5 - x7);
        const T e04 = T(2) * az * (x0 - x4), e15 = az * (x1 - x5), e26 = az * (x2 - x6), e37 = T(2) * az * (x3 - x7);
        lo0[r] = m * (T(6) * x0 + S6) + e01 + e02 + e04;
        lo1[r] = m * (T(2) * x1 + t1 + t2) - e01 + e13 + e15;
        lo2[r] = m * (T(2) * x2 + t3 + t4) + e23 - e02 + e26;
        lo3[r] = m * (T(2) * x3 + t1 + t3) - e23 - e13 + e37;
        up4[r] = m * (T(2) * x4 + t5 + t6) + e45 + e46 - e04;
        up5[r] = m * (T(2) * x5 + t2 + t5) - e45 + e57 - e15;
        up6[r] = m * (T(2) * x6 + t4 + t6) + e67 - e46 - e26;
        up7[r] = m * (T(6) * x7 + S6) - e67 - e57 - e37;
      }
      src.after_elements(lg, t, tzl);
      const int lv = L - 1;
      const bool lvin = lv <= lg.gnz;
      const bool dzl = (lg.dz0 && lv == 0) || (lg.dz1 && lv == lg.gnz);
#pragma unroll
      for (int r = 1; r <= NY; ++r) {
        // node row r: boxes r (cy = 0) and r - 1 (cy = 1)
        const T from_left_lo = __shfl_up_sync(FULL, lo1[r] + lo3[r - 1], 1, SX);
        const T from_left_up = __shfl_up_sync(FULL, up5[r] + up7[r - 1], 1, SX);
        const T y = ((carry[r - 1] + lo0[r]) + lo2[r - 1]) + from_left_lo;
        carry[r - 1] = (up4[r] + up6[r - 1]) + from_left_up;
        const int m = lg.nbase + r * lg.px + lv * lg.pxy;
        if (t >= 2 && lg.out_lane && lvin && ((lg.rin >> r) & 1u) && HEAT_INDEX_OK(lg.sc, m, lg.nn)) {
          const bool dir = ((lg.rdxy >> r) & 1u) || dzl;
          out(m, dir, y, prv[r]);
        }
      }
      if (t >= 2) lev(t);
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      prv[r] = cur[r];
      prvR[r] = curR[r];
    }
  }
}

// The march of element type E and its constants.
template <int E, class T>
using MarchE = typename std::conditional<E == E_P1, MarchP1<T>, MarchQ1<T>>::type;
template <int E, class T, int SX, int NY, class Src, class Out, class Lev = NoLev>
__device__ __forceinline__ void warp_march_c(const LaneGeo<NY>& lg, const MarchE<E, T>& mc, Src& src, int tzl,
                                             Out&& out, Lev&& lev = Lev{}) {
  if constexpr (E == E_P1)
    warp_tile_march_p1<T, SX, NY>(lg, mc, src, tzl, out, lev);
  else
    warp_tile_march<T, SX, NY>(lg, mc, src, tzl, out, lev);
}
template <int E, class T, int SX, int NY, class Src, class Out, class Lev = NoLev>
__device__ __forceinline__ void warp_march_e(const LaneGeo<NY>& lg, const SimDev& s, Src& src, int tzl, T sa, T sb,
                                             Out&& out, Lev&& lev = Lev{}) {
  warp_march_c<E, T, SX, NY>(lg, MarchE<E, T>(s, sa, sb), src, tzl, out, lev);
}

// The register-prefetch form with functor loads (see RegSrc), for element E.
template <int E, class T, int SX, int NY, class Coef, class Fetch, class Value, class Out, class Lev = NoLev>
__device__ __forceinline__ void warp_tile_op_e(const Geo& g, const SimDev& s, const Coef* __restrict__ coef,
                                               bool active, int i0, int j0, int k0, int tzl, T sa, T sb, bool mask,
                                               Fetch&& fetch, Value&& value, Out&& out, Lev&& lev = Lev{}) {
  const LaneGeo<NY> lg(g, active, (int)threadIdx.x % SX, SX, i0, j0, mask, s.sc);
  using CoefT = typename std::remove_cv<typename std::remove_reference<decltype(coef[0])>::type>::type;
  RegSrc<T, NY, CoefT, typename std::remove_reference<Fetch>::type, typename std::remove_reference<Value>::type> src(
      coef, fetch, value, k0);
  warp_march_e<E, T, SX, NY>(lg, s, src, tzl, sa, sb, out, lev);
}

}  // namespace heat
