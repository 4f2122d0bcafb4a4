// The inner CG solve held on the chip (k_cg_res): one persistent cooperative
// kernel whose blocks keep a simulation's direction, residual and
// coefficients in shared memory from the first iteration of an inner solve to
// its last, instead of two launches per iteration that stream them through L2.
//
// What bounds an iteration of a mesh that fits (FP32: 152 SMs x 227 KB at about
// 28 bytes per node with halos, cubes of up to 103 elements an edge) is not bandwidth: the
// streaming kernels spend it on launch boundaries, on the descriptor and
// scalar loads each block starts with, and on the last block's reduction tail
// (fence, counter, partials, division: each an L2 round trip). Here the mesh
// is cut into boxes, one per block. An iteration (Algorithm 1, §3.3) is
//   q = A d by the warp-segment march from shared memory, dot d.q   -> all-sum
//   x += alpha d, r -= alpha q, z = P^-1 r, dot r.z                 -> all-sum
//   d = z + beta d on the box and on its one-node halo
// and its two all-sums are the only places where blocks wait for each other.
//
// All-sum: every block stores its partial as two 64-bit words, each holding
// 32 bits of the value and a tag (a counter that never repeats), and one warp
// of every block polls all blocks' words until their tags match. A word is
// written by one store, so value and tag arrive together and neither a fence
// nor an atomic is needed; the sum runs in block order, so every block gets
// the same bits and takes the same decision. Halo values travel the same way:
// the owner of a boundary node stores {z, tag} to the node's slot, the
// neighbours poll the slot. A slot is rewritten only after another all-sum,
// which every reader enters after reading it.
//
// Every wait is bounded like the grid barrier's (loop_kernels.cuh): a poll that
// exceeds GridSync::limit_ns sets GridSync::abort and the kernel returns.
//
// The boxes depend on the mesh and the GPU only (engine.cu: res_plan), so a
// simulation's results are the same alone and in a batch; the blocks of one
// launch carry as many simulations side by side as fit, the rest after them.
#pragma once

#include "loop_kernels.cuh"
#include "tile_kernels.cuh"

namespace heat {

using ResFn = void (*)(const SimDev*, const int*, const int2*, GridSync*);

constexpr int kResThreads = 256;
constexpr int kResNY = 4;       // rows per lane of the FP32 march
constexpr int kResCols = 30;    // output columns of a 16-lane segment (2 per lane, the first lane only feeds its neighbour)
constexpr int kResMaxQ = 9;     // FP32: groups of 4 nodes per thread
constexpr int kResMaxN = 4;     // FP64: nodes per thread

// FP32: groups of 4 nodes per thread of a box.
__host__ __device__ inline int res_groups(const ResGeo& r) {
  return (((r.bx + 3) / 4) * r.by * r.bz + kResThreads - 1) / kResThreads;
}

// Shared-memory layout of a box of bx x by x bz nodes.
//   FP32: direction d with its halo, coefficients (rho_c part, k part), q, r,
//   and per group of 4 nodes where it lies in d.
//   FP64: d with its halo, 27 row coefficients per node.
// Both: a row table and the halo rows' table.
struct ResLayout {
  int nseg, nyt;   // FP32 march: segments in x, row groups in y
  int pd, dr, dl;  // d: row pitch, rows, levels (own node i at 4 + i)
  int pc, er, el;  // coefficients: row pitch, element rows, layers (element e at e + 2)
  int pw;          // own values: row pitch
  int off_c, off_q, off_r, off_at, off_row, off_halo, bytes;
};
__host__ __device__ inline ResLayout res_layout(const ResGeo& g, bool fp64) {
  ResLayout l;
  auto up = [](int b) { return (b + 15) & ~15; };
  const int nodes = g.bx * g.by * g.bz;
  l.pw = (g.bx + 3) & ~3;
  l.dl = g.bz + 2;
  int o;
  if (fp64) {
    l.nseg = l.nyt = l.pc = l.er = l.el = 0;
    l.pd = g.bx + 2;
    l.dr = g.by + 2;
    o = up(l.pd * l.dr * l.dl * 8);
    l.off_c = o;
    o += up(27 * 8 * nodes);
    l.off_q = l.off_r = l.off_at = o;
  } else {
    l.nseg = (g.bx + kResCols - 1) / kResCols;
    l.nyt = (g.by + kResNY - 1) / kResNY;
    l.pd = (kResCols * l.nseg + 8) & ~3;
    if (l.pd < l.pw + 8) l.pd = l.pw + 8;
    l.dr = l.nyt * kResNY + 2;
    l.pc = kResCols * l.nseg + 2;
    l.er = l.nyt * kResNY + 1;
    l.el = g.bz + 1;
    o = up(l.pd * l.dr * l.dl * 4);
    l.off_c = o;
    o += up(l.pc * l.er * l.el * 8);
    l.off_q = o;
    o += l.pw * g.by * g.bz * 4;
    l.off_r = o;
    o += l.pw * g.by * g.bz * 4;
    l.off_at = o;
    o += up(l.pw * g.by * g.bz);
  }
  l.off_row = o;
  o += 16 * g.by * g.bz;
  l.off_halo = o;
  o += 8 * (2 * (g.by + 2) + 2 * g.bz);
  l.bytes = up(o);
  return l;
}

// n / d by one multiplication, exact for the small n of a box (n d < 2^32);
// d = 1 has no 32-bit factor and is marked by 0.
__device__ __forceinline__ unsigned int div_magic(int d) { return d > 1 ? 0xffffffffu / (unsigned int)d + 1u : 0u; }
__device__ __forceinline__ int fast_div(int n, unsigned int m) { return m ? (int)__umulhi((unsigned int)n, m) : n; }

// ---------------------------------------------------------- tagged words

__device__ __forceinline__ unsigned long long ld_word(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void ld_word2(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_word2(unsigned long long* p, unsigned long long a, unsigned long long b) {
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ unsigned long long tagged(unsigned int v, unsigned int tag) {
  return (unsigned long long)v | ((unsigned long long)tag << 32);
}

// A bounded wait: call after a failed poll; true when the wait is over its
// limit (or another block's is) and the caller has to give up.
struct Patience {
  unsigned int polls = 0;
  unsigned long long t0 = 0;
  __device__ __forceinline__ bool over(GridSync* gs) {
    if ((++polls & 127u) != 0u) return false;
    if (ld_acquire_gpu(reinterpret_cast<const unsigned int*>(&gs->abort)) != 0u) return true;
    const unsigned long long t = global_ns();
    if (t0 == 0) t0 = t;
    if (t - t0 > gs->limit_ns) {
      atomicExch(&gs->abort, 1);
      return true;
    }
    return false;
  }
};

// One node's exchanged value: {value, tag} in 8 bytes (float), the two halves
// with a tag each in 16 (double).
template <class T> struct Exch;
template <> struct Exch<float> {
  static constexpr int words = 1;
  struct Raw { unsigned long long a; };
  static __device__ __forceinline__ Raw load(const unsigned long long* p) { return {ld_word(p)}; }
  static __device__ __forceinline__ bool ready(const Raw& r, unsigned int tag) { return (unsigned int)(r.a >> 32) == tag; }
  static __device__ __forceinline__ float value(const Raw& r) { return __uint_as_float((unsigned int)r.a); }
  static __device__ __forceinline__ void store4(unsigned long long* p, float2 a, float2 b, unsigned int tag) {
    st_word2(p, tagged(__float_as_uint(a.x), tag), tagged(__float_as_uint(a.y), tag));
    st_word2(p + 2, tagged(__float_as_uint(b.x), tag), tagged(__float_as_uint(b.y), tag));
  }
};
template <> struct Exch<double> {
  static constexpr int words = 2;
  struct Raw { unsigned long long a, b; };
  static __device__ __forceinline__ Raw load(const unsigned long long* p) {
    Raw r;
    ld_word2(p, r.a, r.b);
    return r;
  }
  static __device__ __forceinline__ bool ready(const Raw& r, unsigned int tag) {
    return (unsigned int)(r.a >> 32) == tag && (unsigned int)(r.b >> 32) == tag;
  }
  static __device__ __forceinline__ double value(const Raw& r) {
    return __hiloint2double((int)(unsigned int)r.b, (int)(unsigned int)r.a);
  }
  static __device__ __forceinline__ void store(unsigned long long* p, double v, unsigned int tag) {
    st_word2(p, tagged((unsigned int)__double2loint(v), tag), tagged((unsigned int)__double2hiint(v), tag));
  }
};

// ------------------------------------------------------------- all-sums

// The sums' arithmetic: FP64 on the FP64 path; on the FP32 path the warps'
// FP32 sums are added in double-float (48 bits; FP64 adds on this GPU take 64
// cycles of a scheduler each, and these chains are on the critical path: 960
// cycles a sum within a block against 1,900, a time step on 100^3 3.3% and one on
// 80^3 4.7% slower with them). FP32's range would be lost with its width, so
// the partials are scaled by the power of two nearest 1 / delta as the solve
// is taken up (exact; r.z and d.q stay within a few powers of ten of delta).
// The FP32 parts are no longer than the streaming kernels': r.z has two
// partials a warp, of at most 10 + 6 additions in a row over 576 nodes (k_update:
// 16 + 5 over 512). Relative error of r.z over a million random nodes, root mean
// square: 0.9e-9 in k_update's order, 0.8e-9 in this one, 1.3e-9 with one partial
// a warp; the double-float additions after it were exact.
__device__ __forceinline__ DF res_xor(const DF& v, int o) {
  return DF(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}
__device__ __forceinline__ double res_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ void res_split(const DF& v, unsigned int& a, unsigned int& b) {
  a = __float_as_uint(v.hi);
  b = __float_as_uint(v.lo);
}
__device__ __forceinline__ void res_split(double v, unsigned int& a, unsigned int& b) {
  a = (unsigned int)__double2loint(v);
  b = (unsigned int)__double2hiint(v);
}
template <class S> __device__ __forceinline__ S res_join(unsigned int a, unsigned int b);
template <> __device__ __forceinline__ DF res_join<DF>(unsigned int a, unsigned int b) {
  return DF(__uint_as_float(a), __uint_as_float(b));
}
template <> __device__ __forceinline__ double res_join<double>(unsigned int a, unsigned int b) {
  return __hiloint2double((int)b, (int)a);
}
__device__ __forceinline__ DF res_from(float v, DF) { return DF(v, 0.f); }
__device__ __forceinline__ DF res_from(double v, DF) { return DF(v); }
__device__ __forceinline__ double res_from(double v, double) { return v; }
__device__ __forceinline__ bool res_finite(const DF& v) { return isfinite(v.hi); }
__device__ __forceinline__ bool res_finite(double v) { return isfinite(v); }
__device__ __forceinline__ bool res_positive(const DF& v) { return v.hi > 0.f; }
__device__ __forceinline__ bool res_positive(double v) { return v > 0.0; }
// v as it is kept between launches (SimScalars, FP64): where a launch ends does not show
__device__ __forceinline__ DF res_kept(const DF& v) { return DF(v.to_double()); }
// v <= t: the double-float form decides in FP32 unless the two are close
__device__ __forceinline__ bool res_below(const DF& v, double t, float tf) {
  if (tf > 1e-30f && (v.hi > 1.001f * tf || v.hi < 0.999f * tf)) return v.hi < tf;
  return v.to_double() <= t;
}
__device__ __forceinline__ bool res_below(double v, double t, float) { return v <= t; }
// a / b: correctly rounded quotient of the leading parts, one correction step
__device__ __forceinline__ float res_div(const DF& a, const DF& b) {
  const float q = __fdiv_rn(a.hi, b.hi);
  const float r = fmaf(-q, b.hi, a.hi) + (a.lo - q * b.lo);
  return q + __fdividef(r, b.hi);
}
__device__ __forceinline__ double res_div(double a, double b) { return a / b; }

// Mailboxes of one all-sum: block r reads its own g + 1 entries at r (g + 1)
// (the last entry is waited for by the wait test only).
__host__ __device__ __forceinline__ int res_mail(int g) { return g * (g + 1); }

// All-sum of one value per block over the simulation's g blocks: every lane of
// warp 0 calls it with the block's sum and gets the total. Every block writes
// its value into every block's mailbox and polls only its own: with one list
// that all blocks poll, the polls queue up at the L2 slices that hold it (144
// blocks: 6,600 cycles an all-sum, against 1,900 with 12 blocks).
template <class S>
__device__ __forceinline__ bool res_all_sum(const S& v, ulonglong2* mail, int g, int rank, unsigned int tag,
                                            GridSync* gs, S& total) {
  const int lane = (int)threadIdx.x & 31;
  unsigned int va, vb;
  res_split(v, va, vb);
  const unsigned long long wa = tagged(va, tag), wb = tagged(vb, tag);
  for (int u = lane; u < g; u += 32) st_word2(reinterpret_cast<unsigned long long*>(mail + u * (g + 1) + rank), wa, wb);
  // A few stores linger on their way for about 4,000 cycles unless something
  // pushes them: with one store instruction or two a fence is cheaper (21
  // blocks: 21,100 -> 18,400 cycles an iteration), with more it only costs
  // (144 blocks: 26,000 -> 27,100).
  if (g <= 48) __threadfence();
  const unsigned long long* w = reinterpret_cast<const unsigned long long*>(mail + rank * (g + 1));
  const int n = g + (int)gs->extra;
  S t = S(0);
  bool ok = true;
  Patience wait;
  constexpr int B = 5;  // entries of one lane in flight (5 x 32 >= 152 SMs)
  for (int u0 = lane; u0 < n && ok; u0 += 32 * B) {
    unsigned long long a[B], b[B];
    unsigned int missing = 0;
#pragma unroll
    for (int k = 0; k < B; ++k) {
      a[k] = b[k] = 0;
      if (u0 + 32 * k < n) missing |= 1u << k;
    }
    while (true) {
#pragma unroll
      for (int k = 0; k < B; ++k)
        if ((missing >> k) & 1u) ld_word2(w + 2 * (u0 + 32 * k), a[k], b[k]);
#pragma unroll
      for (int k = 0; k < B; ++k)
        if ((unsigned int)(a[k] >> 32) == tag && (unsigned int)(b[k] >> 32) == tag) missing &= ~(1u << k);
      if (!missing) break;
      if (wait.over(gs)) {
        ok = false;
        break;
      }
    }
#pragma unroll
    for (int k = 0; k < B; ++k)
      if (u0 + 32 * k < g) t = t + res_join<S>((unsigned int)a[k], (unsigned int)b[k]);
  }
  ok = __all_sync(0xffffffffu, ok);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t = t + res_xor(t, o);
  total = t;
  return ok;
}

// ------------------------------------------------------------ the block's task

// Block-wide state of the running task (S: DF or double).
template <class T, class S>
struct ResShared {
  T wsum[2 * kResThreads / 32];
  S delta, dq;      // in units of unit
  T alpha, beta;
  double thresh;    // in units of unit
  float thresh_f;
  T scale;          // 1 / unit
  double unit;      // a power of two: FP32 of delta's size, FP64 1
  int go;  // what the next phase does: kGo, or how the task ends
  int iter, iter_step;
  unsigned int tag0;
};
enum : int { kGo = 0, kEndIter = 1, kEndOuter = 2, kEndResid = 3, kEndConfirm = 4, kEndFailed = 5, kEndAbort = 6 };

// The box of one block: own nodes, neighbours, tables.
struct ResBox {
  int x0, y0, z0, nx, ny, nz;  // own nodes
  int X, Y, Z, pz;             // nodes of the mesh, row pitch of the exchanged values
  int rows, nhr, span;         // own rows, halo rows, cells of a halo row inside the mesh
  unsigned int hdiv;           // fast_div factor of span
  bool xl, xr;                 // a neighbour before / behind in x

  ResBox() = default;
  __device__ __forceinline__ ResBox(const SimDev& s, int rank) {
    const ResGeo& rg = s.res;
    X = s.nx + 1;
    Y = s.ny + 1;
    Z = s.nz + 1;
    x0 = (rank % rg.gx) * rg.bx;
    y0 = (rank / rg.gx % rg.gy) * rg.by;
    z0 = (rank / (rg.gx * rg.gy)) * rg.bz;
    nx = min(rg.bx, X - x0);
    ny = min(rg.by, Y - y0);
    nz = min(rg.bz, Z - z0);
    pz = (X + 3) & ~3;
    xl = x0 > 0;
    xr = x0 + nx < X;
    span = nx + (xl ? 1 : 0) + (xr ? 1 : 0);
    hdiv = div_magic(span);
    rows = ny * nz;
    nhr = nj() * (klo() + khi()) + nz * ((y0 > 0) + (y0 + ny < Y));
  }
  __device__ __forceinline__ int klo() const { return z0 > 0; }
  __device__ __forceinline__ int khi() const { return z0 + nz < Z; }
  __device__ __forceinline__ int jlo() const { return y0 > 0 ? -1 : 0; }
  __device__ __forceinline__ int nj() const { return (y0 + ny < Y ? ny : ny - 1) - jlo() + 1; }
  // own row t: offset of its node 0 in d, in the exchanged values, in the
  // node vectors, and whether a neighbour needs the whole row. halo row t (the
  // levels below and above, then the rows before and behind): offsets of its
  // first cell in d and in the exchanged values.
  __device__ __forceinline__ void tables(const ResLayout& l, int d0, int4* srow, int2* shalo) const {
    for (int t = threadIdx.x; t < rows; t += blockDim.x) {
      const int k = t / ny, j = t - k * ny;
      const bool pub = (k == 0 && klo()) || (k == nz - 1 && khi()) || (j == 0 && y0 > 0) || (j == ny - 1 && y0 + ny < Y);
      srow[t] = make_int4(((k + 1) * l.dr + j + 1) * l.pd + d0, ((z0 + k) * Y + y0 + j) * pz + x0,
                          x0 + X * (y0 + j) + X * Y * (z0 + k), pub ? 1 : 0);
    }
    const int n = nj();
    for (int t = threadIdx.x; t < nhr; t += blockDim.x) {
      int j, k, u = t;
      if (u < n * (klo() + khi())) {
        k = (u < n && klo()) ? -1 : nz;
        j = jlo() + u % n;
      } else {
        u -= n * (klo() + khi());
        k = u % nz;
        j = (u < nz && y0 > 0) ? -1 : ny;
      }
      const int i = xl ? -1 : 0;
      shalo[t] = make_int2(((k + 1) * l.dr + j + 1) * l.pd + d0 + i, ((z0 + k) * Y + y0 + j) * pz + x0 + i);
    }
  }
};

// z = P^-1 r and d = z + beta d_old, each rounded once: the iteration's own
// arithmetic, so a solve taken up by the next launch goes on bit for bit.
__device__ __forceinline__ float res_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double res_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float res_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double res_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// d on the box and its halo from the node vectors: P^-1 r + beta d_old
// (restart: P^-1 r), zero outside the mesh. own node i of a row at d0 + i.
template <class T>
__device__ __forceinline__ void res_load_d(const SimDev& s, const Ctl& c, const ResBox& b, const ResLayout& l, int d0,
                                           T* sd) {
  const bool rs = c.restart != 0;
  const T beta = rs ? T(0) : (T)c.beta;
  const T* __restrict__ r = IterVecs<T>::r(s);
  const T* __restrict__ pinv = IterVecs<T>::pinv(s);
  const T* __restrict__ dold = IterVecs<T>::d(s, c.id);
  const int lane = (int)threadIdx.x & 31, nw = (int)blockDim.x >> 5;
  for (int row = (int)threadIdx.x >> 5; row < l.dr * l.dl; row += nw) {
    const int k = row / l.dr - 1, j = row - (k + 1) * l.dr - 1;
    const bool in = k <= b.nz && j <= b.ny && b.z0 + k >= 0 && b.z0 + k < b.Z && b.y0 + j >= 0 && b.y0 + j < b.Y;
    const int m0 = b.x0 + b.X * (b.y0 + j) + b.X * b.Y * (b.z0 + k);
    for (int t = lane; t < l.pd; t += 32) {
      const int i = t - d0;
      T v = T(0);
      if (in && i >= -1 && i <= b.nx && b.x0 + i >= 0 && b.x0 + i < b.X && HEAT_INDEX_OK(s.sc, m0 + i, s.nn))
        v = res_fma(beta, rs ? T(0) : dold[m0 + i], res_mul(pinv[m0 + i], r[m0 + i]));
      sd[row * l.pd + t] = v;
    }
  }
}

// Halo cells of the box inside the mesh: the halo rows' cells, then the columns
// before and behind the own rows. where(h): offset in d, in the exchanged values.
__device__ __forceinline__ int res_halo_cells(const ResBox& b) {
  return b.nhr * b.span + b.rows * ((b.xl ? 1 : 0) + (b.xr ? 1 : 0));
}
__device__ __forceinline__ int2 res_halo_at(const ResBox& b, const int4* srow, const int2* shalo, int h) {
  const int n = b.nhr * b.span;
  if (h < n) {
    const int row = fast_div(h, b.hdiv), i = h - row * b.span;
    const int2 t = shalo[row];
    return make_int2(t.x + i, t.y + i);
  }
  h -= n;
  const int4 t = srow[h < b.rows ? h : h - b.rows];
  const int i = (b.xl && h < b.rows) ? -1 : b.nx;
  return make_int2(t.x + i, t.y + i);
}

// The neighbours' z of up to HB halo cells h0, h0 + step, ...: fetched by the
// warps that do not run the second all-sum, while it runs (z does not depend
// on beta). False when a wait ran out.
template <class T, int HB>
__device__ __forceinline__ bool res_halo_fetch(const ResBox& b, const int4* srow, const int2* shalo, int h0, int step,
                                               const unsigned long long* zx, unsigned int tag, GridSync* gs,
                                               T (&z)[HB], int (&at)[HB]) {
  using X = Exch<T>;
  const int n = res_halo_cells(b);
  int zo[HB];
  unsigned int missing = 0;
#pragma unroll
  for (int u = 0; u < HB; ++u) {
    at[u] = -1;
    zo[u] = 0;
    const int h = h0 + u * step;
    if (h < n) {
      const int2 p = res_halo_at(b, srow, shalo, h);
      at[u] = p.x;
      zo[u] = X::words * p.y;
      missing |= 1u << u;
    }
  }
  Patience wait;
  while (missing) {  // all that is missing in flight together
    typename X::Raw w[HB];
#pragma unroll
    for (int u = 0; u < HB; ++u)
      if ((missing >> u) & 1u) w[u] = X::load(zx + zo[u]);
#pragma unroll
    for (int u = 0; u < HB; ++u)
      if (((missing >> u) & 1u) && X::ready(w[u], tag)) {
        z[u] = X::value(w[u]);
        missing &= ~(1u << u);
      }
    if (missing && wait.over(gs)) return false;
  }
  return true;
}

// Sum of the warps' NP partials over the block, in every lane of warp 0.
template <class T, class S, int NP>
__device__ __forceinline__ S res_block_sum(const T* wsum) {
  const int lane = (int)threadIdx.x & 31;
  static_assert(NP == 8 || NP == 16, "every group of NP lanes sums the same partials");
  S v = res_from(wsum[lane & (NP - 1)], S(0));
#pragma unroll
  for (int o = NP / 2; o > 0; o >>= 1) v = v + res_xor(v, o);
  return v;
}

// After the first all-sum (warp 0, lane 0): alpha = delta / d.q, or the task fails.
template <class T, class S>
__device__ __forceinline__ void res_decide_alpha(ResShared<T, S>& sh, bool ok, const S& dq) {
  sh.dq = dq;
  if (!ok) {
    sh.go = kEndAbort;
  } else if (res_finite(dq) && res_positive(dq)) {
    sh.go = kGo;
    sh.alpha = res_div(sh.delta, dq);
  } else {
    sh.go = kEndFailed;
  }
}

// After the second (warp 0, lane 0): beta and the tests of k_update
// (Algorithm 1's rule on r^T P^-1 r).
template <class T, class S>
__device__ __forceinline__ void res_decide_beta(ResShared<T, S>& sh, const SimDev& s, bool ok, const S& dn,
                                                bool resid_it, bool last_round) {
  constexpr bool F64 = sizeof(T) == 8;
  int e = kGo;
  if (!ok) {
    e = kEndAbort;
  } else if (resid_it) {
    e = kEndResid;
  } else {
    sh.beta = res_div(dn, sh.delta);
    sh.delta = dn;
    sh.iter += 1;
    sh.iter_step += 1;
    if (!res_finite(dn)) {
      e = kEndFailed;
    } else if (F64) {
      if (res_below(dn, sh.thresh, sh.thresh_f)) e = kEndConfirm;
      else if (sh.iter_step >= s.max_iter) e = kEndFailed;
    } else {
      const int cap = s.prec == P_FP32_PLAIN ? s.max_iter : s.inner_max_iter;
      if (sh.iter_step >= s.max_iter) e = kEndFailed;
      else if (sh.iter >= cap || res_below(dn, sh.thresh, sh.thresh_f)) e = kEndOuter;
    }
    if (e == kGo && last_round) e = kEndIter;
  }
  sh.go = e;
}

// The end of a task: the simulation's scalars (one thread).
template <class T, class S>
__device__ __forceinline__ void res_finish(const SimDev& s, const ResShared<T, S>& sh, int go, bool after_alpha,
                                           unsigned int tag) {
  SimScalars* sc = s.sc;
  sc->dq = to_d(sh.dq) * sh.unit;
  if (!after_alpha) {
    fail(sc, res_finite(sh.dq) ? ST_BREAKDOWN : ST_NONFINITE);
  } else {
    sc->alpha = (double)sh.alpha;
    sc->restart = 0;
    sc->iter = sh.iter;
    sc->iter_step = sh.iter_step;
    sc->delta = to_d(sh.delta) * sh.unit;
    if (go != kEndResid) sc->beta = (double)sh.beta;
    if (go == kEndFailed) fail(sc, res_finite(sh.delta) ? ST_NOT_CONVERGED : ST_NONFINITE);
    else if (go == kEndOuter) sc->phase = PH_OUTER;
    else if (go == kEndResid) sc->phase = PH_RESID;
    else if (go == kEndConfirm) {
      sc->confirm = 1;
      sc->phase = PH_RESID;
    }
  }
  *s.res_tag = tag;
}

// Makes task's simulation current in shared memory; false: not in PH_ITER.
template <class T, class S>
__device__ __forceinline__ bool res_open_task(const SimDev* __restrict__ sims, int sim, SimDev& s, Ctl& c,
                                              ResShared<T, S>& sh) {
  const int tid = (int)threadIdx.x;
  __syncthreads();  // the previous task's users of the shared state are done
  if (tid < 32) {
    const uint4* src = reinterpret_cast<const uint4*>(&sims[sim]);
    uint4* dst = reinterpret_cast<uint4*>(&s);
    for (int t = tid; t < (int)(sizeof(SimDev) / sizeof(uint4)); t += 32) dst[t] = src[t];
    __syncwarp();
    if (tid == 0) c = load_ctl(s.sc);
  }
  __syncthreads();
  if (c.phase != PH_ITER) return false;
  if (tid == 0) {
    const double delta = __ldcg(&s.sc->delta);
    double inv = 1.0;
    if (sizeof(T) == 4) {  // within what its reciprocal has as a normal float
      const int e = min(max(((__double2hiint(delta) >> 20) & 0x7ff) - 1023, -120), 120);
      inv = __hiloint2double((1023 - e) << 20, 0);
      sh.unit = __hiloint2double((1023 + e) << 20, 0);
    } else {
      sh.unit = 1.0;
    }
    sh.scale = (T)inv;
    sh.delta = res_from(delta * inv, S(0));
    sh.thresh = (sizeof(T) == 8 ? __ldcg(&s.sc->thresh) : __ldcg(&s.sc->thresh_in)) * inv;
    sh.thresh_f = (float)sh.thresh;
    sh.iter_step = __ldcg(&s.sc->iter_step);
    sh.iter = c.iter;
    sh.tag0 = __ldcg(s.res_tag);
    sh.go = kGo;
    sh.dq = S(0);
  }
  return true;
}

// ------------------------------------------------------------- the FP32 march

// One warp's tile of the operator from shared memory: 16-lane segments, two
// adjacent columns per lane in packed FP32x2 arithmetic, kResNY rows, tzl
// levels; everything outside the mesh is stored as zero, so no load is
// predicated. Against the streaming march (op_warp.cuh: one column per lane,
// loads from L2, 120 instructions per node) this one takes about 35.
struct ResTile {
  const float* d;             // the lane's first column in row 0 of the level below the tile
  const float *ca, *cb;       // its first element in row 0 of the layer below (rho_c part, k part)
  float* q;                   // its first column's output in (row 1, first level)
  int drow, dlev, crow, clev, qrow, qlev;
  unsigned int mc0, mc1;      // all ones: the column is an own free node's
  unsigned int mr[kResNY];    // the same by row
  unsigned int rows;          // bit r - 1: the lane stores row r (own row, own columns)
  int lev0, zlo, zhi;         // first level; Dirichlet levels (or -1)
};

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 mask2(float2 v, unsigned int a, unsigned int b) {
  return f2(__uint_as_float(__float_as_uint(v.x) & a), __uint_as_float(__float_as_uint(v.y) & b));
}

// Row r's result y (summed over its elements) masked to the own free nodes,
// and its part of the dot with the row's own values v; res_out also stores it.
__device__ __forceinline__ void res_mask(const ResTile& t, int r, float2& y, float2 v, unsigned int m0, unsigned int m1,
                                         float2& acc) {
  y = mask2(y, m0 & t.mr[r - 1], m1 & t.mr[r - 1]);
  acc = __ffma2_rn(v, y, acc);
}
__device__ __forceinline__ void res_out(const ResTile& t, int r, float2 y, float2 v, unsigned int m0, unsigned int m1,
                                        float* q, float2& acc) {
  y = mask2(y, m0 & t.mr[r - 1], m1 & t.mr[r - 1]);
  acc = __ffma2_rn(v, y, acc);
  if ((t.rows >> (r - 1)) & 1u) *reinterpret_cast<float2*>(q + (r - 1) * t.qrow) = y;
}

// Trilinear boxes, in the form of MarchQ1T<T, true> (op_warp.cuh): A_q = R + k al_q,
// B_q = R / 2 + k be_q, 4.5 packed operations per element instead of the 8 of
// march_coeffs. R is formed once, when the block loads its coefficients.
struct ResQ1 {
  float al[4], be[4];
  float ra, ka;  // the rho_c part is ra rho_c, the k part ka k
  __device__ __forceinline__ void set(const SimDev& s) {
    for (int q = 0; q < 4; ++q) {
      al[q] = (float)(s.tal[q] * s.theta);
      be[q] = (float)(s.tbe[q] * s.theta);
    }
    ra = (float)(s.m43 * s.inv_dt);
    ka = 1.f;
  }
};
__device__ __forceinline__ float2 res_march(const ResTile& t, const ResQ1& mc, int tzl) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int NY = kResNY, NF = NY + 1;
  const float2 M1 = f2(-1.f, -1.f), TH = f2(1.f / 3.f, 1.f / 3.f), MTH = f2(-1.f / 3.f, -1.f / 3.f);
  float2 al[4], be[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    al[q] = f2(mc.al[q], mc.al[q]);
    be[q] = f2(mc.be[q], mc.be[q]);
  }
  float2 Fp[NF][4], Tp[NF][4], vp[NY];
  // a row's x edges: sums and differences of its two column pairs
  auto edges = [&](const float* p, float2& v, float2& S, float2& D) {
    v = *reinterpret_cast<const float2*>(p);
    const float2 w = f2(v.y, p[2]);
    S = __fadd2_rn(v, w);
    D = __ffma2_rn(w, M1, v);
  };
  auto faces = [&](float2 S0, float2 D0, float2 S1, float2 D1, float2 (&F)[4]) {
    F[0] = __fadd2_rn(S0, S1);
    F[1] = __fadd2_rn(D0, D1);
    F[2] = __ffma2_rn(S1, M1, S0);
    F[3] = __ffma2_rn(D1, M1, D0);
  };
  const float* d = t.d;
  {
    float2 v, S0, D0;
    edges(d, v, S0, D0);
#pragma unroll
    for (int r = 0; r < NF; ++r) {
      float2 S1, D1;
      edges(d + (r + 1) * t.drow, v, S1, D1);
      faces(S0, D0, S1, D1, Fp[r]);
#pragma unroll
      for (int q = 0; q < 4; ++q) Tp[r][q] = f2(0.f, 0.f);
      if (r < NY) vp[r] = v;
      S0 = S1;
      D0 = D1;
    }
  }
  float2 acc = f2(0.f, 0.f);
  const float *ca = t.ca, *cb = t.cb;
  float* q = t.q;
  // elements between levels lev0 + lev - 1 and lev0 + lev; the first layer
  // only feeds the second (no level is complete)
  auto layer = [&](int lev, auto first) {
    constexpr bool FIRST = decltype(first)::value;
    d += t.dlev;
    const int lv = t.lev0 + lev - 1;  // the level this layer completes
    const unsigned int ml = (lv == t.zlo || lv == t.zhi) ? 0u : 0xffffffffu;
    const unsigned int m0 = t.mc0 & ml, m1 = t.mc1 & ml;
    float2 vr, v, S0, D0, up0 = f2(0.f, 0.f), up1 = f2(0.f, 0.f), y[NY];  // vr: row r's own values
    edges(d, vr, S0, D0);
#pragma unroll
    for (int r = 0; r < NF; ++r) {
      float2 S1, D1, F[4], G[4];
      edges(d + (r + 1) * t.drow, v, S1, D1);
      faces(S0, D0, S1, D1, F);
      const float2 R = *reinterpret_cast<const float2*>(ca + r * t.crow);
      const float2 K = *reinterpret_cast<const float2*>(cb + r * t.crow);
      const float2 H = __fmul2_rn(R, f2(0.5f, 0.5f));
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float2 A = __ffma2_rn(K, al[k], R), B = __ffma2_rn(K, be[k], H);
        if (!FIRST) G[k] = __ffma2_rn(B, F[k], __ffma2_rn(A, Fp[r][k], Tp[r][k]));
        Tp[r][k] = __ffma2_rn(A, F[k], __fmul2_rn(B, Fp[r][k]));
        Fp[r][k] = F[k];
      }
      if (!FIRST) {
        if (r >= 1) {
          const float2 g0 = __fadd2_rn(__ffma2_rn(G[2], TH, G[0]), up0), g1 = __fadd2_rn(__ffma2_rn(G[3], TH, G[1]), up1);
          const float2 nl = __ffma2_rn(g1, TH, g0), nr = __ffma2_rn(g1, MTH, g0);
          const float left = __shfl_up_sync(FULL, nr.y, 1, 16);
          y[r - 1] = f2(nl.x + left, nl.y + nr.x);
        }
        up0 = __ffma2_rn(G[2], MTH, G[0]);
        up1 = __ffma2_rn(G[3], MTH, G[1]);
      }
      if (r < NY) {
        S0 = S1;
        D0 = D1;
      }
      if (r >= 1) {
        if (!FIRST) res_mask(t, r, y[r - 1], vp[r - 1], m0, m1, acc);
        vp[r - 1] = vr;
      }
      vr = v;
    }
    if (!FIRST) {
#pragma unroll
      for (int r = 0; r < NY; ++r)
        if ((t.rows >> r) & 1u) *reinterpret_cast<float2*>(q + r * t.qrow) = y[r];
      q += t.qlev;
    }
    ca += t.clev;
    cb += t.clev;
  };
  layer(0, std::true_type{});
  for (int lev = 1; lev <= tzl; ++lev) layer(lev, std::false_type{});
  return acc;
}

// Six-tetrahedra boxes: warp_tile_march_p1's form (op_warp.cuh) on column
// pairs; the rho_c part is V / 20 sa rho_c, the k part sb k.
struct ResP1 {
  float kx, ky, kz;
  float ra, ka;
  __device__ __forceinline__ void set(const SimDev& s) {
    kx = (float)s.p1c[1];
    ky = (float)s.p1c[2];
    kz = (float)s.p1c[3];
    ra = (float)(s.inv_dt * s.p1c[0]);
    ka = (float)s.theta;
  }
};
__device__ __forceinline__ float2 res_march(const ResTile& t, const ResP1& mc, int tzl) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int NY = kResNY, NR = NY + 2, NF = NY + 1;
  const float2 M1 = f2(-1.f, -1.f), TWO = f2(2.f, 2.f), SIX = f2(6.f, 6.f);
  const float2 kx = f2(mc.kx, mc.kx), ky = f2(mc.ky, mc.ky), kz = f2(mc.kz, mc.kz);
  auto sub = [&](float2 a, float2 b) { return __ffma2_rn(b, M1, a); };
  auto shifted = [](float2 v, float r) { return f2(v.y, r); };
  float2 prv[NR], carry[NY];
  float prr[NR];
  const float* d = t.d;
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    prv[r] = *reinterpret_cast<const float2*>(d + r * t.drow);
    prr[r] = d[r * t.drow + 2];
  }
#pragma unroll
  for (int r = 0; r < NY; ++r) carry[r] = f2(0.f, 0.f);
  float2 acc = f2(0.f, 0.f);
  const float *ca = t.ca, *cb = t.cb;
  float* q = t.q - t.qlev;
  for (int lev = 0; lev <= tzl; ++lev) {
    d += t.dlev;
    const int lv = t.lev0 + lev - 1;
    const unsigned int ml = (lv == t.zlo || lv == t.zhi) ? 0u : 0xffffffffu;
    const unsigned int m0 = t.mc0 & ml, m1 = t.mc1 & ml;
    float2 cur = *reinterpret_cast<const float2*>(d);
    float cuR = d[2];
    float2 lo2 = f2(0.f, 0.f), lo3 = lo2, up6 = lo2, up7 = lo2;  // of the box row below
#pragma unroll
    for (int r = 0; r < NF; ++r) {
      const float2 nxt = *reinterpret_cast<const float2*>(d + (r + 1) * t.drow);
      const float nxR = d[(r + 1) * t.drow + 2];
      const float2 x0 = prv[r], x1 = shifted(prv[r], prr[r]), x2 = prv[r + 1], x3 = shifted(prv[r + 1], prr[r + 1]);
      const float2 x4 = cur, x5 = shifted(cur, cuR), x6 = nxt, x7 = shifted(nxt, nxR);
      const float2 m = *reinterpret_cast<const float2*>(ca + r * t.crow);
      const float2 K = *reinterpret_cast<const float2*>(cb + r * t.crow);
      const float2 s07 = __fadd2_rn(x0, x7);
      const float2 a1 = __fadd2_rn(s07, x1), a2 = __fadd2_rn(s07, x2), a4 = __fadd2_rn(s07, x4);
      const float2 t1 = __fadd2_rn(a1, x3), t2 = __fadd2_rn(a1, x5), t3 = __fadd2_rn(a2, x3);
      const float2 t4 = __fadd2_rn(a2, x6), t5 = __fadd2_rn(a4, x5), t6 = __fadd2_rn(a4, x6);
      const float2 u12 = __fadd2_rn(t1, t2), u34 = __fadd2_rn(t3, t4), u56 = __fadd2_rn(t5, t6);
      const float2 S6 = __fadd2_rn(__fadd2_rn(u12, u34), u56);
      const float2 ax = __fmul2_rn(kx, K), ay = __fmul2_rn(ky, K), az = __fmul2_rn(kz, K);
      const float2 ax2 = __fadd2_rn(ax, ax), ay2 = __fadd2_rn(ay, ay), az2 = __fadd2_rn(az, az);
      // edge terms w_e V / h_a^2 (x_i - x_j)
      const float2 e01 = __fmul2_rn(ax2, sub(x0, x1)), e23 = __fmul2_rn(ax, sub(x2, x3));
      const float2 e45 = __fmul2_rn(ax, sub(x4, x5)), e67 = __fmul2_rn(ax2, sub(x6, x7));
      const float2 e02 = __fmul2_rn(ay2, sub(x0, x2)), e13 = __fmul2_rn(ay, sub(x1, x3));
      const float2 e46 = __fmul2_rn(ay, sub(x4, x6)), e57 = __fmul2_rn(ay2, sub(x5, x7));
      const float2 e04 = __fmul2_rn(az2, sub(x0, x4)), e15 = __fmul2_rn(az, sub(x1, x5));
      const float2 e26 = __fmul2_rn(az, sub(x2, x6)), e37 = __fmul2_rn(az2, sub(x3, x7));
      const float2 lo0 = __ffma2_rn(m, __ffma2_rn(SIX, x0, S6), __fadd2_rn(__fadd2_rn(e01, e02), e04));
      const float2 lo1 = __ffma2_rn(m, __ffma2_rn(TWO, x1, u12), __fadd2_rn(sub(e13, e01), e15));
      const float2 n2 = __ffma2_rn(m, __ffma2_rn(TWO, x2, u34), __fadd2_rn(sub(e23, e02), e26));
      const float2 n3 = __ffma2_rn(m, __ffma2_rn(TWO, x3, __fadd2_rn(t1, t3)), sub(sub(e37, e23), e13));
      const float2 up4 = __ffma2_rn(m, __ffma2_rn(TWO, x4, u56), sub(__fadd2_rn(e45, e46), e04));
      const float2 up5 = __ffma2_rn(m, __ffma2_rn(TWO, x5, __fadd2_rn(t2, t5)), sub(sub(e57, e45), e15));
      const float2 n6 = __ffma2_rn(m, __ffma2_rn(TWO, x6, __fadd2_rn(t4, t6)), sub(sub(e67, e46), e26));
      const float2 n7 = sub(sub(sub(__fmul2_rn(m, __ffma2_rn(SIX, x7, S6)), e67), e57), e37);
      if (r >= 1) {  // node row r: this box row's lower corners and the row below's upper ones
        const float2 pl = __fadd2_rn(lo1, lo3), pu = __fadd2_rn(up5, up7);
        const float ll = __shfl_up_sync(FULL, pl.y, 1, 16), lu = __shfl_up_sync(FULL, pu.y, 1, 16);
        const float2 y = __fadd2_rn(__fadd2_rn(__fadd2_rn(carry[r - 1], lo0), lo2), f2(ll, pl.x));
        carry[r - 1] = __fadd2_rn(__fadd2_rn(up4, up6), f2(lu, pu.x));
        if (lev >= 1) res_out(t, r, y, prv[r], m0, m1, q, acc);
      }
      lo2 = n2;
      lo3 = n3;
      up6 = n6;
      up7 = n7;
      if (r >= 1) {  // row r of the level below has had its last use as a lower neighbour
        prv[r] = cur;
        prr[r] = cuR;
      } else {
        prv[0] = cur;
        prr[0] = cuR;
      }
      cur = nxt;
      cuR = nxR;
    }
    prv[NF] = cur;
    prr[NF] = cuR;
    ca += t.clev;
    cb += t.clev;
    q += t.qlev;
  }
  return acc;
}

// ------------------------------------------------------------------ k_cg_res

// What every phase of a task reads and no phase changes. In shared memory,
// so that the iteration loop does not carry it in registers (as locals these
// values cost 150 registers' worth of spills).
struct ResTask {
  ResLayout l;
  ResBox b;
  int zc, g, dir, gnx, gny, gnz;
  int qpr, nq, npair, ntiles;
  int pass;  // float4 entries of one array in a block's part of the exchange area
  unsigned int qdiv;  // fast_div factor of qpr
};

// q = A d on the block's own nodes (its warps' tiles) and this thread's part
// of d.q. A function of its own: inlined, the march and the pointwise passes
// share one register allocation and spill into each other.
template <class MC>
__device__ __noinline__ float2 res_apply(const ResTask& tk, const MC& mc, const float* sd, const float* sca, float* sq) {
  constexpr int NW = kResThreads / 32, NY = kResNY;
  const ResLayout& l = tk.l;
  const ResBox& b = tk.b;
  const int lane = (int)threadIdx.x & 31, warp = (int)threadIdx.x >> 5;
  float2 acc2 = f2(0.f, 0.f);
  for (int tile = warp; tile < tk.ntiles; tile += NW) {
    const int chunk = tile / tk.npair, pr = 2 * (tile - chunk * tk.npair) + (lane >> 4);
    const bool active = pr < l.nseg * l.nyt;
    const int yt = active ? pr / l.nseg : 0, seg = active ? pr - yt * l.nseg : 0, lx = lane & 15;
    const int kc = chunk * tk.zc, c0 = seg * kResCols - 2 + 2 * lx;
    ResTile t;
    t.drow = l.pd;
    t.dlev = l.pd * l.dr;
    t.crow = l.pc;
    t.clev = l.pc * l.er;
    t.qrow = l.pw;
    t.qlev = l.pw * b.ny;
    t.d = sd + 4 + c0 + yt * NY * t.drow + kc * t.dlev;
    t.ca = sca + c0 + 2 + yt * NY * t.crow + kc * t.clev;
    t.cb = t.ca + l.pc * l.er * l.el;
    t.q = sq + c0 + yt * NY * t.qrow + kc * t.qlev;
    const bool store = active && lx >= 1 && c0 < b.nx;
    const int gx = b.x0 + c0;
    const bool xd0 = ((tk.dir & 1u) && gx == 0) || ((tk.dir & 2u) && gx == tk.gnx);
    const bool xd1 = (tk.dir & 2u) && gx + 1 == tk.gnx;
    t.mc0 = store && !xd0 ? 0xffffffffu : 0u;
    t.mc1 = store && c0 + 1 < b.nx && !xd1 ? 0xffffffffu : 0u;
    t.rows = 0u;
#pragma unroll
    for (int r = 0; r < NY; ++r) {
      const int j = yt * NY + r, gy = b.y0 + j;
      const bool own = j < b.ny;
      if (own && store) t.rows |= 1u << r;
      t.mr[r] = own && !(((tk.dir & 4u) && gy == 0) || ((tk.dir & 8u) && gy == tk.gny)) ? 0xffffffffu : 0u;
    }
    t.lev0 = b.z0 + kc;
    t.zlo = (tk.dir & 16u) ? 0 : -1;
    t.zhi = (tk.dir & 32u) ? tk.gnz : -1;
    acc2 = __fadd2_rn(acc2, res_march(t, mc, min(tk.zc, b.nz - kc)));
  }
  return acc2;
}

// A group of 4 nodes: its place in d and among the exchanged values (-4: not
// exchanged), both multiples of 4, in 13 and 19 bits (d takes less than a
// third of the shared memory, and less than 2 million nodes fit the chip).
__device__ __forceinline__ unsigned int res_group(int d, int z) {
  return (unsigned int)(d >> 2) | ((unsigned int)((z >> 2) + 1) << 13);
}
__device__ __forceinline__ int res_group_d(unsigned int p) { return (int)(p & 0x1fffu) << 2; }
__device__ __forceinline__ int res_group_z(unsigned int p) { return ((int)(p >> 13) - 1) << 2; }

// The block's shared memory and its part of the exchange area from the node
// vectors: d, the coefficients, r, tables, x and P^-1.
template <class MC>
__device__ __noinline__ void res_setup(const SimDev& s, const Ctl& c, const ResTask& tk, const MC& mc,
                                       unsigned char* smem, float4* pp, float4* px) {
  constexpr int TH = kResThreads, NW = TH / 32, MAXQ = kResMaxQ;
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const ResLayout& l = tk.l;
  const ResBox& b = tk.b;
  float* sd = reinterpret_cast<float*>(smem);
  float* sca = reinterpret_cast<float*>(smem + l.off_c);
  float* scb = sca + l.pc * l.er * l.el;
  float* sq = reinterpret_cast<float*>(smem + l.off_q);
  float* sr = reinterpret_cast<float*>(smem + l.off_r);
  unsigned int* sat = reinterpret_cast<unsigned int*>(smem + l.off_at);
  int4* srow = reinterpret_cast<int4*>(smem + l.off_row);
  int2* shalo = reinterpret_cast<int2*>(smem + l.off_halo);
  b.tables(l, 4, srow, shalo);
  // ---------------------------------------------------------- the state in
  res_load_d<float>(s, c, b, l, 4, sd);
  __syncthreads();  // mc, tables
  for (int row = warp; row < l.er * l.el; row += NW) {
    const int e = row / l.er, er = row - e * l.er;
    const int ez = b.z0 - 1 + e, ey = b.y0 - 1 + er;
    const bool in = e <= b.nz && ez >= 0 && ez < tk.gnz && ey >= 0 && ey < tk.gny;
    const int m0 = b.x0 - 2 + tk.gnx * (ey + tk.gny * ez);
    for (int t = lane; t < l.pc; t += 32) {
      const int ex = b.x0 - 2 + t;
      float2 v = f2(0.f, 0.f);
      if (in && ex >= 0 && ex < tk.gnx && HEAT_INDEX_OK(s.sc, m0 + t, (long long)tk.gnx * tk.gny * tk.gnz)) v = s.coef32[m0 + t];
      sca[row * l.pc + t] = mc.ra * v.x;
      scb[row * l.pc + t] = mc.ka * v.y;
    }
  }
  for (int t = tid; t < l.pw * s.res.by * s.res.bz; t += TH) sq[t] = 0.f;
  // x and P^-1 in this thread's groups of the exchange area
  const bool zero_x = c.iter == 0;  // the inner solve starts from e = 0
  // where each group lies in d and, if its nodes are exchanged, there (else -1)
  for (int u = 0; u < MAXQ; ++u) {
    const int qd = tid + u * TH;
    if (qd < tk.nq) {
      const int row = fast_div(qd, tk.qdiv), xq = 4 * (qd - row * tk.qpr);
      const int4 rt = srow[row];
      float pv[4], xv[4], rv[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const bool in = xq + a < b.nx && HEAT_INDEX_OK(s.sc, rt.z + xq + a, s.nn);
        const int m = rt.z + xq + a;
        pv[a] = in ? s.pinv32[m] : 0.f;
        xv[a] = in && !zero_x ? s.e32[m] : 0.f;
        rv[a] = in ? s.r32[m] : 0.f;
      }
      pp[u * TH] = make_float4(pv[0], pv[1], pv[2], pv[3]);
      px[u * TH] = make_float4(xv[0], xv[1], xv[2], xv[3]);
      *reinterpret_cast<float4*>(sr + 4 * qd) = make_float4(rv[0], rv[1], rv[2], rv[3]);
      const bool pub = xq < b.nx && (rt.w || (b.xl && xq == 0) || (b.xr && xq + 4 >= b.nx));
      sat[qd] = res_group(rt.x + xq, pub ? rt.y + xq : -4);
    }
  }
}

template <int E>
__global__ void __launch_bounds__(kResThreads, 1)
    k_cg_res(const SimDev* __restrict__ sims, const int* __restrict__ task_off, const int2* __restrict__ tasks,
             GridSync* __restrict__ gs) {
  constexpr int TH = kResThreads, NW = TH / 32, MAXQ = kResMaxQ;
  constexpr int HB = 16;  // halo cells a thread fetches during the second all-sum
  using X = Exch<float>;
  using MC = typename std::conditional<E == E_P1, ResP1, ResQ1>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ SimDev s;
  __shared__ Ctl c;
  __shared__ ResShared<float, DF> sh;
  __shared__ MC mc;
  __shared__ ResTask tk;
  const ResLayout& l = tk.l;
  const ResBox& b = tk.b;
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int task_end = task_off[blockIdx.x + 1];
  for (int ti = task_off[blockIdx.x]; ti < task_end; ++ti) {
    const int2 task = tasks[ti];
    const int rank = task.y;
    if (!res_open_task<float, DF>(sims, task.x, s, c, sh)) continue;
    if (tid == 32) mc.set(s);
    if (tid == 64) {
      tk.l = res_layout(s.res, false);
      tk.b = ResBox(s, rank);
      tk.zc = s.res.zc;
      tk.g = s.res.g;
      tk.dir = (int)s.dir_faces;
      tk.gnx = s.nx;
      tk.gny = s.ny;
      tk.gnz = s.nz;
      tk.qpr = tk.l.pw >> 2;
      tk.nq = tk.qpr * tk.b.rows;
      tk.qdiv = div_magic(tk.qpr);
      tk.pass = res_groups(s.res) * TH;
      tk.npair = (tk.l.nseg * tk.l.nyt + 1) / 2;
      tk.ntiles = tk.npair * ((tk.b.nz + tk.zc - 1) / tk.zc);
    }
    __syncthreads();
    float* sd = reinterpret_cast<float*>(smem);
    float* sca = reinterpret_cast<float*>(smem + l.off_c);
    float* sq = reinterpret_cast<float*>(smem + l.off_q);
    float* sr = reinterpret_cast<float*>(smem + l.off_r);
    unsigned int* sat = reinterpret_cast<unsigned int*>(smem + l.off_at);
    int4* srow = reinterpret_cast<int4*>(smem + l.off_row);
    int2* shalo = reinterpret_cast<int2*>(smem + l.off_halo);
    unsigned long long* zx = reinterpret_cast<unsigned long long*>(s.res_z);
    float4* const pp0 = reinterpret_cast<float4*>(s.res_x) + (size_t)rank * 2 * tk.pass;
    res_setup(s, c, tk, mc, smem, pp0 + tid, pp0 + tk.pass + tid);
    __syncthreads();
    // ---------------------------------------------------------- iterations
    const int max_rounds = gs->rounds;
    for (int round = 0;; ++round) {
      const unsigned int tag = sh.tag0 + 1u + (unsigned int)round;
      const float2 acc2 = res_apply<MC>(tk, mc, sd, sca, sq);
      // a fresh copy each round: what is derived from it is formed again instead
      // of being kept (and spilled) across the march
      int tn = tid;
      asm volatile("" : "+r"(tn));
      float4* const pp = pp0 + tn;
      float4* const px = pp + tk.pass;
      float4 pv[MAXQ];  // in flight during the sum
#pragma unroll
      for (int u = 0; u < MAXQ; ++u)
        pv[u] = tn + u * TH < tk.nq ? pp[u * TH] : make_float4(0.f, 0.f, 0.f, 0.f);
      float acc = acc2.x + acc2.y;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) sh.wsum[warp] = acc * sh.scale;
      __syncthreads();
      if (warp == 0) {
        const DF v = res_block_sum<float, DF, NW>(sh.wsum);
        DF tot = v;
        bool ok = true;
        if (tk.g > 1 || gs->extra) ok = res_all_sum<DF>(v, s.res_slots, tk.g, rank, tag, gs, tot);
        if (lane == 0) res_decide_alpha<float, DF>(sh, ok, tot);
      }
      __syncthreads();
      int go = sh.go;
      if (go == kEndAbort) return;
      if (go == kEndFailed) {
        if (rank == 0 && tid == 0) res_finish<float, DF>(s, sh, go, false, tag);
        break;
      }
      const float alpha = sh.alpha;
      const float2 ma = f2(-alpha, -alpha);
      float2 z[MAXQ][2], racc[2] = {f2(0.f, 0.f), f2(0.f, 0.f)};
#pragma unroll
      for (int u = 0; u < MAXQ; ++u) {
        const int qd = tn + u * TH;
        // (a value for every group: one left undefined would count as carried
        // from round to round, and the arrays would spill)
        z[u][0] = z[u][1] = f2(0.f, 0.f);
        if (qd < tk.nq) {
          const float4 rv = *reinterpret_cast<const float4*>(sr + 4 * qd);
          const float4 qv = *reinterpret_cast<const float4*>(sq + 4 * qd);
          z[u][0] = __ffma2_rn(ma, f2(qv.x, qv.y), f2(rv.x, rv.y));  // r for now
          z[u][1] = __ffma2_rn(ma, f2(qv.z, qv.w), f2(rv.z, rv.w));
        }
      }
#pragma unroll
      for (int u = 0; u < MAXQ; ++u) {
        const int qd = tn + u * TH;
        if (qd < tk.nq) {
          const float2 r0 = z[u][0], r1 = z[u][1];
          *reinterpret_cast<float4*>(sr + 4 * qd) = make_float4(r0.x, r0.y, r1.x, r1.y);
          z[u][0] = __fmul2_rn(r0, f2(pv[u].x, pv[u].y));
          z[u][1] = __fmul2_rn(r1, f2(pv[u].z, pv[u].w));
          racc[u & 1] = __ffma2_rn(r0, z[u][0], racc[u & 1]);
          racc[u & 1] = __ffma2_rn(r1, z[u][1], racc[u & 1]);
        }
      }
      if (tk.g > 1) {
#pragma unroll
        for (int u = 0; u < MAXQ; ++u) {
          if (tn + u * TH < tk.nq) {
            const int zo = res_group_z(sat[tn + u * TH]);
            if (zo >= 0) X::store4(zx + zo, z[u][0], z[u][1], tag);
          }
        }
      }
      float2 rz = f2(racc[0].x + racc[0].y, racc[1].x + racc[1].y);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        rz = __fadd2_rn(rz, f2(__shfl_xor_sync(0xffffffffu, rz.x, o), __shfl_xor_sync(0xffffffffu, rz.y, o)));
      if (lane == 0) {
        sh.wsum[warp] = rz.x * sh.scale;
        sh.wsum[NW + warp] = rz.y * sh.scale;
      }
      float4 xv[MAXQ];  // in flight during the sum
#pragma unroll
      for (int u = 0; u < MAXQ; ++u)
        xv[u] = tn + u * TH < tk.nq ? px[u * TH] : make_float4(0.f, 0.f, 0.f, 0.f);
      __syncthreads();
      float hz[HB] = {};
      int hat[HB];
#pragma unroll
      for (int u = 0; u < HB; ++u) hat[u] = -1;
      bool ok = true;
      if (warp == 0) {
        const DF v = res_block_sum<float, DF, 2 * NW>(sh.wsum);
        DF tot = v;
        if (tk.g > 1) ok = res_all_sum<DF>(v, s.res_slots + res_mail(tk.g), tk.g, rank, tag, gs, tot);
        if (lane == 0) res_decide_beta<float, DF>(sh, s, ok, tot, false, round + 1 >= max_rounds);
      } else if (tk.g > 1) {
        ok = res_halo_fetch<float, HB>(b, srow, shalo, tn - 32, TH - 32, zx, tag, gs, hz, hat);
      }
      if (__syncthreads_or(!ok)) return;
      go = sh.go;
      const float2 pa = f2(alpha, alpha);
      if (go == kGo) {
        if (tid == 0) sh.delta = res_kept(sh.delta);  // its warp has no halo to write
        const float beta = sh.beta;
        const float2 be = f2(beta, beta);
        float4 dv[MAXQ];
        int at[MAXQ];
#pragma unroll
        for (int u = 0; u < MAXQ; ++u) {
          at[u] = 0;
          dv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (tn + u * TH < tk.nq) {
            at[u] = res_group_d(sat[tn + u * TH]);
            dv[u] = *reinterpret_cast<const float4*>(sd + at[u]);
          }
        }
#pragma unroll
        for (int u = 0; u < MAXQ; ++u) {
          if (tn + u * TH < tk.nq) {
            const float2 d0 = f2(dv[u].x, dv[u].y), d1 = f2(dv[u].z, dv[u].w);
            const float2 x0 = __ffma2_rn(pa, d0, f2(xv[u].x, xv[u].y)), x1 = __ffma2_rn(pa, d1, f2(xv[u].z, xv[u].w));
            px[u * TH] = make_float4(x0.x, x0.y, x1.x, x1.y);
            const float2 n0 = __ffma2_rn(be, d0, z[u][0]), n1 = __ffma2_rn(be, d1, z[u][1]);
            // a group that ends its row reaches past the mesh only (boxes with a
            // neighbour behind are a multiple of 4 wide), where d stays zero
            *reinterpret_cast<float4*>(sd + at[u]) = make_float4(n0.x, n0.y, n1.x, n1.y);
          }
        }
        if (tk.g > 1) {
          if (warp > 0) {
#pragma unroll
            for (int u = 0; u < HB; ++u)
              if (hat[u] >= 0) sd[hat[u]] = res_fma(beta, sd[hat[u]], hz[u]);
          }
          // what the fetch has not covered
          for (int h = HB * (TH - 32) + tn; h < res_halo_cells(b) && ok; h += TH) {
            float z1[1];
            int a1[1];
            ok = res_halo_fetch<float, 1>(b, srow, shalo, h, 1 << 30, zx, tag, gs, z1, a1);
            sd[a1[0]] = res_fma(beta, sd[a1[0]], z1[0]);
          }
        }
        if (__syncthreads_or(!ok)) return;
        continue;
      }
      // ------------------------------------------------------ the state out
#pragma unroll
      for (int u = 0; u < MAXQ; ++u) {
        const int qd = tid + u * TH;
        if (qd < tk.nq) {
          const int row = fast_div(qd, tk.qdiv), xq = 4 * (qd - row * tk.qpr);
          const int4 rt = srow[row];
          const float xo[4] = {xv[u].x, xv[u].y, xv[u].z, xv[u].w};
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const int m = rt.z + xq + a;
            if (xq + a < b.nx && HEAT_INDEX_OK(s.sc, m, s.nn)) {
              const float dv = sd[rt.x + xq + a];
              s.e32[m] = fmaf(alpha, dv, xo[a]);
              if (go == kEndIter) {
                s.d32[c.id][m] = dv;
                s.r32[m] = sr[4 * qd + a];
              }
            }
          }
        }
      }
      if (rank == 0 && tid == 0) res_finish<float, DF>(s, sh, go, true, tag);
      break;
    }
  }
}

// ---------------------------------------------------------------- k_cg_res64

// The FP64 form. FP64 runs at 1/58 of the FP32 rate on this GPU (a warp's FP64
// instruction takes a scheduler 64 cycles), so the operator's arithmetic is
// the whole cost: the factorised product takes about 60 operations per node
// with its halo, a row of the assembled operator 27. Each block therefore
// sums its nodes' 27 row coefficients over their elements once per launch,
// keeps them in shared memory (216 bytes per node, so cubes of up to 49
// elements an edge fit) and applies them 27 FMAs per node and iteration. x, r, q, z and
// P^-1 stay in registers. Row layout: coefficient o = (ox+1) + 3 (oy+1) +
// 9 (oz+1) of node n at sw[o * nodes + n].
template <int E>
__global__ void __launch_bounds__(kResThreads, 1)
    k_cg_res64(const SimDev* __restrict__ sims, const int* __restrict__ task_off, const int2* __restrict__ tasks,
               GridSync* __restrict__ gs) {
  constexpr int TH = kResThreads, MAXN = kResMaxN, HB = 4;
  using X = Exch<double>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ SimDev s;
  __shared__ Ctl c;
  __shared__ ResShared<double, double> sh;
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int task_end = task_off[blockIdx.x + 1];
  for (int ti = task_off[blockIdx.x]; ti < task_end; ++ti) {
    const int2 task = tasks[ti];
    const int rank = task.y;
    if (!res_open_task<double, double>(sims, task.x, s, c, sh)) continue;
    const ResGeo rg = s.res;
    const ResLayout l = res_layout(rg, true);
    const ResBox b(s, rank);
    double* sd = reinterpret_cast<double*>(smem);
    double* sw = reinterpret_cast<double*>(smem + l.off_c);
    int4* srow = reinterpret_cast<int4*>(smem + l.off_row);
    int2* shalo = reinterpret_cast<int2*>(smem + l.off_halo);
    unsigned long long* zx = reinterpret_cast<unsigned long long*>(s.res_z);
    const int nn = b.rows * b.nx, cap = rg.bx * rg.by * rg.bz;
    const unsigned int ndiv = div_magic(b.nx);
    b.tables(l, 1, srow, shalo);
    res_load_d<double>(s, c, b, l, 1, sd);
    __syncthreads();
    double x[MAXN], r[MAXN], p[MAXN], q[MAXN], z[MAXN];
    int at[MAXN], zo[MAXN], gm[MAXN];  // in d; in the exchanged values (-1: not exchanged); in the node vectors
    const double* __restrict__ rin = s.r;
    double* __restrict__ xg = s.vec64[c.ix];
#pragma unroll
    for (int u = 0; u < MAXN; ++u) {
      const int n = tid + u * TH;
      x[u] = r[u] = p[u] = q[u] = z[u] = 0.0;
      at[u] = 0;
      gm[u] = 0;
      zo[u] = -1;
      if (n < nn) {
        const int row = fast_div(n, ndiv), i = n - row * b.nx;
        const int4 rt = srow[row];
        at[u] = rt.x + i;
        gm[u] = rt.z + i;
        if (rt.w || (b.xl && i == 0) || (b.xr && i == b.nx - 1)) zo[u] = rt.y + i;
        if (HEAT_INDEX_OK(s.sc, gm[u], s.nn)) {
          x[u] = xg[gm[u]];
          r[u] = rin[gm[u]];
          p[u] = s.pinv[gm[u]];
        }
        // the node's row of A (Dirichlet rows zero: q = 0 there)
        double w[27];
#pragma unroll
        for (int o = 0; o < 27; ++o) w[o] = 0.0;
        int gi, gj, gk;
        node_of(s, gm[u], gi, gj, gk);
        if (!is_dirichlet(s, gi, gj, gk)) {
#pragma unroll
          for (int cc = 0; cc < 8; ++cc) {
            const int cx = cc & 1, cy = (cc >> 1) & 1, cz = (cc >> 2) & 1;
            const int ex = gi - cx, ey = gj - cy, ez = gk - cz;
            if (ex < 0 || ey < 0 || ez < 0 || ex >= s.nx || ey >= s.ny || ez >= s.nz) continue;
            const double2 cf = s.coef[ex + (long long)s.nx * (ey + (long long)s.ny * ez)];
            const double wa = s.inv_dt * cf.x, wb = s.theta * cf.y;
#pragma unroll
            for (int dd = 0; dd < 8; ++dd) {
              const int o = ((dd & 1) - cx + 1) + 3 * (((dd >> 1) & 1) - cy + 1) + 9 * (((dd >> 2) & 1) - cz + 1);
              if (E == E_P1) {
                if (!p1_mass_nz(cc, dd)) continue;
                w[o] += wa * s.p1w[8 * cc + dd] + (p1_stiff_nz(cc, dd) ? wb * s.p1w[64 + 8 * cc + dd] : 0.0);
              } else {
                w[o] += wa * s.mhat[cc ^ dd] + wb * s.khat[cc ^ dd];
              }
            }
          }
        }
#pragma unroll
        for (int o = 0; o < 27; ++o) sw[o * cap + n] = w[o];
      }
    }
    const int dy = l.pd, dz = l.pd * l.dr;
    // ---------------------------------------------------------- iterations
    const int max_rounds = gs->rounds;
    for (int round = 0;; ++round) {
      const unsigned int tag = sh.tag0 + 1u + (unsigned int)round;
      double acc = 0.0;
#pragma unroll
      for (int u = 0; u < MAXN; ++u) {
        const int n = tid + u * TH;
        if (n < nn) {
          const double* dp = sd + at[u];
          const double* wp = sw + n;
          double y[3] = {0.0, 0.0, 0.0};  // one chain per level
#pragma unroll
          for (int o = 0; o < 27; ++o)
            y[o / 9] += wp[o * cap] * dp[(o % 3 - 1) + (o / 3 % 3 - 1) * dy + (o / 9 - 1) * dz];
          q[u] = (y[0] + y[1]) + y[2];
          acc += dp[0] * q[u];
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) sh.wsum[warp] = acc;
      __syncthreads();
      if (warp == 0) {
        const double v = res_block_sum<double, double, TH / 32>(sh.wsum);
        double tot = v;
        bool ok = true;
        if (rg.g > 1 || gs->extra) ok = res_all_sum<double>(v, s.res_slots, rg.g, rank, tag, gs, tot);
        if (lane == 0) res_decide_alpha<double, double>(sh, ok, tot);
      }
      __syncthreads();
      int go = sh.go;
      if (go == kEndAbort) return;
      if (go == kEndFailed) {
        if (rank == 0 && tid == 0) res_finish<double, double>(s, sh, go, false, tag);
        break;
      }
      const double alpha = sh.alpha;
      // the periodic true residual: x advances, k_open forms r (Algorithm 1)
      const bool resid_it = s.resid_period > 0 && sh.iter > 0 && sh.iter % s.resid_period == 0;
      acc = 0.0;
      if (!resid_it) {
#pragma unroll
        for (int u = 0; u < MAXN; ++u)
          if (tid + u * TH < nn) {
            r[u] -= alpha * q[u];
            z[u] = res_mul(p[u], r[u]);
            acc += r[u] * z[u];
            if (zo[u] >= 0) X::store(zx + 2 * (size_t)zo[u], z[u], tag);
          }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      __syncthreads();  // every thread has read sh.iter
      if (lane == 0) sh.wsum[warp] = acc;
      __syncthreads();
      double hz[HB];
      int hat[HB];
      bool ok = true;
      if (warp == 0) {
        const double v = res_block_sum<double, double, TH / 32>(sh.wsum);
        double tot = v;
        if (rg.g > 1) ok = res_all_sum<double>(v, s.res_slots + res_mail(rg.g), rg.g, rank, tag, gs, tot);
        if (lane == 0) res_decide_beta<double, double>(sh, s, ok, tot, resid_it, round + 1 >= max_rounds);
      } else if (rg.g > 1 && !resid_it) {
        ok = res_halo_fetch<double, HB>(b, srow, shalo, tid - 32, TH - 32, zx, tag, gs, hz, hat);
      }
      // x in the shadow of the sum
#pragma unroll
      for (int u = 0; u < MAXN; ++u)
        if (tid + u * TH < nn) x[u] += alpha * sd[at[u]];
      if (__syncthreads_or(!ok)) return;
      go = sh.go;
      if (go == kGo) {
        const double beta = sh.beta;
#pragma unroll
        for (int u = 0; u < MAXN; ++u)
          if (tid + u * TH < nn) sd[at[u]] = res_fma(beta, sd[at[u]], z[u]);
        if (rg.g > 1) {
          if (warp > 0) {
#pragma unroll
            for (int u = 0; u < HB; ++u)
              if (hat[u] >= 0) sd[hat[u]] = res_fma(beta, sd[hat[u]], hz[u]);
          }
          for (int h = HB * (TH - 32) + tid; h < res_halo_cells(b) && ok; h += TH) {
            double z1[1];
            int a1[1];
            ok = res_halo_fetch<double, 1>(b, srow, shalo, h, 1 << 30, zx, tag, gs, z1, a1);
            sd[a1[0]] = res_fma(beta, sd[a1[0]], z1[0]);
          }
        }
        if (__syncthreads_or(!ok)) return;
        continue;
      }
      // ------------------------------------------------------ the state out
#pragma unroll
      for (int u = 0; u < MAXN; ++u)
        if (tid + u * TH < nn && HEAT_INDEX_OK(s.sc, gm[u], s.nn)) {
          xg[gm[u]] = x[u];
          s.d[c.id][gm[u]] = sd[at[u]];
          if (go == kEndIter) s.r[gm[u]] = r[u];
        }
      if (rank == 0 && tid == 0) res_finish<double, double>(s, sh, go, true, tag);
      break;
    }
  }
}

}  // namespace heat
