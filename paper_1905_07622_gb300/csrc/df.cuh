// Double-float arithmetic: a value is the unevaluated sum hi + lo of two
// floats with |lo| <= ulp(hi)/2, about 48 significant bits. Built from the
// error-free transformations of Knuth (two-sum: the rounding error of a + b
// is itself a float) and of Dekker with a fused multiply-add (two-product:
// the rounding error of a * b is fma(a, b, -fl(a*b))). Addition is the short
// form (error bounded by about 2^-44 times |a| + |b|, not |a + b|), which is
// what a residual b - A x needs: its error must be small next to the operand
// scale |b|, not next to the small result.
//
// On this GPU FP64 runs at 1/58 of the FP32 rate, so an operator pass in
// double-float, about ten FP32 operations per FP64 one, is several times
// faster than the same pass in FP64 and far more accurate than an FP32 one.
#pragma once

#include <cstring>

#include <cuda_runtime.h>

namespace heat {

// Conversions by integer field arithmetic: a conversion between float and
// double is an FP64 instruction, which takes a scheduler 64 cycles here, and
// the refinement passes were bound by them (62% of the FP64 pipe's cycles with
// the integer pipe at 9%; the outer pass of 1.03e6 unknowns 121 us with them,
// 96 with these and its operands loaded a level ahead). Zero, and values of
// ordinary range, take a dozen integer operations; anything else the plain
// conversion. The results are the plain conversions' (a tie of the leading part
// goes away from zero; the low part takes it up).
__host__ __device__ __forceinline__ unsigned int df_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  unsigned int u;
  std::memcpy(&u, &f, 4);
  return u;
#endif
}
__host__ __device__ __forceinline__ float df_float(unsigned int u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  std::memcpy(&f, &u, 4);
  return f;
#endif
}
__host__ __device__ __forceinline__ double df_widen(float f) {
  const unsigned int u = df_bits(f), e = (u >> 23) & 0xffu;
  if (e - 1u < 254u) {
    const unsigned int h = (u & 0x80000000u) | ((e + 896u) << 20) | ((u >> 3) & 0xfffffu), l = u << 29;
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)h, (int)l);
#else
    const unsigned long long w = ((unsigned long long)h << 32) | l;
    double d;
    std::memcpy(&d, &w, 8);
    return d;
#endif
  }
  return (u << 1) == 0u ? 0.0 : (double)f;
}
// d = hi + lo, hi the nearest float, lo the nearest float to the rest
__host__ __device__ __forceinline__ void df_split(double d, float& hi, float& lo) {
#ifdef __CUDA_ARCH__
  const unsigned int uh = (unsigned int)__double2hiint(d), ul = (unsigned int)__double2loint(d);
#else
  unsigned long long w;
  std::memcpy(&w, &d, 8);
  const unsigned int uh = (unsigned int)(w >> 32), ul = (unsigned int)w;
#endif
  const unsigned int e = (uh >> 20) & 0x7ffu, sign = uh & 0x80000000u;
  if (e - 950u < 200u) {  // both parts normal floats
    const unsigned int rl = ul + 0x10000000u;  // the 29 bits below hi rounded into bit 29
    const unsigned int rh = (uh & 0x7fffffffu) + (rl < 0x10000000u ? 1u : 0u);
    hi = df_float(sign | (((rh << 3) | (rl >> 29)) - (896u << 23)));
    const int rest = (int)(ul - (rl & 0xe0000000u));  // in units of 2^(e - 1075)
    // two exact powers of two: 2^-29 and 2^(e - 1046)
    const float l = (float)rest * 1.862645149230957e-9f * df_float((e - 919u) << 23);
    lo = df_float(df_bits(l) ^ sign);
  } else if (((uh << 1) | ul) == 0u) {
    hi = lo = 0.f;
  } else {
    hi = (float)d;
    lo = (float)(d - (double)hi);
  }
}
__host__ __device__ __forceinline__ float df_narrow(double d) {
  float h, l;
  df_split(d, h, l);
  return h;
}

struct DF {
  float hi, lo;
  DF() = default;
  __host__ __device__ __forceinline__ DF(float h, float l) : hi(h), lo(l) {}
  __host__ __device__ __forceinline__ DF(int v) : hi((float)v), lo(0.f) {}
  __host__ __device__ __forceinline__ DF(double d) { df_split(d, hi, lo); }
  __host__ __device__ __forceinline__ double to_double() const { return df_widen(hi) + df_widen(lo); }
};

// s + e == a + b exactly (Knuth)
__host__ __device__ __forceinline__ void df_two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
// s + e == a + b exactly when |a| >= |b| (Dekker)
__host__ __device__ __forceinline__ void df_fast_two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  e = b - (s - a);
}

__host__ __device__ __forceinline__ DF operator+(const DF& a, const DF& b) {
  float s, e;
  df_two_sum(a.hi, b.hi, s, e);
  e += a.lo + b.lo;
  float h, l;
  df_fast_two_sum(s, e, h, l);
  return DF(h, l);
}
__host__ __device__ __forceinline__ DF operator-(const DF& a) { return DF(-a.hi, -a.lo); }
__host__ __device__ __forceinline__ DF operator-(const DF& a, const DF& b) { return a + (-b); }
__host__ __device__ __forceinline__ DF operator*(const DF& a, const DF& b) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);  // the product's rounding error, exactly
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  float h, l;
  df_fast_two_sum(p, e, h, l);
  return DF(h, l);
}
__host__ __device__ __forceinline__ DF& operator+=(DF& a, const DF& b) {
  a = a + b;
  return a;
}

__host__ __device__ __forceinline__ double to_d(double v) { return v; }
__host__ __device__ __forceinline__ double to_d(const DF& v) { return v.to_double(); }

struct DF2 {
  DF x, y;
};

}  // namespace heat

#ifdef __CUDACC__
// Segment shuffles of a double-float (both halves); at global scope beside
// the built-in overloads so that unqualified calls keep finding those.
__device__ __forceinline__ heat::DF __shfl_down_sync(unsigned mask, const heat::DF& v, unsigned delta, int width) {
  return heat::DF(__shfl_down_sync(mask, v.hi, delta, width), __shfl_down_sync(mask, v.lo, delta, width));
}
__device__ __forceinline__ heat::DF __shfl_up_sync(unsigned mask, const heat::DF& v, unsigned delta, int width) {
  return heat::DF(__shfl_up_sync(mask, v.hi, delta, width), __shfl_up_sync(mask, v.lo, delta, width));
}
#endif
