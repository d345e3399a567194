// Double-float numbers: a value is the unevaluated sum hi + lo of two floats
// with |lo| <= ulp(hi) / 2, about 48 significant bits (relative rounding
// ~3.6e-15).  GB300 issues FP32 FMAs at about 64 times its FP64 rate, so
// vector work that needs more than FP32 but tolerates ~1e-14 relative error
// (the Dslash of a CG reliable update) runs faster on the FP32 pipes in this
// form than in FP64.
//
// Error-free transformations used:
//   two_sum       Knuth, TAOCP vol. 2, sec. 4.2.2: s + e == a + b exactly;
//   fast_two_sum  Dekker (1971), valid when |a| >= |b| or a == 0;
//   product       a * b == p + e exactly with p = fl(a b), e = fma(a, b, -p).
// Addition is the "sloppy" double-float sum (one two_sum of the high parts,
// the low parts added in FP32): its error is bounded by ~2^-47 of the larger
// operand, which is the scale that matters for residuals.  These routines
// must not be compiled with reassociation (no fast-math); nvcc's FMA
// contraction is harmless here because every product is written out.
#pragma once

#include <cuda_runtime.h>

#include "fg_common.cuh"

namespace fg {

struct DF {
  float hi, lo;
  DF() = default;
  __host__ __device__ __forceinline__ constexpr DF(float h) : hi(h), lo(0.0f) {}
  __host__ __device__ __forceinline__ constexpr DF(int h) : hi((float)h), lo(0.0f) {}
  // Nearest double-float to a double (host or device; FP64 arithmetic, which
  // the compiler folds away for a literal argument).
  __host__ __device__ __forceinline__ constexpr explicit DF(double d)
      : hi((float)d), lo((float)(d - (double)(float)d)) {}
  __host__ __device__ __forceinline__ constexpr DF(float h, float l) : hi(h), lo(l) {}
  __host__ __device__ __forceinline__ explicit operator double() const { return (double)hi + (double)lo; }
};

__device__ __forceinline__ DF df_fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return DF(s, __fsub_rn(b, __fsub_rn(s, a)));
}

__device__ __forceinline__ DF df_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return DF(s, e);
}

__device__ __forceinline__ DF operator+(DF a, DF b) {
  const DF s = df_two_sum(a.hi, b.hi);
  return df_fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ DF& operator+=(DF& a, DF b) { return a = a + b; }
__device__ __forceinline__ DF operator-(DF a) { return DF(-a.hi, -a.lo); }
__device__ __forceinline__ DF operator-(DF a, DF b) { return a + (-b); }
// Products keep the lo * lo term: it is ~2^-48 of the result, but for a
// square it is never negative, so dropping it (the usual "sloppy" product)
// biases every x * x low by ~6e-16 on average; in the exponential of the
// link update that made each drift shrink |U|^2 by ~4e-15, which moved the
// dH of a 32^4 trajectory by ~7e-7.
__device__ __forceinline__ DF operator*(DF a, DF b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.lo, b.lo, e);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return df_fast_two_sum(p, e);
}
// a * b + c with one normalisation.  Generic code calls fma, sqrt and
// fabs unqualified; the using-declarations keep the float and double
// overloads visible next to the double-float ones declared here (otherwise
// those would hide them, and a float argument would convert to DF).
using ::fma;
using ::sqrt;
using ::fabs;
__device__ __forceinline__ DF fma(DF a, DF b, DF c) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  const DF s = df_two_sum(p, c.hi);
  e = __fmaf_rn(a.lo, b.lo, e);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  e = __fadd_rn(e, __fadd_rn(s.lo, c.lo));
  return df_fast_two_sum(s.hi, e);
}
// a + f for a float f (CG solution updates)
__device__ __forceinline__ DF df_add_f(DF a, float f) {
  const DF s = df_two_sum(a.hi, f);
  return df_fast_two_sum(s.hi, __fadd_rn(s.lo, a.lo));
}
__device__ __forceinline__ DF& operator-=(DF& a, DF b) { return a = a - b; }
__device__ __forceinline__ DF& operator*=(DF& a, DF b) { return a = a * b; }
// a * f for a float f
__device__ __forceinline__ DF operator*(DF a, float f) {
  const float p = __fmul_rn(a.hi, f);
  float e = __fmaf_rn(a.hi, f, -p);
  e = __fmaf_rn(a.lo, f, e);
  return df_fast_two_sum(p, e);
}
// Quotient by two correction steps: q1 = a.hi / b.hi, q2 = r1.hi / b.hi
// with the remainder r1 = a - q1 b, q3 = r2.hi / b.hi with r2 = r1 - q2 b.
// One step is accurate to ~2^-47 but not unbiased: dividing r1 (which
// contains -q1 b.lo) by b.hi instead of b leaves -q (b.lo / b.hi)^2, never
// positive, so 1/x came out low by 6.5e-16 on average, and whatever was
// scaled by such a quotient shrank.  The second step's own error is ~2^-72.
__device__ __forceinline__ DF operator/(DF a, DF b) {
  const float q1 = __fdiv_rn(a.hi, b.hi);
  const DF r1 = a - b * q1;
  const float q2 = __fdiv_rn(r1.hi, b.hi);
  const DF r2 = r1 - b * q2;
  const DF q = df_fast_two_sum(q1, q2);
  return df_add_f(q, __fdiv_rn(r2.hi, b.hi));
}
// Ordering of normalised double-floats (|lo| <= ulp(hi) / 2).
__device__ __forceinline__ bool operator<(DF a, DF b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }
__device__ __forceinline__ bool operator>(DF a, DF b) { return b < a; }
__device__ __forceinline__ DF fabs(DF a) { return (a.hi < 0.0f || (a.hi == 0.0f && a.lo < 0.0f)) ? -a : a; }
// Square root: s = sqrt(a.hi) in FP32, then a Newton step on s^2 = a with
// the residual a - s^2 formed exactly (s^2 = p + e by the FMA product, and
// a.hi - p is exact by Sterbenz's lemma), then a second one in double-float.
// One step leaves an error of one sign (a Newton step for sqrt always lands
// above the root, here by ~2^-49 relative); the second removes it.
__device__ __forceinline__ DF sqrt(DF a) {
  if (!(a.hi > 0.0f)) return DF(0.0f);
  const float s = __fsqrt_rn(a.hi);
  const float p = __fmul_rn(s, s);
  const float e = __fmaf_rn(s, s, -p);
  const float d = __fadd_rn(__fsub_rn(__fsub_rn(a.hi, p), e), a.lo);
  const DF y = df_fast_two_sum(s, __fdiv_rn(d, __fadd_rn(s, s)));
  const DF r = a - y * y;
  return y + DF(__fdiv_rn(r.hi, __fadd_rn(y.hi, y.hi)));
}

// Storage: one complex double-float is a float4 (re.hi, re.lo, im.hi, im.lo),
// the same 16 bytes as a complex double; a pair of entries is two float4.
template <> struct Vec2<DF> { typedef float4 T; };
template <> struct Quad<DF> {
  static __device__ __forceinline__ Cx<DF> c(float4 v) { return cx<DF>(DF(v.x, v.y), DF(v.z, v.w)); }
  static __device__ __forceinline__ Cx<DF> load1(const void* base, size_t idx) {
    return c(__ldg((const float4*)base + idx));
  }
  static __device__ __forceinline__ void store1(void* base, size_t idx, Cx<DF> a) {
    ((float4*)base)[idx] = make_float4(a.re.hi, a.re.lo, a.im.hi, a.im.lo);
  }
  static __device__ __forceinline__ void load(const void* base, size_t idx, Cx<DF>& a, Cx<DF>& b) {
    const float4* p = (const float4*)base + 2 * idx;
    a = c(__ldg(p));
    b = c(__ldg(p + 1));
  }
  static __device__ __forceinline__ void load_cg(const void* base, size_t idx, Cx<DF>& a, Cx<DF>& b) {
    const float4* p = (const float4*)base + 2 * idx;
    a = c(p[0]);
    b = c(p[1]);
  }
  static __device__ __forceinline__ void store(void* base, size_t idx, Cx<DF> a, Cx<DF> b) {
    float4* p = (float4*)base + 2 * idx;
    p[0] = make_float4(a.re.hi, a.re.lo, a.im.hi, a.im.lo);
    p[1] = make_float4(b.re.hi, b.re.lo, b.im.hi, b.im.lo);
  }
};

// block_reduce_store (fg_common.cuh) for double-float values (fixed tree, FP32 arithmetic only); the
// partials are stored as doubles.
template <int NV>
__device__ __forceinline__ void block_reduce_store_df(DF v[NV], double* __restrict__ partial,
                                                      int nblocks_stride) {
  __shared__ DF shd[NV][32];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int nwarps = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    DF x = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      x = x + DF(__shfl_down_sync(0xffffffffu, x.hi, o), __shfl_down_sync(0xffffffffu, x.lo, o));
    if (lane == 0) shd[k][warp] = x;
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      DF x = lane < nwarps ? shd[k][lane] : DF(0.0f);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        x = x + DF(__shfl_down_sync(0xffffffffu, x.hi, o), __shfl_down_sync(0xffffffffu, x.lo, o));
      if (lane == 0) partial[(size_t)k * nblocks_stride + blockIdx.x] = double(x);
    }
  }
}

// Horner's rule of exp_coeffs in double-float, to order 16 (the first
// omitted term is below 1e-17, far below the rounding, as it must be: a
// truncation error has one sign).  Orders 16 to 10 contribute less than 2e-9
// and run in FP32 (1e-16); a conversion to double-float follows.
template <> __device__ __forceinline__ void exp_coeffs<DF>(DF c0, DF c1, Cx<DF> f[3]) {
  Cx<float> q[3] = {cx<float>(0.0f, 0.0f), cx<float>(0.0f, 0.0f), cx<float>(0.0f, 0.0f)};
  exp_horner<float, 16, 10>(c0.hi, c1.hi, q);
#pragma unroll
  for (int j = 0; j < 3; ++j) f[j] = cx<DF>(DF(q[j].re), DF(q[j].im));
  exp_horner<DF, 9, 0>(c0, c1, f);
}
template <> __device__ __forceinline__ int exp_halvings<DF>(DF c1) { return exp_halvings(c1.hi); }

// ---------------------------------------------------------------------------
// Products of SU(3) matrices in double-float with an anchored accumulator.
// For unitary a and b every partial sum of the real or imaginary part of an
// entry of a b lies in [-1, 1] (each term is bounded by |a_ik| |b_kj| and
// those sum to at most |row i of a| |column j of b| = 1, Cauchy-Schwarz), so
// t = 3 + (partial sum) stays in [2, 4], where the FP32 grid is 2^-22.  A
// term x_h y_h enters t by one FMA; its rounding error
// rho = t_old + x_h y_h - t_new (|rho| <= 2^-23) is recovered by a second FMA,
// fma(x_h, y_h, t_old - t_new), whose operand t_old - t_new is exact
// (Sterbenz's lemma) and whose result is within 2^-24 |rho| <= 2^-47 of rho;
// the low parts enter as x_h y_l + x_l y_h in FP32.  The value is
// (t - 3) + lo, t - 3 being exact, normalised by two_sum: six FP32
// operations per term instead of the fifteen of a double-float FMA, at the
// same ~2^-47 accuracy.  Callers guarantee unitary factors (the links of a
// staple and products of them); other inputs lose accuracy gracefully as t
// leaves [2, 4].
struct Anchored {
  float t, lo;
  __device__ __forceinline__ Anchored() : t(3.0f), lo(0.0f) {}
  // += x y
  __device__ __forceinline__ void add(DF x, DF y) {
    const float t0 = t;
    t = __fmaf_rn(x.hi, y.hi, t0);
    lo = __fadd_rn(lo, __fmaf_rn(x.hi, y.hi, __fsub_rn(t0, t)));
    lo = __fmaf_rn(x.hi, y.lo, lo);
    lo = __fmaf_rn(x.lo, y.hi, lo);
  }
  // -= x y
  __device__ __forceinline__ void sub(DF x, DF y) { add(-x, y); }
  __device__ __forceinline__ DF value() const { return df_two_sum(__fsub_rn(t, 3.0f), lo); }
};

// m^dagger if d, else m (run-time choice by selects, so that one code path
// serves both).
__device__ __forceinline__ M3<DF> dagger_if(const M3<DF>& m, bool d) {
  M3<DF> r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const Cx<DF> v = d ? m.e[j][i] : m.e[i][j];
      r.e[i][j] = cx<DF>(v.re, d ? -v.im : v.im);
    }
  return r;
}

// a b for unitary double-float matrices.
__device__ __forceinline__ M3<DF> su3_mul(const M3<DF>& a, const M3<DF>& b) {
  M3<DF> c;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      Anchored re, im;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        re.add(a.e[i][k].re, b.e[k][j].re);
        re.sub(a.e[i][k].im, b.e[k][j].im);
        im.add(a.e[i][k].re, b.e[k][j].im);
        im.add(a.e[i][k].im, b.e[k][j].re);
      }
      c.e[i][j] = cx<DF>(re.value(), im.value());
    }
  return c;
}

}  // namespace fg
