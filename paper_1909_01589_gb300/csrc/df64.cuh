// Double-float arithmetic on the FP32 pipe: a value is hi + lo with two
// floats, |lo| <= ulp(hi)/2, about 48 significant bits.
//
// GB300 executes FP64 at 1/69 of its FP32 rate, so the hot loops of the
// projection run in this representation and reach the accuracy FP64 parity
// needs (relative error ~1e-14) at a fraction of the FP64 pipe time.
//
// Methods (all error-free transformations use round-to-nearest FP32 and the
// fused multiply-add; intrinsics __fadd_rn / __fmul_rn keep the compiler
// from contracting or reassociating them):
//   two_sum        Knuth, The Art of Computer Programming vol. 2 (1969)
//   fast_two_sum   Dekker, "A floating-point technique for extending the
//                  available precision", Numer. Math. 18 (1971)
//   two_prod       the FMA form of Dekker's product (exact a*b - fl(a*b))
//   add / mul      the double-float operations of Dekker (1971)
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace lrdmc {

struct df {
  float hi, lo;
};

__host__ __device__ __forceinline__ df df_make(float h, float l)
{
  df r;
  r.hi = h;
  r.lo = l;
  return r;
}

#ifdef __CUDA_ARCH__
#define DF_ADD(a, b) __fadd_rn((a), (b))
#define DF_SUB(a, b) __fsub_rn((a), (b))
#define DF_MUL(a, b) __fmul_rn((a), (b))
#define DF_FMA(a, b, c) __fmaf_rn((a), (b), (c))
#else
#define DF_ADD(a, b) ((a) + (b))
#define DF_SUB(a, b) ((a) - (b))
#define DF_MUL(a, b) ((a) * (b))
#define DF_FMA(a, b, c) fmaf((a), (b), (c))
#endif

// |a| >= |b| (or a == 0): s + e == a + b exactly.
__host__ __device__ __forceinline__ df fast_two_sum(float a, float b)
{
  float s = DF_ADD(a, b);
  float e = DF_SUB(b, DF_SUB(s, a));
  return df_make(s, e);
}

__host__ __device__ __forceinline__ df two_sum(float a, float b)
{
  float s = DF_ADD(a, b);
  float bb = DF_SUB(s, a);
  float e = DF_ADD(DF_SUB(a, DF_SUB(s, bb)), DF_SUB(b, bb));
  return df_make(s, e);
}

__host__ __device__ __forceinline__ df two_prod(float a, float b)
{
  float p = DF_MUL(a, b);
  float e = DF_FMA(a, b, -p);
  return df_make(p, e);
}

__host__ __device__ __forceinline__ df df_neg(df a) { return df_make(-a.hi, -a.lo); }

// Absolute error about 2^-44 (|a| + |b|): one two_sum.
__host__ __device__ __forceinline__ df df_add(df a, df b)
{
  df s = two_sum(a.hi, b.hi);
  float e = DF_ADD(s.lo, DF_ADD(a.lo, b.lo));
  return fast_two_sum(s.hi, e);
}

__host__ __device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, df_neg(b)); }

__host__ __device__ __forceinline__ df df_mul(df a, df b)
{
  df p = two_prod(a.hi, b.hi);
  float e = DF_FMA(a.hi, b.lo, p.lo);
  e = DF_FMA(a.lo, b.hi, e);
  return fast_two_sum(p.hi, e);
}

__host__ __device__ __forceinline__ df df_mul_f(df a, float b)
{
  df p = two_prod(a.hi, b);
  float e = DF_FMA(a.lo, b, p.lo);
  return fast_two_sum(p.hi, e);
}

__host__ __device__ __forceinline__ df df_sqr(df a)
{
  df p = two_prod(a.hi, a.hi);
  float e = DF_FMA(DF_ADD(a.hi, a.hi), a.lo, p.lo);
  return fast_two_sum(p.hi, e);
}

// Constants of the exponential (lean64.cuh): ln2/1024 in two floats and its
// reciprocal.
struct LeanExp {
  float c_hi, c_lo, inv;
};

// Conversions (each touches the FP64 pipe: use them outside inner loops).
__host__ __device__ __forceinline__ df df_from_double(double d)
{
  float h = (float)d;
  float l = (float)(d - (double)h);
  return df_make(h, l);
}

__host__ __device__ __forceinline__ double df_to_double(df a) { return (double)a.hi + (double)a.lo; }

}  // namespace lrdmc
