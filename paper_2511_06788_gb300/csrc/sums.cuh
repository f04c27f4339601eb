// Sums of FP32 terms with the precision and range of an FP64 sum, mostly on the FP32 pipe: GB300
// runs two FP64 additions a clock and SM, and a warp's takes 64 clocks of its scheduler.
#pragma once

#include <cuda_runtime.h>

namespace opevo {

// x in FP64, exactly.  On the device by integer instructions: the conversion instruction runs at
// the FP64 rate; it remains for what is not zero or normal in FP32.
__host__ __device__ __forceinline__ double widen(float x) {
#ifdef __CUDA_ARCH__
  const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
  if (m == 0) return __hiloint2double((int)u, 0);
  if ((m >> 23) - 1u > 253u) return (double)x;
  return __hiloint2double((int)(((m >> 3) + (896u << 20)) | (u & 0x80000000u)), (int)(m << 29));
#else
  return (double)x;
#endif
}

// Additions and products that the compiler does not fuse (host code: -ffp-contract=off).
__host__ __device__ __forceinline__ float add_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
__host__ __device__ __forceinline__ float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}

// a + b rounded; *e is the rounding error, exactly (Knuth's two-sum).
__host__ __device__ __forceinline__ float two_sum(float a, float b, float *e) {
  const float s = add_rn(a, b), t = add_rn(s, -a);
  *e = add_rn(add_rn(a, -add_rn(s, -t)), add_rn(b, -t));
  return s;
}

// A running sum as an unevaluated triple of floats: the rounding errors of h go to m, those of m
// to l (Ogita, Rump and Oishi, "Accurate sum and dot product", 2005: SumK with K = 3), 72 bits,
// where an FP64 sum of n terms has 53 less the roundings of n additions.  The range is that of
// FP32: once a term or a sum is infinite or NaN the error terms are NaN and stay so, finite() is
// false, and the terms have to be added again in FP64.
struct Sum3 {
  float h = 0.f, m = 0.f, l = 0.f;
  __host__ __device__ __forceinline__ void add(float x) {
    float e;
    h = two_sum(h, x, &e);
    m = two_sum(m, e, &e);
    l = add_rn(l, e);
  }
  __host__ __device__ __forceinline__ void add(const Sum3 &o) {
    float e, f, g;
    h = two_sum(h, o.h, &e);
    m = two_sum(m, o.m, &f);  // (beside the line above)
    m = two_sum(m, e, &g);
    l = add_rn(add_rn(l, o.l), add_rn(f, g));
  }
  __host__ __device__ __forceinline__ bool finite() const { return l == l; }
  __host__ __device__ __forceinline__ double value() const {
    return widen(h) + (widen(m) + widen(l));
  }
};

#ifdef __CUDACC__
// The sum of n terms, `stride` apart, in FP64: where a triple is not finite.  A call: inlined into a
// reduction its registers halved the warps in flight (the Gram's reduce 12.6 -> 22 us).
__device__ __noinline__ static double sum64(const float *x, long long stride, int n) {
  double s = 0.0;
#pragma unroll 1
  for (int i = 0; i < n; ++i) s += (double)x[i * stride];
  return s;
}
#endif

// q = a / b in FP32 (0 where b <= 0): the quotient of the leading parts corrected by its remainder,
// exact to about 2^-46 before the last rounding.  False, with no q, where a sum is not finite or
// a, b (2^-80 .. 2^100) or the quotient are so small or large that the remainder could leave the
// FP32 range: the quotient is then for FP64.
__host__ __device__ __forceinline__ bool quotient(const Sum3 &a, const Sum3 &b, float *q) {
  float al, bl;
  const float ah = two_sum(a.h, a.m, &al), bh = two_sum(b.h, b.m, &bl);
  al = add_rn(al, a.l);
  bl = add_rn(bl, b.l);
  if (bh <= 0.f && b.finite()) {
    *q = 0.f;
    return true;
  }
  const float rb = 1.f / bh, p = mul_rn(ah, rb);  // (p is within 2 ulp: its remainder has 25 bits)
  *q = fmaf(add_rn(fmaf(-p, bh, ah), fmaf(-p, bl, al)), rb, p);
  return al == al && bl == bl && ah > 8.27e-25f && ah < 1.26e30f && bh > 8.27e-25f &&
         bh < 1.26e30f && p > 1e-30f && p < 1e30f;
}

}  // namespace opevo
