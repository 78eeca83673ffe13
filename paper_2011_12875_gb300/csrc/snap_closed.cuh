// snap_closed.cuh -- what compute_U (snap_u.cu) and the fused dE (snap_pairs.cuh)
// share of the closed form of u: U and dE belong together only if a pair's
// polynomials are the same in both.
#pragma once
#include <cmath>

#include "snap_internal.h"

namespace snap {
namespace pr {

// the arithmetic of a pair is the host walk's too (snap_pair_host)
#define SNAP_HD __host__ __device__ __forceinline__

template <typename R>
struct __align__(2 * sizeof(R)) r2 {
  R x, y;
};
// alpha_k, beta_k of a step.  Their rounding is the same for every pair, so its
// effect adds up over them, where the rest of a pair's rounding averages out.
// FP64 takes them rounded to FP32 and turns the weighted Y, once an atom, into
// the coefficients in the polynomials that those give (fix_class).  The error
// that all pairs share, of the size of S, 2J8 / 2J11 / 2J14, in units of 2^-53:
// 0.7 each, which is the scales' and Y's own rounding; rounded to FP64 and left
// so 0.8 / 1.1 / 1.4 (tests/test_pair_closed_form.py).  It takes 1% of a step.
// FP32: with the part that their rounding leaves off, z and w, at four operations
// a step.  Mean error of the virial over 24 inputs, layer recursion / closed form
// with z and w rounded away again (as it was) / now: 2J8 2000 atoms 2.2e-7 / 1.9e-7 /
// 1.6e-7, 2J10 432 atoms 5.0e-7 / 4.2e-7 / 3.0e-7, 2J14 250 atoms 8.1e-7 / 7.9e-7 /
// 3.6e-7.
template <typename R>
struct rec_ab;
template <>
struct __align__(16) rec_ab<float> {
  float x, y, z, w;
};
template <>
struct __align__(16) rec_ab<double> {
  double x, y;
};

// The scale of a step, in FP32 with what its rounding leaves off: that, too, is the
// same for every atom.
template <typename R>
struct step_scale;
template <>
struct __align__(8) step_scale<float> {
  float x, y;
};
template <>
struct step_scale<double> {
  double x;
};

// x * y + z in one rounding, also where the compiler would split it
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float fm(float x, float y, float z) { return __fmaf_rn(x, y, z); }
__device__ __forceinline__ double fm(double x, double y, double z) { return __fma_rn(x, y, z); }
#else
__host__ __device__ inline float fm(float x, float y, float z) { return std::fma(x, y, z); }
__host__ __device__ inline double fm(double x, double y, double z) { return std::fma(x, y, z); }
#endif

// alpha x + beta.  FP32: the remainders' part goes into the first rounding; added
// to a rounded alpha x + beta, less than half of whose last place it is, it would
// be rounded away.
SNAP_HD float rec_t(const rec_ab<float>& c, float x) { return fm(c.x, x, fm(c.z, x, c.w)) + c.y; }
SNAP_HD double rec_t(const rec_ab<double>& c, double x) { return fm(c.x, x, c.y); }
// t d1 + alpha p - d0
SNAP_HD float rec_d(const rec_ab<float>& c, float t, float d1, float p, float d0) {
  return fm(c.x, p, fm(t, d1, c.z * p)) - d0;
}
SNAP_HD double rec_d(const rec_ab<double>& c, double t, double d1, double p, double d0) {
  return fm(t, d1, fm(c.x, p, -d0));
}

SNAP_HD float scaled(step_scale<float> c, float v) { return fm(c.x, v, c.y * v); }
SNAP_HD double scaled(step_scale<double> c, double v) { return c.x * v; }

// v * b + c (complex)
template <typename R>
SNAP_HD r2<R> cfma(r2<R> v, r2<R> b, r2<R> c) {
  r2<R> o;
  o.x = fm(-v.y, b.y, fm(v.x, b.x, c.x));
  o.y = fm(v.y, b.x, fm(v.x, b.y, c.y));
  return o;
}
template <typename R>
SNAP_HD r2<R> cmul(r2<R> v, r2<R> b) {
  r2<R> o;
  o.x = fm(-v.y, b.y, v.x * b.x);
  o.y = fm(v.y, b.x, v.x * b.y);
  return o;
}

}  // namespace pr
}  // namespace snap
