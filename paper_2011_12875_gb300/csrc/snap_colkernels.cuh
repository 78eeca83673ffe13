// snap_colkernels.cuh -- compute_U (FP32 up to 2J = 9, FP64 up to 5) and the tangent
// of Ulisttot with the layer recursion in registers, one lane per half-matrix column.
//
// Eq. (hysphrecur) of arXiv:2011.12875 builds u_t from u_{t-1}; element
// (ma, mb) only reads elements (ma, mb) and (ma-1, mb) of the previous layer,
// so every column mb evolves on its own:
//   u_t[ma][mb] = sqrt((t-ma)/(t-mb)) conj(a) u_{t-1}[ma][mb]
//               - sqrt(ma/(t-mb))     conj(b) u_{t-1}[ma-1][mb].
// Column mb enters the stored half at layer t = 2 mb, from column mb of layer
// t-1, which is the mirror of column mb-1 of that layer:
//   u_{t-1}[m][mb] = (-1)^(m+mb) conj(u_{t-1}[t-1-m][mb-1]).
// Here one lane carries one column of one neighbour pair through all layers
// (twojmax/2 + 1 lanes per pair, several pairs per warp); the layer loop is
// unrolled at compile time, so the column lives in registers and the seed is
// one warp shuffle per element.  This file is included by one translation
// unit per working precision.
#pragma once
#include <algorithm>
#include <type_traits>

#include "snap_geom.cuh"
#include "snap_internal.h"
#include "snap_neigh.cuh"

namespace snap {
namespace col {

constexpr unsigned kFull = 0xffffffffu;

template <typename R>
struct __align__(2 * sizeof(R)) c2 {
  R re, im;
};

template <typename R>
__device__ __forceinline__ c2<R> mk(R re, R im) {
  c2<R> c;
  c.re = re;
  c.im = im;
  return c;
}

// Compile-time loop B..E (inclusive): f(std::integral_constant<int, k>).
template <int B, int E, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (B <= E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(f);
  }
}

template <typename R>
__device__ __forceinline__ R shfl_up(R v) {
  return __shfl_up_sync(kFull, v, 1);
}

// Lane layout: NC = J2/2 + 1 lanes per pair, P pairs per warp.
template <int J2>
struct Shape {
  static constexpr int NC = J2 / 2 + 1;
  static constexpr int P = 32 / NC;
};

// ------------------------------------------- scaled layer recursion
// With u_t[ma][mb] = S_t(ma, mb) v_t[ma][mb], S_t(ma, mb) =
// sqrt((t - ma)! ma! / (t - mb)!), the recursion of Eq. (hysphrecur) becomes
//   v_t[ma] = conj(a) v_{t-1}[ma] - conj(b) v_{t-1}[ma-1]
// (S_t(ma, mb) = sqrt((t-ma)/(t-mb)) S_{t-1}(ma, mb) = sqrt(ma/(t-mb))
// S_{t-1}(ma-1, mb) absorbs both root factors): 8 real operations an element
// instead of 12.  S splits into sqrt((t - ma)! ma!), a constant of the
// unrolled element, and 1 / sqrt((t - mb)!), one value per lane and layer.
// The mirror that seeds column mc at layer 2 mc - 1 picks up S's ratio
// between the two columns, 1 / sqrt(mc).
__host__ __device__ constexpr double c_fact(int n) { return n <= 1 ? 1.0 : n * c_fact(n - 1); }
__host__ __device__ constexpr double c_sqrt_iter(double x, double y, int k) {
  return k == 0 ? y : c_sqrt_iter(x, 0.5 * (y + x / y), k - 1);
}
// square root of x >= 1 by Newton's iteration from x (64 steps: converged
// for every argument below 2^64)
__host__ __device__ constexpr double c_sqrt(double x) { return x <= 1.0 ? 1.0 : c_sqrt_iter(x, x, 64); }
template <int T, int MA>
__host__ __device__ constexpr double v_scale() { return c_sqrt(c_fact(T - MA) * c_fact(MA)); }

// x * y + z, one rounding (the sums below are written as chains of these:
// a component of a complex multiply-add is two fused operations, where
// x += a*b + c*d would round a product, a fused sum and an addition)
template <typename R>
__device__ __forceinline__ R fm(R x, R y, R z) {
  if constexpr (sizeof(R) == 4) return fmaf(x, y, z);
  else return fma(x, y, z);
}

// One layer of the scaled recursion on a lane's column, in place, ma
// descending; A = conj(a), B = conj(b).  An element is four fused
// multiply-adds a component.
template <typename R, int T, int N>
__device__ __forceinline__ void v_layer(c2<R> (&v)[N], const c2<R> A, const c2<R> B) {
  static_assert(T < N, "column too short");
  c2<R> w = mk<R>(fm(B.im, v[T - 1].im, -(B.re * v[T - 1].re)), fm(-B.im, v[T - 1].re, -(B.re * v[T - 1].im)));
  v[T] = w;
#pragma unroll
  for (int ma = T - 1; ma >= 1; --ma) {
    const c2<R> x = v[ma], y = v[ma - 1];
    w.re = fm(B.im, y.im, fm(-B.re, y.re, fm(-A.im, x.im, A.re * x.re)));
    w.im = fm(-B.im, y.re, fm(-B.re, y.im, fm(A.im, x.re, A.re * x.im)));
    v[ma] = w;
  }
  v[0] = mk<R>(fm(-A.im, v[0].im, A.re * v[0].re), fm(A.im, v[0].re, A.re * v[0].im));
}

// Seed of column T / 2 (lanes with take) for layer T - 1 in the scaled form:
// the mirror of the column one lane below, times 1 / sqrt(T / 2).
template <typename R, int T, int N>
__device__ __forceinline__ void v_seed(c2<R> (&v)[N], bool take) {
  constexpr int mc = T / 2;
  constexpr double qd = 1.0 / c_sqrt(double(mc));
  const R q = R(qd);
  c2<R> src[T];
#pragma unroll
  for (int k = 0; k < T; ++k) {
    src[k].re = shfl_up(v[k].re);
    src[k].im = shfl_up(v[k].im);
  }
  if (take) {
#pragma unroll
    for (int m = 0; m < T; ++m) {
      const R sq = (((T - 1 - m) + (mc - 1)) & 1) ? -q : q;
      v[m] = mk<R>(sq * src[T - 1 - m].re, -sq * src[T - 1 - m].im);
    }
  }
}

// ------------------------------------------------------------- compute_U
// An atom's pairs are taken in passes of P pairs (a lane per column of a
// pair); f_c u_t of a pass is summed over its pair groups in two steps:
//  * LV levels of shuffles first add the groups g, g + 1, ..., g + 2^LV - 1
//    on the lanes of group g (a multiple of 2^LV), which leaves
//    CPW = ceil(P / 2^LV) partial sums of each element;
//  * those lanes store their partial sums (CPW copies of the half matrix) in
//    the warp's scratch, and after the pass each lane adds the copies of the
//    elements e = lane, lane + 32, ... to the warp's running sum.
// LV is the fewest levels that keep the scratch under 4 KB in FP32 (2J = 8:
// one level, three copies) and none in FP64, whose pipe, not the shuffles'
// latency, bounds that path.  Q warps share an atom (warp q takes passes q,
// q + Q, ...), and the atom's Ulisttot is the sum of the Q running sums plus
// w_self on the diagonal.  Q, LV and P are constants of the instance, so the
// order of every sum is fixed by the slot indices alone.
template <typename R, int J2>
struct UiPlan {
  static constexpr int NC = Shape<J2>::NC, P = Shape<J2>::P;
  static constexpr int HH = half_size(J2);
  static constexpr int kMaxLv = P > 16 ? 5 : P > 8 ? 4 : P > 4 ? 3 : P > 2 ? 2 : P > 1 ? 1 : 0;
  static constexpr int copies(int lv) { return (P + (1 << lv) - 1) >> lv; }
  static constexpr int pick(int lv) {
    return (sizeof(R) == 8 || lv >= kMaxLv || copies(lv) * HH * (int)sizeof(c2<R>) <= 4096) ? lv : pick(lv + 1);
  }
  static constexpr int LV = pick(0);
  static constexpr int CPW = copies(LV);
  static constexpr int Q = (26 + P - 1) / P >= 2 ? 2 : 1;  // warps per atom
  static constexpr int A = Q == 1 ? 2 : 1;                  // atoms per CTA
  static constexpr size_t warp_bytes = sizeof(c2<R>) * (size_t)(CPW + 1) * HH;
};

// Sum of v over the pair groups g, g + 1, ..., g + 2^LV - 1 (on the lanes of
// writer groups; lanes past the warp add nothing).
template <int LV, int NC, typename R>
__device__ __forceinline__ R group_sum(R v, int lane) {
#pragma unroll
  for (int l = 0; l < LV; ++l) {
    const R o = __shfl_down_sync(kFull, v, NC << l);
    if (lane + (NC << l) < 32) v += o;
  }
  return v;
}

// The passes of one warp of an atom (warp wq of its Q): abf = the atom's
// [K][5] (a, b, f_c) in shared memory, scr = the warp's [CPW + 1][H] scratch
// (CPW partial sums of a pass, then the warp's running sum).
template <typename R, int J2>
__device__ __forceinline__ void u_passes(const R* __restrict__ abf, int cnt, int wq, int lane,
                                         c2<R>* __restrict__ scr) {
  using S = Shape<J2>;
  using UP = UiPlan<R, J2>;
  constexpr int NC = S::NC, P = S::P, LV = UP::LV, CPW = UP::CPW, Q = UP::Q, H = UP::HH;
  c2<R>* run = scr + (size_t)CPW * H;
  for (int e = lane; e < H; e += 32) run[e] = mk<R>(0, 0);
  const int g = lane / NC, mb = lane - g * NC;
  const bool grp = g < P;
  const bool writer = grp && (g & ((1 << LV) - 1)) == 0;
  c2<R>* my = scr + (size_t)(writer ? (g >> LV) : 0) * H;
  const int npass = (cnt + P - 1) / P;
  for (int pass = wq; pass < npass; pass += Q) {
    const int s = pass * P + g;
    const bool ok = grp && s < cnt;
    c2<R> ca = mk<R>(1, 0), cb = mk<R>(0, 0);
    R fc = 0;
    if (ok) {
      const R* gm = abf + 5 * s;
      ca = mk<R>(gm[0], -gm[1]);  // conj(a)
      cb = mk<R>(gm[2], -gm[3]);  // conj(b)
      fc = gm[4];
    }
    // the scaled column times f_c (the recursion is linear, so f_c rides
    // along from layer 0); S is applied once, to the atom's sums
    c2<R> v[J2 + 1];
#pragma unroll
    for (int k = 0; k <= J2; ++k) v[k] = mk<R>(0, 0);
    if (mb == 0) v[0] = mk<R>(fc, 0);
    {
      const R v0 = group_sum<LV, NC>(v[0].re, lane);
      if (writer && mb == 0) my[0] = mk<R>(v0, 0);
    }
    static_for<1, J2>([&](auto tc) {
      constexpr int t = decltype(tc)::value;
      if constexpr ((t & 1) == 0) v_seed<R, t>(v, mb == t / 2);
      v_layer<R, t>(v, ca, cb);
      c2<R>* dst = my + half_base(t) + mb * (t + 1);
#pragma unroll
      for (int ma = 0; ma <= t; ++ma) {
        const R vr = group_sum<LV, NC>(v[ma].re, lane);
        const R vi = group_sum<LV, NC>(v[ma].im, lane);
        if (writer && 2 * mb <= t) dst[ma] = mk<R>(vr, vi);
      }
    });
    __syncwarp();
    for (int e = lane; e < H; e += 32) {
      c2<R> v = run[e];
#pragma unroll
      for (int c = 0; c < CPW; ++c) {
        const c2<R> w = scr[(size_t)c * H + e];
        v.re += w.re;
        v.im += w.im;
      }
      run[e] = v;
    }
    __syncwarp();
  }
}

// Ulisttot of atom i from its Q warps' running sums (ascr = the atom's
// [Q][CPW + 1][H] scratch): their sum in warp order, times S, plus w_self on
// the diagonal; elements e0, e0 + estride, ...
template <typename R, int J2>
__device__ __forceinline__ void u_store(const WorkArgs& a, const c2<R>* __restrict__ ascr, long i, int e0,
                                        int estride) {
  using UP = UiPlan<R, J2>;
  constexpr int CPW = UP::CPW, Q = UP::Q, H = UP::HH;
  c2<R>* Ug = reinterpret_cast<c2<R>*>(a.U);
  for (int e = e0; e < H; e += estride) {
    const c2<R>* rr = ascr + (size_t)CPW * H + e;
    R sr = 0, si = 0;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const c2<R> v = rr[(size_t)q * (CPW + 1) * H];
      sr += v.re;
      si += v.im;
    }
    const R sc = reinterpret_cast<const R*>(a.hscale)[e];
    sr *= sc;
    si *= sc;
    const int p = a.half_tmm[e];
    if (tmm_ma(p) == tmm_mb(p)) sr += (R)a.wself;
    Ug[((i >> 5) * H + e) * 32 + (i & 31)] = mk<R>(sr, si);
  }
}

// Resident CTAs an SM the register allocation is sized for: 16 two-warp CTAs
// (64 registers) in FP32 up to 2J = 8, 8 above and in FP64.
template <typename R, int J2>
constexpr int ui_min_ctas() { return sizeof(R) == 8 ? 8 : (J2 <= 8 ? 16 : 8); }

// compute_U for a neighbour table built elsewhere (caller-supplied lists):
// CTA = A atoms of Q warps; the atom's first warp evaluates the slot
// geometry from the stored separations (dense lanes), then the passes.
template <typename R, int J2>
__global__ void __launch_bounds__(64, ui_min_ctas<R, J2>()) ui_col_kernel(WorkArgs a) {
  using UP = UiPlan<R, J2>;
  constexpr int Q = UP::Q, A = UP::A;
  extern __shared__ __align__(16) unsigned char smem[];
  const int K = a.K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int al = warp / Q, wq = warp - al * Q;
  const long i0 = (long)blockIdx.x * A;
  const long i = i0 + al;
  const bool have = i < a.n;  // warp-uniform
  c2<R>* scr = reinterpret_cast<c2<R>*>(smem) + (size_t)warp * (UP::CPW + 1) * UP::HH;
  R* myabf = reinterpret_cast<R*>(smem + (size_t)A * Q * UP::warp_bytes) + (size_t)al * K * 5;
  const int cnt = have ? a.cnt[i] : 0;
  if (have && wq == 0)
    for (int s = lane; s < cnt; s += 32) geo::slot_geom<R>(a, i * K + s, myabf + 5 * s);
  __syncthreads();
  if (have) u_passes<R, J2>(myabf, cnt, wq, lane, scr);
  __syncthreads();
  for (int a2 = 0; a2 < A; ++a2) {
    if (i0 + a2 >= a.n) break;
    u_store<R, J2>(a, reinterpret_cast<const c2<R>*>(smem) + (size_t)a2 * Q * (UP::CPW + 1) * UP::HH, i0 + a2,
                   threadIdx.x, blockDim.x);
  }
}

// ---------------------------------------- neighbour build fused with compute_U
// The neighbour build of snap_neigh.cuh (two atoms a CTA, SPLIT warps each)
// and, in the same CTA, compute_U of those atoms: each stored pair's slot
// geometry is evaluated on the lane that accepts it, from the exact FP64
// separation in its registers (dense lanes, no reload), with a, b and f_c
// kept in shared memory; then the first Q warps of each atom take its
// passes.  One launch and one pass over the pairs instead of two.
template <bool BATCH>
struct NuShape {
  static constexpr int SPLIT = BATCH ? 4 : 2;  // build warps per atom
  static constexpr int NW = 2 * SPLIT;         // warps per CTA (two atoms)
};

template <typename R, int J2, bool BATCH>
__global__ void __launch_bounds__(NuShape<BATCH>::NW * 32) neigh_u_kernel(NeighArgs na, WorkArgs a) {
  using UP = UiPlan<R, J2>;
  constexpr int SPLIT = NuShape<BATCH>::SPLIT, NW = NuShape<BATCH>::NW, Q = UP::Q;
  static_assert(Q <= SPLIT, "an atom's passes run on its build warps");
  extern __shared__ __align__(16) unsigned char smem[];
  const int K = a.K;
  R* abf = reinterpret_cast<R*>(smem + (size_t)2 * Q * UP::warp_bytes);  // [2][K][5]
  nb::neigh_build_cta<BATCH, SPLIT, NW>(na, [&](int al, long i, int slot, long q, double ex, double ey,
                                               double ez) {
    (void)i;
    geo::pair_geom<R>(a, q, ex, ey, ez, abf + ((size_t)al * K + slot) * 5);
  });
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int al = warp / SPLIT, wq = warp - al * SPLIT;
  long i, hi;
  if (BATCH) {
    const int2 m = na.cta_map[blockIdx.x];
    const NeighConf c = na.confs[m.x];
    i = c.start + m.y + al;
    hi = c.start + c.n;
  } else {
    i = (long)blockIdx.x * 2 + al;
    hi = na.n;
  }
  const bool have = i < hi;
  c2<R>* ascr = reinterpret_cast<c2<R>*>(smem) + (size_t)al * Q * (UP::CPW + 1) * UP::HH;
  if (have && wq < Q)
    u_passes<R, J2>(abf + (size_t)al * K * 5, min(na.cnt[i], K), wq, lane,
                    ascr + (size_t)wq * (UP::CPW + 1) * UP::HH);
  __syncthreads();
  if (have) u_store<R, J2>(a, ascr, i, wq * 32 + lane, SPLIT * 32);
}

// ------------------------------------------- tangent of Ulisttot along g
// Forward-mode derivative of Eq. (u) along a displacement field g of the
// atoms: the pair (i, k) moves by delta = g_k - g_i, so
//   dU_t = sum_k d/de [ f_c(r_ik + e delta) u_t(r_ik + e delta) ] at e = 0
//        = sum_k (grad f_c . delta) u_t + f_c (du_t/dr . delta).
// In the scaled form w = f_c v (u = S v): w_t = conj(a) w_{t-1}[ma] -
// conj(b) w_{t-1}[ma-1] from w_0 = f_c, and its tangent
//   dw_t = conj(da) w[ma] + conj(a) dw[ma] - conj(db) w[ma-1] - conj(b) dw[ma-1]
// from dw_0 = grad f_c . delta, so dU_t = S sum_k dw_t (no w_self).  Launch
// shape, reduction and order of the sums as compute_U (UiPlan).
template <typename R, int J2>
__device__ __forceinline__ void du_passes(const R* __restrict__ tg, int cnt, int wq, int lane,
                                          c2<R>* __restrict__ scr) {
  using S = Shape<J2>;
  using UP = UiPlan<R, J2>;
  constexpr int NC = S::NC, P = S::P, LV = UP::LV, CPW = UP::CPW, Q = UP::Q, H = UP::HH;
  c2<R>* run = scr + (size_t)CPW * H;
  for (int e = lane; e < H; e += 32) run[e] = mk<R>(0, 0);
  const int g = lane / NC, mb = lane - g * NC;
  const bool grp = g < P;
  const bool writer = grp && (g & ((1 << LV) - 1)) == 0;
  c2<R>* my = scr + (size_t)(writer ? (g >> LV) : 0) * H;
  const int npass = (cnt + P - 1) / P;
  for (int pass = wq; pass < npass; pass += Q) {
    const int s = pass * P + g;
    const bool ok = grp && s < cnt;
    c2<R> ca = mk<R>(1, 0), cb = mk<R>(0, 0), cda = mk<R>(0, 0), cdb = mk<R>(0, 0);
    R fc = 0, dfc = 0;
    if (ok) {  // [10]: a, b, f_c, d f_c, da, db along delta
      const R* t = tg + 10 * s;
      ca = mk<R>(t[0], -t[1]);
      cb = mk<R>(t[2], -t[3]);
      fc = t[4];
      dfc = t[5];
      cda = mk<R>(t[6], -t[7]);
      cdb = mk<R>(t[8], -t[9]);
    }
    c2<R> w[J2 + 1], dw[J2 + 1];
#pragma unroll
    for (int k = 0; k <= J2; ++k) w[k] = dw[k] = mk<R>(0, 0);
    if (mb == 0) {
      w[0] = mk<R>(fc, 0);
      dw[0] = mk<R>(dfc, 0);
    }
    {
      const R v0 = group_sum<LV, NC>(dw[0].re, lane);
      if (writer && mb == 0) my[0] = mk<R>(v0, 0);
    }
    static_for<1, J2>([&](auto tc) {
      constexpr int t = decltype(tc)::value;
      if constexpr ((t & 1) == 0) {
        v_seed<R, t>(w, mb == t / 2);
        v_seed<R, t>(dw, mb == t / 2);
      }
      // dw first (it reads the old w), then w
#pragma unroll
      for (int ma = t; ma >= 0; --ma) {
        c2<R> y = mk<R>(0, 0);
        if (ma < t) {
          const c2<R> p = w[ma], q = dw[ma];
          y.re = fm(-ca.im, q.im, fm(ca.re, q.re, fm(-cda.im, p.im, fm(cda.re, p.re, y.re))));
          y.im = fm(ca.im, q.re, fm(ca.re, q.im, fm(cda.im, p.re, fm(cda.re, p.im, y.im))));
        }
        if (ma > 0) {
          const c2<R> p = w[ma - 1], q = dw[ma - 1];
          y.re = fm(cb.im, q.im, fm(-cb.re, q.re, fm(cdb.im, p.im, fm(-cdb.re, p.re, y.re))));
          y.im = fm(-cb.im, q.re, fm(-cb.re, q.im, fm(-cdb.im, p.re, fm(-cdb.re, p.im, y.im))));
        }
        dw[ma] = y;
      }
      v_layer<R, t>(w, ca, cb);
      c2<R>* dst = my + half_base(t) + mb * (t + 1);
#pragma unroll
      for (int ma = 0; ma <= t; ++ma) {
        const R vr = group_sum<LV, NC>(dw[ma].re, lane);
        const R vi = group_sum<LV, NC>(dw[ma].im, lane);
        if (writer && 2 * mb <= t) dst[ma] = mk<R>(vr, vi);
      }
    });
    __syncwarp();
    for (int e = lane; e < H; e += 32) {
      c2<R> v = run[e];
#pragma unroll
      for (int c = 0; c < CPW; ++c) {
        const c2<R> q = scr[(size_t)c * H + e];
        v.re += q.re;
        v.im += q.im;
      }
      run[e] = v;
    }
    __syncwarp();
  }
}

template <typename R, int J2>
__global__ void __launch_bounds__(64, ui_min_ctas<R, J2>()) tan_col_kernel(WorkArgs a, const double* __restrict__ gd,
                                                                         void* dUout) {
  using UP = UiPlan<R, J2>;
  constexpr int Q = UP::Q, A = UP::A, CPW = UP::CPW, H = UP::HH;
  extern __shared__ __align__(16) unsigned char smem[];
  const int K = a.K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int al = warp / Q, wq = warp - al * Q;
  const long i0 = (long)blockIdx.x * A;
  const long i = i0 + al;
  const bool have = i < a.n;  // warp-uniform
  c2<R>* scr = reinterpret_cast<c2<R>*>(smem) + (size_t)warp * (CPW + 1) * H;
  R* tg = reinterpret_cast<R*>(smem + (size_t)A * Q * UP::warp_bytes) + (size_t)al * K * 10;
  const int cnt = have ? a.cnt[i] : 0;
  if (have && wq == 0)  // the pair data along delta = g_k - g_i, a lane per slot
    for (int s = lane; s < cnt; s += 32) {
      const long slot = i * K + s;
      const R* gm = reinterpret_cast<const R*>(a.geom) + slot * kGeomStride;
      const int k = a.nbr[slot];
      R dl[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) dl[d] = (R)(gd[3 * (long)k + d] - gd[3 * i + d]);
      R dfc = 0, ar = 0, ai = 0, br = 0, bi = 0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        dfc += dl[d] * gm[5 + d];
        ar += dl[d] * gm[8 + 2 * d];
        ai += dl[d] * gm[9 + 2 * d];
        br += dl[d] * gm[14 + 2 * d];
        bi += dl[d] * gm[15 + 2 * d];
      }
      R* t = tg + 10 * s;
      t[0] = gm[0];
      t[1] = gm[1];
      t[2] = gm[2];
      t[3] = gm[3];
      t[4] = gm[4];
      t[5] = dfc;
      t[6] = ar;
      t[7] = ai;
      t[8] = br;
      t[9] = bi;
    }
  __syncthreads();
  if (have) du_passes<R, J2>(tg, cnt, wq, lane, scr);
  __syncthreads();
  c2<R>* Ug = reinterpret_cast<c2<R>*>(dUout);
  for (int a2 = 0; a2 < A; ++a2) {
    const long ii = i0 + a2;
    if (ii >= a.n) break;
    const c2<R>* rr = reinterpret_cast<const c2<R>*>(smem) + (size_t)a2 * Q * (CPW + 1) * H + (size_t)CPW * H;
    for (int e = threadIdx.x; e < H; e += blockDim.x) {
      R sr = 0, si = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const c2<R> v = rr[(size_t)q * (CPW + 1) * H + e];
        sr += v.re;
        si += v.im;
      }
      const R sc = reinterpret_cast<const R*>(a.hscale)[e];
      Ug[((ii >> 5) * H + e) * 32 + (ii & 31)] = mk<R>(sr * sc, si * sc);
    }
  }
}

template <typename R, int J2>
cudaError_t launch_ui_col_t(const WorkArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  using UP = UiPlan<R, J2>;
  if (a.H != UP::HH) return cudaErrorInvalidValue;
  const size_t smem = (size_t)UP::A * (UP::Q * UP::warp_bytes + sizeof(R) * 5 * (size_t)a.K);
  cudaError_t e = allow_smem(ui_col_kernel<R, J2>, smem);
  if (e != cudaSuccess) return e;
  return launch_k(ui_col_kernel<R, J2>, dim3((unsigned)((a.n + UP::A - 1) / UP::A)), dim3(UP::A * UP::Q * 32),
                  smem, s, a);
}

// Fused neighbour build + compute_U: single configuration (ncta = 0: two
// atoms a CTA in order) or a batch (ncta CTAs of na.cta_map).
template <typename R, int J2>
cudaError_t launch_neigh_u_t(const NeighArgs& na, const WorkArgs& a, int ncta, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  using UP = UiPlan<R, J2>;
  if (a.H != UP::HH) return cudaErrorInvalidValue;
  const size_t smem = (size_t)2 * (UP::Q * UP::warp_bytes + sizeof(R) * 5 * (size_t)a.K);
  if (ncta > 0) {
    cudaError_t e = allow_smem(neigh_u_kernel<R, J2, true>, smem);
    if (e != cudaSuccess) return e;
    return launch_k(neigh_u_kernel<R, J2, true>, dim3((unsigned)ncta), dim3(NuShape<true>::NW * 32), smem, s, na,
                    a);
  }
  cudaError_t e = allow_smem(neigh_u_kernel<R, J2, false>, smem);
  if (e != cudaSuccess) return e;
  return launch_k(neigh_u_kernel<R, J2, false>, dim3((unsigned)((a.n + 1) / 2)), dim3(NuShape<false>::NW * 32),
                  smem, s, na, a);
}

template <typename R, int J2>
cudaError_t launch_tan_col_t(const WorkArgs& a, const double* g, void* dU, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  using UP = UiPlan<R, J2>;
  if (a.H != UP::HH) return cudaErrorInvalidValue;
  const size_t smem = (size_t)UP::A * (UP::Q * UP::warp_bytes + sizeof(R) * 10 * (size_t)a.K);
  cudaError_t e = allow_smem(tan_col_kernel<R, J2>, smem);
  if (e != cudaSuccess) return e;
  return launch_k(tan_col_kernel<R, J2>, dim3((unsigned)((a.n + UP::A - 1) / UP::A)), dim3(UP::A * UP::Q * 32),
                  smem, s, a, g, dU);
}

}  // namespace col
}  // namespace snap
