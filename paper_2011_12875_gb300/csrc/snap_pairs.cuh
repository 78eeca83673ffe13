// snap_pairs.cuh -- fused dU + dE/dr with u in closed form, one lane per
// neighbour pair.
//
// A Wigner matrix element of rank t = 2j is a monomial of the Cayley-Klein
// parameters times a real Jacobi polynomial of x = |a|^2 - |b|^2 (Wigner's
// d-matrix formula).  The elements with ma + mb <= t (the others follow from
// the inversion symmetry) are, with p = t - ma - mb, q = |mb - ma| and
// k = min(ma, mb), so t = p + q + 2k,
//   u_t[k][k+q] = n conj(a)^p b^q pi_k(x),   u_t[k+q][k] = n conj(a)^p (-conj(b))^q pi_k(x),
//   n = t! / (2^k sqrt((t-ma)! ma! (t-mb)! mb!)),
// with pi_k the monic polynomial P_k^(q,p).  For a class (p, q) the rising k
// is a three-term recursion in real numbers,
//   P_0 = 1, P_1 = alpha_0 x + beta_0, P_{k+1} = (alpha_k x + beta_k) P_k - P_{k-1},
// pi_k = s_k P_k (HostTables::pair_*: n s_k is folded into the weighted Y, so
// alpha, beta and the scale are the only tables).
//
// For one pair S(a, b) = Re sum_t Y_t : conj(u_t), so with Yw the weighted,
// scaled Y of the two elements of (p, q, k),
//   S = Re sum_p a^p sum_q [ conj(b)^q sum_k Yw+ P_k(x) + (-b)^q sum_k Yw- P_k(x) ],
// and its derivatives in a, conj(b), -b and x come from the same sums with
// P_k' and from Horner's scheme in q.  Then
//   dE_i/dr_ik = S grad f_c + f_c (<g_a, da/dr> + <g_b, db/dr>)   (Eq. snapforce2),
// g_a with the part of x: dx = 4 Re(conj(a) da) on the sphere |a|^2 + |b|^2 = 1.
//
// What bounds it and why this form: the layer recursion and its adjoint pass
// (the form before) took 26 multiply-adds an element with a lane per column, 31%
// of the lanes idle on the half-matrix triangle, and kept every layer in shared
// memory.  Here an element takes 4 multiply-adds for its part of the value and
// the x-derivative, a share of the polynomials' 4 a step (the two elements of a
// step use the same ones) and of Horner's scheme (24 a class): about 1,450 a
// pair at 2J8 against 4,030, every lane a pair.  FP64 is bound by the FP64 pipe
// either way; FP32 by the latency of about three warps a scheduler.  Measured,
// 2000 atoms of 26 neighbours, before -> now: 2J8 FP64 725 -> 141 us, 2J14 FP64
// 2850 -> 512, 2J8 FP32 37 -> 12.7, 2J14 FP32 137 -> 28.1 (16000 atoms: 1094 ->
// 197); 128 atoms at 2J8 FP64 74 -> 27.
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

#include "snap_closed.cuh"
#include "snap_internal.h"

namespace snap {
namespace pr {

constexpr unsigned kFull = 0xffffffffu;

// the two elements of (p, q, k): re and im of the b^q one, re and im of the
// (-conj b)^q one
template <typename R>
struct __align__(16) y4 {
  R pr, pi, mr, mi;
};

// steps (p, q, k) of the classes with p' < p: a class of remainder
// r = 2J - p - q has r / 2 + 1 steps, stored p rising, then r rising
__host__ __device__ constexpr int steps_of(int m) { return (m + 2) * (m + 2) / 4; }  // sum over r = 0..m
__host__ __device__ constexpr int steps_before(int J2, int p) {
  int s = 0;
  for (int k = 0; k < p; ++k) s += steps_of(J2 - k);
  return s;
}
__host__ __device__ constexpr int steps_total(int J2) { return steps_before(J2, J2 + 1); }
// multiply-adds of the classes of p, for the split of the p range
__host__ __device__ constexpr int cost_of(int J2, int p) {
  int c = 24;
  for (int r = 0; r <= J2 - p; ++r) {
    const int k = r / 2;
    c += (p == 0 || r == J2 - p) ? 12 + 8 * k : 24 + 12 * k;
  }
  return c;
}
// The p range is cut into kParts parts of about equal work, always the same
// ones: a pair's sums are added part by part, whether one warp takes all
// parts or each part has a warp of its own, so no result bit depends on that.
constexpr int kParts = 4;
__host__ __device__ constexpr int part_begin(int J2, int part) {
  long total = 0, run = 0;
  for (int p = 0; p <= J2; ++p) total += cost_of(J2, p);
  for (int p = 0; p <= J2; ++p) {
    // p opens `part` once half of its own work lies past the part's share
    if ((2 * run + cost_of(J2, p)) * kParts >= 2 * total * part) return p;
    run += cost_of(J2, p);
  }
  return J2 + 1;
}

template <typename R>
struct Sums {
  R s, gar, gai, gbr, gbi, x;
};

// The weighted, scaled Y of a step (w: HostTables::pair_idx) from the Y of its
// two elements, at(element) each.
template <typename R, typename F>
SNAP_HD y4<R> weighted_y(unsigned w, step_scale<R> sc, F&& at) {
  const r2<R> u = at(w & 1023u);
  y4<R> v;
  const bool neg = (w >> 11) & 1u, conj = (w >> 10) & 1u;
  v.pr = scaled(sc, neg ? -u.x : u.x);
  v.pi = scaled(sc, neg != conj ? -u.y : u.y);
  v.mr = v.mi = R(0);
  if ((w >> 22) & 1u) {
    const r2<R> m = at((w >> 12) & 1023u);
    v.mr = scaled(sc, m.x);
    v.mi = scaled(sc, m.y);
  }
  return v;
}

// One component (y: its values of the steps, 4 apart) of a class of K steps,
// in place: sum_k Y_k P_k = sum_j (Y_j + sum_{k > j} f_kj Y_k) PP_j, 1 + d_kk being
// in the scale (fix: HostTables::pair_fix from the class's first step on).
template <int K>
SNAP_HD void fix_steps(double* __restrict__ y, const double* __restrict__ fix) {
  double v[K];
#pragma unroll
  for (int j = 0; j < K; ++j) v[j] = y[4 * j];
#pragma unroll
  for (int j = 0; j + 1 < K; ++j) {
#pragma unroll
    for (int i = 1; j + i < K; ++i) v[j] = fm(fix[j * kPairFix + i], v[j + i], v[j]);
    y[4 * j] = v[j];
  }
}
SNAP_HD void fix_class(double* y, const double* fix, int K) {
  switch (K) {
    case 2: return fix_steps<2>(y, fix);
    case 3: return fix_steps<3>(y, fix);
    case 4: return fix_steps<4>(y, fix);
    case 5: return fix_steps<5>(y, fix);
    case 6: return fix_steps<6>(y, fix);
    case 7: return fix_steps<7>(y, fix);
    case 8: return fix_steps<8>(y, fix);
    default: return;
  }
}

// Q = sum_k Y P_k and X = sum_k Y P_k' of a class of K steps, one or both
// elements.
template <typename R, int K, bool BOTH>
SNAP_HD void class_sums(const y4<R>* __restrict__ y, const rec_ab<R>* __restrict__ ab, R x, r2<R>& qp,
                                           r2<R>& qm, r2<R>& xp, r2<R>& xm) {
  qp.x = y[0].pr;
  qp.y = y[0].pi;
  if (BOTH) {
    qm.x = y[0].mr;
    qm.y = y[0].mi;
  }
  R p0 = R(1), p1 = R(1), d0 = R(0), d1 = R(0);
#pragma unroll
  for (int k = 1; k < K; ++k) {
    const rec_ab<R> c = ab[k];
    const R t = rec_t(c, x);
    R p, d;
    if (k == 1) {
      p = t;
      d = c.x;
    } else if (k == 2) {
      p = fm(t, p1, R(-1));
      d = rec_d(c, t, d1, p1, R(0));
    } else {
      p = fm(t, p1, -p0);
      d = rec_d(c, t, d1, p1, d0);
    }
    p0 = p1;
    p1 = p;
    d0 = d1;
    d1 = d;
    const y4<R> v = y[k];
    qp.x = fm(v.pr, p, qp.x);
    qp.y = fm(v.pi, p, qp.y);
    xp.x = k == 1 ? v.pr * d : fm(v.pr, d, xp.x);
    xp.y = k == 1 ? v.pi * d : fm(v.pi, d, xp.y);
    if (BOTH) {
      qm.x = fm(v.mr, p, qm.x);
      qm.y = fm(v.mi, p, qm.y);
      xm.x = k == 1 ? v.mr * d : fm(v.mr, d, xm.x);
      xm.y = k == 1 ? v.mi * d : fm(v.mi, d, xm.y);
    }
  }
}

// Horner state in q of one p: value, derivative and x-derivative of the two
// element kinds.
template <typename R>
struct Horner {
  r2<R> w, d, x, wm, dm, xm;
};

// The classes r = r0, r0 + 1, ... of one p (q = J2 - p - r falling); `last` =
// J2 - p.  BOTH: p > 0 (both elements for q > 0).
template <typename R, int J2, int RR, bool BOTH>
SNAP_HD void q_steps(const y4<R>* __restrict__ y, const rec_ab<R>* __restrict__ ab, R x, r2<R> cb,
                                        r2<R> mb, int last, Horner<R>& h) {
  if constexpr (RR <= J2) {
    constexpr int K = RR / 2 + 1;
    constexpr int at = RR == 0 ? 0 : steps_of(RR - 1);
    r2<R> qp, qm, xp, xm;
    qp = qm = xp = xm = r2<R>{R(0), R(0)};
    const bool end = RR == last;
    if (BOTH && !end) class_sums<R, K, true>(y + at, ab + at, x, qp, qm, xp, xm);
    else class_sums<R, K, false>(y + at, ab + at, x, qp, qm, xp, xm);
    if constexpr (RR == 0) {
      h.w = qp;
      h.d = h.x = r2<R>{R(0), R(0)};
    } else {
      h.d = RR == 1 ? h.w : cfma(h.d, cb, h.w);
      h.w = cfma(h.w, cb, qp);
      if constexpr (RR >= 2) h.x = RR == 2 ? xp : cfma(h.x, cb, xp);
    }
    if (BOTH) {
      // at the end (q = 0) the second element is the first: its sums take the
      // last factor -b and nothing is added
      if constexpr (RR == 0) {
        h.wm = end ? r2<R>{R(0), R(0)} : qm;
        h.dm = h.xm = r2<R>{R(0), R(0)};
      } else {
        h.dm = RR == 1 ? h.wm : cfma(h.dm, mb, h.wm);
        h.wm = cfma(h.wm, mb, qm);
        if constexpr (RR >= 2) h.xm = RR == 2 ? xm : cfma(h.xm, mb, xm);
      }
    }
    if (!end) q_steps<R, J2, RR + 1, BOTH>(y, ab, x, cb, mb, last, h);
  }
}

// The parts [part0, part1) of one pair's sums.
template <typename R, int J2>
SNAP_HD Sums<R> pair_sums(const y4<R>* __restrict__ yat, const rec_ab<R>* __restrict__ abt, r2<R> a,
                                             r2<R> b, int part) {
  // x: the smaller of |a|^2 and |b|^2 from 1 (both carry the rounding of a, b)
  const R na = fm(a.x, a.x, a.y * a.y), nb = fm(b.x, b.x, b.y * b.y);
  const R x = na < nb ? fm(R(2), na, R(-1)) : fm(R(-2), nb, R(1));
  const r2<R> cb = {b.x, -b.y}, mb = {-b.x, -b.y};
  constexpr int B1 = part_begin(J2, 1), B2 = part_begin(J2, 2), B3 = part_begin(J2, 3);
  int p = part == 0 ? 0 : part == 1 ? B1 : part == 2 ? B2 : B3;
  const int pe = part == 0 ? B1 : part == 1 ? B2 : part == 2 ? B3 : J2 + 1;
  constexpr int S1 = steps_before(J2, B1), S2 = steps_before(J2, B2), S3 = steps_before(J2, B3);
  const int s0 = part == 0 ? 0 : part == 1 ? S1 : part == 2 ? S2 : S3;
  const y4<R>* y = yat + s0;
  const rec_ab<R>* ab = abt + s0;
  Sums<R> o = {R(0), R(0), R(0), R(0), R(0), R(0)};
  r2<R> pw = {R(1), R(0)}, pw1 = {R(0), R(0)};  // a^p, a^(p-1)
  for (int k = 0; k < p; ++k) {
    pw1 = pw;
    pw = cmul(pw, a);
  }
  if (p == 0 && pe > 0) {  // one element a class
    Horner<R> h;
    q_steps<R, J2, 0, false>(y, ab, x, cb, mb, J2, h);
    o.s = h.w.x;
    o.gbr = h.d.x;
    o.gbi = h.d.y;
    o.x = h.x.x;
    y += steps_of(J2);
    ab += steps_of(J2);
    pw1 = pw;
    pw = a;
    p = 1;
  }
#pragma unroll 1
  for (; p < pe; ++p) {
    Horner<R> h;
    q_steps<R, J2, 0, true>(y, ab, x, cb, mb, J2 - p, h);
    const r2<R> v = {h.w.x + h.wm.x, h.w.y + h.wm.y}, xx = {h.x.x + h.xm.x, h.x.y + h.xm.y};
    const R pv = R(p), vr = pv * v.x, vi = pv * v.y;
    o.s = fm(-pw.y, v.y, fm(pw.x, v.x, o.s));
    o.x = fm(-pw.y, xx.y, fm(pw.x, xx.x, o.x));
    o.gar = fm(-pw1.y, vi, fm(pw1.x, vr, o.gar));
    o.gai = fm(-pw1.y, vr, fm(-pw1.x, vi, o.gai));
    // Re[D+ conj(db)] + Re[D- (-db)]
    o.gbr = fm(-pw.y, h.d.y - h.dm.y, fm(pw.x, h.d.x - h.dm.x, o.gbr));
    o.gbi = fm(pw.y, h.d.x + h.dm.x, fm(pw.x, h.d.y + h.dm.y, o.gbi));
    y += steps_of(J2 - p);
    ab += steps_of(J2 - p);
    pw1 = pw;
    pw = cmul(pw, a);
  }
  return o;
}

template <typename R>
SNAP_HD void add_sums(Sums<R>& t, const Sums<R>& o) {
  t.s += o.s;
  t.gar += o.gar;
  t.gai += o.gai;
  t.gbr += o.gbr;
  t.gbi += o.gbi;
  t.x += o.x;
}

// component d of dE_i/dr_ik in the working precision (the per-atom force and
// virial sums over pairs are FP64, force_kernel)
template <typename R>
__device__ __forceinline__ double pair_dedr(const R* __restrict__ g, const Sums<R>& q, int d) {
  const R fx = R(4) * q.x;
  R ga = fm(fx, g[0], q.gar), gi = fm(fx, g[1], q.gai);
  // Only the part of (g_a, g_b) tangent to the sphere counts.  da and db are
  // tangent up to their rounding (FP32: a few 1e-7, more near the cutoff),
  // and the radial part of the closed form is several times the tangent one:
  // taken out first, or it brings their rounding in (relative error of a
  // pair's dE/dr in FP32, 2J8 / 2J14: 5.4e-7 / 12e-7 with it, 2.4e-7 / 7e-7
  // without; the layer recursion's 3.9e-7 / 12e-7).
  const R rad = fm(q.gbi, g[3], fm(q.gbr, g[2], fm(gi, g[1], ga * g[0])));
  ga = fm(-rad, g[0], ga);
  gi = fm(-rad, g[1], gi);
  const R br = fm(-rad, g[2], q.gbr), bi = fm(-rad, g[3], q.gbi);
  R ds = ga * g[8 + 2 * d];
  ds = fm(gi, g[9 + 2 * d], ds);
  ds = fm(br, g[14 + 2 * d], ds);
  ds = fm(bi, g[15 + 2 * d], ds);
  return (double)fm(g[5 + d], q.s, g[4] * ds);
}

// CTA = A consecutive atoms (A is a launch parameter, see de_plan); their
// pairs, atom after atom, in batches of 32 (a lane a pair, so only the CTA's
// last batch has idle lanes).  SPLIT = 1: warp w takes batches w, w + NW, ...
// SPLIT = kParts: kParts warps share a batch, one part of the p range each (few
// pairs: the chip has more schedulers than batches).  A pair's arithmetic does
// not depend on any of that.
//
// QUEUE: a persistent launch over a work queue -- a grid of resident CTAs,
// each taking CTA-sized items (A consecutive atoms) from a device counter
// (flags[6], zeroed with the flags by every evaluation) until they run out.
template <typename R>
constexpr int de_max_warps() { return sizeof(R) == 4 ? 16 : 8; }

template <typename R, int J2, int SPLIT, bool QUEUE>
__global__ void __launch_bounds__(de_max_warps<R>() * 32, 1) de_pair_kernel(WorkArgs a, int A) {
  static_assert(SPLIT == 1 || SPLIT == kParts, "all parts on one warp or a warp each");
  constexpr int NS = steps_total(J2);
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ long item_s;
  y4<R>* Yw = reinterpret_cast<y4<R>*>(smem);                              // [A][NS]
  rec_ab<R>* abt = reinterpret_cast<rec_ab<R>*>(Yw + (size_t)A * NS);      // [NS]
  Sums<R>* part_s = reinterpret_cast<Sums<R>*>(abt + NS);                  // [NW][32], SPLIT > 1
  const int nw = blockDim.x >> 5;
  int* coff = reinterpret_cast<int*>(part_s + (SPLIT > 1 ? (size_t)nw * 32 : 0));  // [A+1] first pair of each atom
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int H = a.H;
  const rec_ab<R>* abg = reinterpret_cast<const rec_ab<R>*>(a.pair_ab);
  const step_scale<R>* scg = reinterpret_cast<const step_scale<R>*>(a.pair_scale);
  for (int st = threadIdx.x; st < NS; st += blockDim.x) abt[st] = abg[st];
  const long nitems = (a.n + A - 1) / A;
  for (long item = blockIdx.x;;) {
    if (QUEUE) {
      if (threadIdx.x == 0) item_s = atomicAdd(&a.flags[6], 1);
      __syncthreads();
      item = item_s;
      if (item >= nitems) break;
    }
    const long i0 = item * A;  // the CTA's atoms i0 .. i0 + na - 1
    const int na = (int)min((long)A, a.n - i0);
    // the weighted, scaled Y of every step and atom (atoms fastest: the
    // reads of neighbouring lanes share sectors of the [H][32] blocks)
    for (int k = threadIdx.x; k < NS * na; k += blockDim.x) {
      const int st = k / na, al = k - st * na;
      const long i = i0 + al;
      const r2<R>* Yg = reinterpret_cast<const r2<R>*>(a.Y) + (i >> 5) * (long)H * 32 + (i & 31);
      Yw[(size_t)al * NS + st] = weighted_y<R>(__ldg(a.pair_idx + st), scg[st], [&](unsigned e) { return Yg[e * 32]; });
    }
    if (warp == 0) {  // exclusive offsets of the atoms' pairs (inclusive scan, 32 at a time)
      int carry = 0;
      if (lane == 0) coff[0] = 0;
      for (int b = 0; b < na; b += 32) {
        int c = b + lane < na ? a.cnt[i0 + b + lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int u = __shfl_up_sync(kFull, c, o);
          if (lane >= o) c += u;
        }
        if (b + lane < na) coff[b + lane + 1] = carry + c;
        carry += __shfl_sync(kFull, c, 31);
      }
    }
    __syncthreads();
    if constexpr (sizeof(R) == 8) {  // a thread a component of a class (2% of the pairs' work at 2J14)
      for (int k = threadIdx.x; k < a.npair_cls * na * 4; k += blockDim.x) {
        const int c = __ldg(a.pair_cls + k / (4 * na)), st = c & 0xFFFF, al = (k >> 2) % na;
        fix_class(reinterpret_cast<double*>(Yw + (size_t)al * NS + st) + (k & 3), a.pair_fix + st * kPairFix, c >> 16);
      }
      __syncthreads();
    }
    const int total = coff[na];
    const int per = nw / SPLIT;  // batches in flight
    const int nbatch = (total + 31) / 32;
    for (int b0 = 0; b0 < nbatch; b0 += per) {  // CTA-uniform
      const int bt = b0 + warp / SPLIT;
      const bool mine = bt < nbatch;  // warp-uniform
      if (SPLIT == 1 && !mine) break;
      const int f = bt * 32 + lane;
      const bool ok = f < total;
      // the pair's atom: the last al with coff[al] <= f (empty atoms skipped)
      const int fk = min(f, total - 1);
      int lo = 0, hi = na - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (coff[mid] <= fk) lo = mid;
        else hi = mid - 1;
      }
      const long slot = (i0 + lo) * a.K + (fk - coff[lo]);
      const R* gm = reinterpret_cast<const R*>(a.geom) + slot * kGeomStride;
      const r2<R>* g2 = reinterpret_cast<const r2<R>*>(gm);
      Sums<R> q;
      if (mine) {
        const r2<R> ka = g2[0], kb = g2[1];
        const y4<R>* yat = Yw + (size_t)lo * NS;
        if (SPLIT == 1) {
          q = Sums<R>{R(0), R(0), R(0), R(0), R(0), R(0)};
#pragma unroll 1
          for (int part = 0; part < kParts; ++part) add_sums(q, pair_sums<R, J2>(yat, abt, ka, kb, part));
        } else {
          q = pair_sums<R, J2>(yat, abt, ka, kb, warp % SPLIT);
          part_s[warp * 32 + lane] = q;
        }
      }
      if (SPLIT == 1) {
        if (ok) {
#pragma unroll
          for (int d = 0; d < 3; ++d) a.dedr[slot * 3 + d] = pair_dedr<R>(gm, q, d);
        }
      } else {
        __syncthreads();
        const int d = warp % SPLIT;  // a component a warp
        if (mine && ok && d < 3) {
          const Sums<R>* ps = part_s + (size_t)(warp - d) * 32 + lane;
          q = ps[0];
#pragma unroll
          for (int k = 1; k < kParts; ++k) add_sums(q, ps[k * 32]);
          a.dedr[slot * 3 + d] = pair_dedr<R>(gm, q, d);
        }
        __syncthreads();
      }
    }
    if (!QUEUE) break;
    __syncthreads();  // the item's shared memory is reused by the next item
  }
}

// Launch plan: atoms per CTA (A), warps (nw) and whether kParts warps share a
// batch.  A batch of 32 pairs costs a warp the same whether its lanes are full
// or not, so A minimises the batches that the busiest SM takes,
//   ceil(CTAs / SMs) ceil(A maxcnt / 32),
// plus a tenth of a batch a CTA for its staging (2000 atoms: 143 CTAs of 14
// atoms, 12 batches, one CTA an SM).  The batch is shared when an SM would hold
// fewer than col_warps batch-warps (the tunable; default 4, one a scheduler; FP32
// above 2J = 9 twice as many: its chains are long, and two warps a scheduler hide
// each other's latency): each FP64 unit and scheduler serves its own warps, so a
// lone batch-warp would leave three quarters of the SM idle, but sharing costs
// a barrier a round and empty parts at small orders.  1024 atoms (6 batches an
// SM), shared / not: FP64 2J1 18 / 12 us, 2J4 31 / 25, 2J8 88 / 76; FP32 2J2 10 / 8, 2J8
// 13.5 / 12.3, 2J11 15.6 / 17.2.
// force_A > 0 (SNAP_KNOB_DE_ATOMS): that A, if its shared memory fits.
struct DePlan {
  int nw, A, split;
  size_t smem;
};

template <typename R, int J2>
inline DePlan de_plan(int n, int maxcnt, int nsm, int col_warps, int force_A) {
  constexpr int NS = steps_total(J2);
  DePlan best{0, 0, 1, 0};
  double best_cost = 1e300;
  for (int A = force_A > 0 ? force_A : 1; A <= (force_A > 0 ? force_A : 32); ++A) {
    const int batches = std::max(1, (A * maxcnt + 31) / 32);
    const long ctas = (n + A - 1) / A, per_sm = (ctas + nsm - 1) / nsm;
    DePlan p;
    p.A = A;
    p.split = per_sm * batches < (sizeof(R) == 4 && J2 > 9 ? 2 : 1) * col_warps ? kParts : 1;
    p.nw = std::min(batches * p.split, de_max_warps<R>());
    p.smem = sizeof(y4<R>) * (size_t)A * NS + sizeof(rec_ab<R>) * NS +
             (p.split > 1 ? sizeof(Sums<R>) * (size_t)p.nw * 32 : 0) + sizeof(int) * (A + 1);
    if (p.smem > (size_t)224 * 1024) break;
    const double cost = (double)per_sm * (batches + 0.1);
    if (cost < best_cost - 1e-9) {
      best_cost = cost;
      best = p;
    }
  }
  return best;
}

template <typename R, int J2, int SPLIT>
cudaError_t launch_de_split(const WorkArgs& a, const DePlan& p, cudaStream_t s) {
  const long nitems = (a.n + p.A - 1) / p.A;
  if (a.persist & 2) {
    // persistent: as many CTAs as stay resident, items from the queue
    auto kq = de_pair_kernel<R, J2, SPLIT, true>;
    cudaError_t e = allow_smem(kq, p.smem);
    if (e != cudaSuccess) return e;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kq, p.nw * 32, p.smem);
    if (e != cudaSuccess) return e;
    const long grid = std::min<long>(nitems, (long)std::max(1, a.nsm) * std::max(1, occ));
    return launch_k(kq, dim3((unsigned)grid), dim3(p.nw * 32), p.smem, s, a, p.A);
  }
  auto kn = de_pair_kernel<R, J2, SPLIT, false>;
  cudaError_t e = allow_smem(kn, p.smem);
  if (e != cudaSuccess) return e;
  return launch_k(kn, dim3((unsigned)nitems), dim3(p.nw * 32), p.smem, s, a, p.A);
}

template <typename R, int J2>
cudaError_t launch_de_t(const WorkArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  if (a.H != half_size(J2)) return cudaErrorInvalidValue;
  const int maxcnt = std::max(1, a.de_maxcnt), nsm = std::max(1, a.nsm);
  DePlan p = de_plan<R, J2>(a.n, maxcnt, nsm, a.col_warps, a.de_atoms);
  if (p.A == 0) p = de_plan<R, J2>(a.n, maxcnt, nsm, a.col_warps, 0);  // a forced A that does not fit
  return p.split > 1 ? launch_de_split<R, J2, kParts>(a, p, s) : launch_de_split<R, J2, 1>(a, p, s);
}

// The pairs' sums on the host, in the kernel's arithmetic: ab [npairs][4] the
// Cayley-Klein parameters, y [H][2], out [npairs][6] the Sums.
template <typename R, int J2>
void pair_host_t(const std::vector<unsigned>& idx, const std::vector<double>& scale, const std::vector<double>& ab,
                 const std::vector<double>& fix, const std::vector<int>& cls, int npairs, const double* par,
                 const double* y, double* out) {
  constexpr int NS = steps_total(J2);
  std::vector<y4<R>> Y(NS);
  std::vector<rec_ab<R>> t(NS);
  constexpr int W = sizeof(rec_ab<R>) / sizeof(R), V = sizeof(step_scale<R>) / sizeof(R);
  for (int st = 0; st < NS; ++st) {
    step_scale<R> sc;
    for (int k = 0; k < V; ++k) (&sc.x)[k] = (R)scale[V * st + k];
    Y[st] = weighted_y<R>(idx[st], sc, [&](unsigned e) { return r2<R>{(R)y[2 * e], (R)y[2 * e + 1]}; });
    for (int k = 0; k < W; ++k) (&t[st].x)[k] = (R)ab[W * st + k];
  }
  if constexpr (sizeof(R) == 8)
    for (int c : cls)
      for (int k = 0; k < 4; ++k) fix_class(&Y[c & 0xFFFF].pr + k, &fix[(c & 0xFFFF) * kPairFix], c >> 16);
  for (int n = 0; n < npairs; ++n) {
    const double* g = par + 4 * n;
    Sums<R> q{R(0), R(0), R(0), R(0), R(0), R(0)};
    for (int part = 0; part < kParts; ++part)
      add_sums(q, pair_sums<R, J2>(Y.data(), t.data(), r2<R>{(R)g[0], (R)g[1]}, r2<R>{(R)g[2], (R)g[3]}, part));
    for (int k = 0; k < 6; ++k) out[6 * n + k] = (double)(&q.s)[k];
  }
}

}  // namespace pr
}  // namespace snap
