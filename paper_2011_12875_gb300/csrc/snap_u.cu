// snap_u.cu -- the neighbour build with the pairs' geometry, and compute_U.
//
// compute_U in closed form, lanes = the 32 atoms of a block.  With the classes
// (p, q) of snap_pairs.cuh, t = p + q + 2k, the elements of a pair are
//   u_t[k][k+q] = n s_k conj(a)^p b^q P_k(x),
//   u_t[k+q][k] = n s_k conj(a)^p (-conj(b))^q P_k(x),
// so Ulisttot (Eq. u) is, per class, sums over the atom's pairs of the real
// P_k(x) times two complex monomials, M+ = f_c conj(a)^p b^q and M- = f_c
// conj(a)^p conj(b)^q (its sign (-1)^q and n s_k are applied to the sums).
// A warp has a few classes of one length (a unit, HostTables::u_units), whose
// sums it keeps in registers over all pair slots of its 32 atoms: no exchange
// between lanes, no partial sums, and U is written once, coalesced.  The powers
// f_c conj(a)^p and b^q and x of a few slots at a time are tabulated in shared
// memory by the CTA's warps, one chain of powers a warp, while the slots before
// are summed (two buffers).
//
// A step (two elements) takes 2 multiply-adds for P_k and 4 for the sums, a
// class 8 for its monomials, up to 8 J for the powers: about 840 a pair at 2J8,
// 2,700 at 2J14, where the layer recursion (the form before) took 1,550 and 6,500,
// with a lane a column (31% of the lanes idle).  FP64 is bound by the FP64 pipe
// (a warp's multiply-add takes 15 cycles of an SM) and by SMs that hold one CTA
// more than others; FP32 by latency and instruction fetch, which is why the CTAs'
// warps run the same code.  A block's slots follow one another, so a launch
// takes 30 us and more in FP64 however few the atoms: FP64 takes this form above
// 2J = 5 and FP32 above 2J = 9 (u_by_layers).  Neighbour build and compute_U
// together, before -> now, 2000 atoms: FP64 2J6 153 -> 116 us, 2J8 278 -> 165, 2J11 692
// -> 278, 2J14 1146 -> 397; FP32 2J11 57 -> 53, 2J14 84 -> 61, 16000 atoms 561 -> 365;
// 128 atoms FP64 2J8 59 -> 48.
#include <algorithm>

#include "snap_geom.cuh"
#include "snap_internal.h"
#include "snap_neigh.cuh"
#include "snap_closed.cuh"

namespace snap {
namespace {

constexpr unsigned kFull = 0xffffffffu;

using pr::cmul;
using pr::fm;
using pr::r2;
using pr::rec_ab;
using pr::rec_t;
using pr::scaled;
using pr::step_scale;

constexpr int kUMaxWarps = 18;  // 112 registers: the longest unit's sums in FP64
// pair slots of a chunk, by the size of R: two buffers of 2J14 take 61 KB
__host__ __device__ constexpr int u_slots(int rsize) { return rsize == 4 ? 4 : 2; }
// values of R of one slot: x, J + 1 powers of a, J + 1 of b, for 32 atoms
__host__ __device__ constexpr int u_slot_len(int J) { return 32 * (1 + 4 * (J + 1)); }
// values of R of a unit's sums, at most eight steps
constexpr int kUSums = 8 * 4 * 32;

// One slot's tables: A[p] = f_c conj(a)^p, B[q] = b^q (complex, [.][32]), x.
template <typename R>
struct Slot {
  r2<R>*A, *B;
  R* x;
  __device__ __forceinline__ Slot(R* t, int J) {
    A = reinterpret_cast<r2<R>*>(t);
    B = A + (J + 1) * 32;
    x = t + 4 * (J + 1) * 32;
  }
};

// The chains of powers of a chunk's slots [s0, s0 + S) from the staged geometry
// ([slot][a, b, f_c][32]), up to the CTA's highest: warp w takes chains w, w +
// nw, ...
template <typename R>
__device__ __noinline__ void u_tables(const R* __restrict__ geo, R* t, int J, int pmax, int qmax, int s0, int nslots,
                                       int warp, int nw, int lane) {
  constexpr int S = u_slots(sizeof(R));
  for (int j = warp; j < 2 * S; j += nw) {
    const int s = s0 + (j >> 1);
    if (s >= nslots) continue;  // warp-uniform
    Slot<R> T(t + (size_t)(j >> 1) * u_slot_len(J), J);
    const R* g = geo + (size_t)s * 160 + lane;
    const r2<R> b = {g[64], g[96]};
    if ((j & 1) == 0) {
      const r2<R> ca = {g[0], -g[32]};
      // x: the smaller of |a|^2 and |b|^2 from 1 (both carry the rounding of a, b)
      const R na = fm(ca.x, ca.x, ca.y * ca.y), nb = fm(b.x, b.x, b.y * b.y);
      T.x[lane] = na < nb ? fm(R(2), na, R(-1)) : fm(R(-2), nb, R(1));
      r2<R> v = {g[128], R(0)};
      T.A[lane] = v;
      for (int p = 1; p <= pmax; ++p) {
        v = cmul(v, ca);
        T.A[p * 32 + lane] = v;
      }
    } else {
      r2<R> v = {R(1), R(0)};
      T.B[lane] = v;
      for (int q = 1; q <= qmax; ++q) {
        v = q == 1 ? b : cmul(v, b);
        T.B[q * 32 + lane] = v;
      }
    }
  }
}

struct UArgs {
  const int* un;  // the warp's unit
  int part, sums;  // half of the slots, place of the unit's sums in shared memory
  int warp, nw, lane, nslots;
  int pmax, qmax;  // highest powers of the CTA's classes
  long blk;
};

// A warp's half of a unit: M classes of K steps (M = 0: none, the warp only
// helps with the tables), the even or the odd slots; the two halves are added
// at the end, always in this way.  un: {K, M, (p, q, first step) x M}.
template <typename R, int K, int M>
__device__ __forceinline__ void u_unit(const WorkArgs& a, const UArgs& u, const R* __restrict__ geo, R* tab,
                                       const rec_ab<R>* __restrict__ ab) {
  constexpr int S = u_slots(sizeof(R)), MM = M > 0 ? M : 1;
  static_assert(K * M * 4 * 32 <= kUSums, "the unit's sums fit");
  const int J = a.twojmax, len = u_slot_len(J), lane = u.lane;
  int p[MM], q[MM], st[MM];
  r2<R> sp[MM][K], sm[MM][K];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int w = __ldg(u.un + 2 + m);
    p[m] = w & 15;
    q[m] = (w >> 4) & 15;
    st[m] = w >> 8;
#pragma unroll
    for (int k = 0; k < K; ++k) sp[m][k] = sm[m][k] = r2<R>{R(0), R(0)};
  }
  u_tables<R>(geo, tab, J, u.pmax, u.qmax, 0, u.nslots, u.warp, u.nw, lane);
  __syncthreads();
  for (int s0 = 0, buf = 0; s0 < u.nslots; s0 += S, buf ^= 1) {
    u_tables<R>(geo, tab + (size_t)(buf ^ 1) * S * len, J, u.pmax, u.qmax, s0 + S, u.nslots, u.warp, u.nw,
                lane);
    if (M > 0) {
#pragma unroll 1
      for (int j = u.part; j < S; j += 2) {
        if (s0 + j >= u.nslots) break;
        Slot<R> T(tab + ((size_t)buf * S + j) * len, J);
        const R x = T.x[lane];
#pragma unroll
        for (int m = 0; m < M; ++m) {
          const r2<R> A = T.A[p[m] * 32 + lane], B = T.B[q[m] * 32 + lane];
          const R rr = A.x * B.x, ri = A.x * B.y;
          const r2<R> mp = {fm(-A.y, B.y, rr), fm(A.y, B.x, ri)};
          const bool both = p[m] > 0 && q[m] > 0;  // warp-uniform
          R P[K];
          P[0] = R(1);
#pragma unroll
          for (int k = 1; k < K; ++k) {
            const R t = rec_t(ab[st[m] + k], x);
            P[k] = k == 1 ? t : fm(t, P[k - 1], k == 2 ? R(-1) : -P[k - 2]);
          }
          sp[m][0].x += mp.x;
          sp[m][0].y += mp.y;
#pragma unroll
          for (int k = 1; k < K; ++k) {
            sp[m][k].x = fm(P[k], mp.x, sp[m][k].x);
            sp[m][k].y = fm(P[k], mp.y, sp[m][k].y);
          }
          if (both) {
            const r2<R> mm = {fm(A.y, B.y, rr), fm(A.y, B.x, -ri)};
            sm[m][0].x += mm.x;
            sm[m][0].y += mm.y;
#pragma unroll
            for (int k = 1; k < K; ++k) {
              sm[m][k].x = fm(P[k], mm.x, sm[m][k].x);
              sm[m][k].y = fm(P[k], mm.y, sm[m][k].y);
            }
          }
        }
      }
    }
    __syncthreads();
  }
  // the odd half's sums, over the tables
  R* sums = tab + (size_t)u.sums * kUSums + lane;
  if (M > 0 && u.part == 1) {
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
      for (int k = 0; k < K; ++k) {
        R* d = sums + (m * K + k) * 128;
        d[0] = sp[m][k].x;
        d[32] = sp[m][k].y;
        d[64] = sm[m][k].x;
        d[96] = sm[m][k].y;
      }
  }
  __syncthreads();
  if (M == 0 || u.part == 1 || u.blk * 32 + lane >= a.n) return;
  r2<R>* U = reinterpret_cast<r2<R>*>(a.U) + u.blk * a.H * 32 + lane;
#pragma unroll
  for (int m = 0; m < M; ++m) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const R* d = sums + (m * K + k) * 128;
      sp[m][k].x += d[0];
      sp[m][k].y += d[32];
      sm[m][k].x += d[64];
      sm[m][k].y += d[96];
    }
    if constexpr (sizeof(R) == 8) {
      // P_k from the rounded recursion's PP_k (HostTables::pair_fix)
#pragma unroll
      for (int k = K - 1; k > 0; --k)
#pragma unroll
        for (int j = 0; j < k; ++j) {
          const double f = __ldg(a.pair_fix + (st[m] + j) * kPairFix + k - j);
          sp[m][k].x = fm(f, sp[m][j].x, sp[m][k].x);
          sp[m][k].y = fm(f, sp[m][j].y, sp[m][k].y);
          sm[m][k].x = fm(f, sm[m][j].x, sm[m][k].x);
          sm[m][k].y = fm(f, sm[m][j].y, sm[m][k].y);
        }
    }
  }
#pragma unroll
  for (int m = 0; m < M; ++m)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const unsigned w = __ldg(a.pair_idx + st[m] + k);
      const step_scale<R> n = reinterpret_cast<const step_scale<R>*>(a.pair_norm)[st[m] + k];
      const R odd = (q[m] & 1) ? R(-1) : R(1);
      // (k, k + q): stored, or its mirror (-1)^q conj is
      r2<R> v = {scaled(n, sp[m][k].x), scaled(n, sp[m][k].y)};
      if (q[m] == 0) v.x += (R)a.wself;
      const r2<R> mir = {odd * v.x, -odd * v.y};
      U[(w & 1023u) * 32] = ((w >> 10) & 1u) ? mir : v;
      if (p[m] > 0 && q[m] > 0) {
        U[((w >> 12) & 1023u) * 32] = r2<R>{odd * scaled(n, sm[m][k].x), odd * scaled(n, sm[m][k].y)};
        // on the middle column (2 (k + q) = t, p = q) the mirror is stored too
        if (p[m] == q[m]) {
          const int t = p[m] + q[m] + 2 * k, mb = k + q[m];
          U[(half_base(t) + mb * (t + 1) + t - k) * 32] = mir;
        }
      }
    }
}

// CTA = a block of 32 atoms x one of gridDim.y groups of the units u0 .. u0 +
// nu - 1: unit per blockIdx.y + w / 2 on warps w, w + 1 (w even; neighbouring
// units have the same K and M, so a CTA's warps run the same code).  A unit's
// sums do not depend on the groups.
template <typename R>
__global__ void __launch_bounds__(kUMaxWarps * 32, 1) u_kernel(WorkArgs a, int u0, int nu, int per) {
  extern __shared__ __align__(16) unsigned char smem[];
  UArgs u;
  u.warp = threadIdx.x >> 5;
  u.lane = threadIdx.x & 31;
  u.nw = blockDim.x >> 5;
  u.blk = blockIdx.x;
  rec_ab<R>* ab = reinterpret_cast<rec_ab<R>*>(smem);  // [steps]
  R* geo = reinterpret_cast<R*>(ab + a.npair_steps);
  R* tab = geo + (size_t)a.K * 160;
  for (int k = threadIdx.x; k < a.npair_steps; k += blockDim.x) ab[k] = reinterpret_cast<const rec_ab<R>*>(a.pair_ab)[k];
  {  // a lane a class of the CTA's units
    const int n = min(per, nu - per * (int)blockIdx.y) * (kUUnit - 2);
    int p = 0, q = 0;
    for (int k = u.lane; k < n; k += 32) {
      const int* un = a.u_units + (size_t)(u0 + per * (int)blockIdx.y + k / (kUUnit - 2)) * kUUnit;
      const int w = __ldg(un + 2 + k % (kUUnit - 2));  // 0 past the unit's classes
      p = max(p, w & 15);
      q = max(q, (w >> 4) & 15);
    }
    u.pmax = __reduce_max_sync(kFull, p);
    u.qmax = __reduce_max_sync(kFull, q);
  }
  const long i = u.blk * 32 + u.lane;
  const int cnt = i < a.n ? min(a.cnt[i], a.K) : 0;
  u.nslots = __reduce_max_sync(kFull, cnt);  // the same on every warp
  for (int s = u.warp; s < u.nslots; s += u.nw) {  // a lane without a pair there has f_c = 0
    r2<R> ga = {R(1), R(0)}, gb = {R(0), R(0)};
    R fc = R(0);
    if (s < cnt) {
      const R* g = reinterpret_cast<const R*>(a.geom) + (i * a.K + s) * kGeomStride;
      ga = *reinterpret_cast<const r2<R>*>(g);
      gb = *reinterpret_cast<const r2<R>*>(g + 2);
      fc = g[4];
    }
    R* d = geo + (size_t)s * 160 + u.lane;
    d[0] = ga.x;
    d[32] = ga.y;
    d[64] = gb.x;
    d[96] = gb.y;
    d[128] = fc;
  }
  __syncthreads();
  u.part = u.warp & 1;
  u.sums = u.warp >> 1;
  const int at = u.sums < per ? per * (int)blockIdx.y + u.sums : nu;
  u.un = a.u_units + (size_t)(u0 + min(at, nu - 1)) * kUUnit;
  const int K = at < nu ? __ldg(u.un) : 0, M = __ldg(u.un + 1);
  // every path has the same barriers
#define SNAP_U(KK, MM) \
  if (K == KK && M == MM) { \
    u_unit<R, KK, MM>(a, u, geo, tab, ab); \
    return; \
  }
  SNAP_U(8, 1) SNAP_U(7, 1) SNAP_U(6, 1) SNAP_U(5, 1) SNAP_U(4, 2) SNAP_U(3, 2) SNAP_U(2, 3) SNAP_U(1, 5)
  SNAP_U(4, 1) SNAP_U(3, 1) SNAP_U(2, 1) SNAP_U(1, 1)
#undef SNAP_U
  u_unit<R, 1, 0>(a, u, geo, tab, ab);
}

// ---------------------------------------- neighbour build with the geometry
// The neighbour build of snap_neigh.cuh (two atoms a CTA, SPLIT warps each: a
// batch scans every block of its configuration, one configuration skips far
// tiles): each stored pair's slot geometry is evaluated on the lane that accepts it,
// from the exact FP64 separation in its registers (dense lanes, no reload).
template <typename R, bool BATCH>
__global__ void __launch_bounds__(BATCH ? 256 : 128) neigh_geom_kernel(NeighArgs na, WorkArgs a) {
  constexpr int SPLIT = BATCH ? 4 : 2;
  static_assert(kNeighAtomsPerCta == 2, "batch CTA map and kernel disagree");
  nb::neigh_build_cta<BATCH, SPLIT, 2 * SPLIT>(na, [&](int, long, int, long q, double ex, double ey, double ez) {
    geo::pair_geom<R>(a, q, ex, ey, ez);
  });
}

}  // namespace

template <typename R>
cudaError_t launch_neigh_geom(const NeighArgs& na, const WorkArgs& a, int ncta, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  if (ncta > 0) return launch_k(neigh_geom_kernel<R, true>, dim3((unsigned)ncta), dim3(256), 0, s, na, a);
  return launch_k(neigh_geom_kernel<R, false>, dim3((unsigned)((a.n + 1) / 2)), dim3(128), 0, s, na, a);
}

// The units (several classes each, or one: HostTables::u_units) and the
// groups.  The CTAs an SM holds share its pipes, a quarter of them each warp:
// in multiply-adds a slot a launch lasts about
//   max(ceil(blocks G / SMs) (cost / G + 4 J) / 4, floor),
// cost = a block's units, 4 J = about the powers that each CTA tabulates; at most
// kUMaxWarps / 2 units a CTA.  Fewer than four warps would build the tables one
// chain after the other.  The floor is the longest unit's warp, which has every
// other slot: about half of the 6 + 6 K of a class of its own (K = J / 2 + 1
// steps; FP64 runs best with 3 K); units of several classes, 40, by their five
// classes of one step, whose monomials count for more than their multiply-adds.
// With the floors of 2J14 for every order, 27 and 30, small FP64 systems waited
// for CTAs of nine units.  All splits of 143 shapes (FP64 2J4 to 2J14, FP32 2J10 to
// 2J14, 16 to 16000 atoms): that choice lies 9.2% (FP64) and 4.9% over the best,
// this one 2.7% and 4.3% (neighbour build and compute_U, 128 atoms: 2J6 55 -> 45 us,
// 2J8 53 -> 49).
template <typename R>
cudaError_t launch_u(const WorkArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  const long nblk = (a.n + 31) / 32, nsm = std::max(1, a.nsm);
  int G = 1, fine = 0;
  double best = 1e300;
  for (int f = 0; f < 2; ++f) {
    const int nu = f ? a.u_nfine : a.u_nunits;
    for (int g = (nu + kUMaxWarps / 2 - 1) / (kUMaxWarps / 2); g <= nu; ++g) {
      const double t = std::max((double)((nblk * g + nsm - 1) / nsm) * ((double)a.u_cost / g + 4.0 * a.twojmax) / 4.0,
                                f ? (sizeof(R) == 8 ? 0.0 : 3.0) + 3.0 * (a.twojmax / 2 + 1) : 40.0);
      if (t < best - 1e-9) {
        best = t;
        G = g;
        fine = f;
      }
    }
  }
  const int nu = fine ? a.u_nfine : a.u_nunits, per = (nu + G - 1) / G, nw = std::max(4, 2 * per);
  G = (nu + per - 1) / per;  // no group without a unit
  const size_t tables = std::max((size_t)2 * u_slots(sizeof(R)) * u_slot_len(a.twojmax), (size_t)per * kUSums);
  const size_t smem = sizeof(rec_ab<R>) * (size_t)a.npair_steps + sizeof(R) * ((size_t)a.K * 160 + tables);
  cudaError_t e = allow_smem(u_kernel<R>, smem);
  if (e != cudaSuccess) return e;
  return launch_k(u_kernel<R>, dim3((unsigned)nblk, (unsigned)G), dim3(nw * 32), smem, s, a, fine ? a.u_nunits : 0, nu,
                  per);
}

template cudaError_t launch_neigh_geom<float>(const NeighArgs&, const WorkArgs&, int, cudaStream_t);
template cudaError_t launch_neigh_geom<double>(const NeighArgs&, const WorkArgs&, int, cudaStream_t);
template cudaError_t launch_u<float>(const WorkArgs&, cudaStream_t);
template cudaError_t launch_u<double>(const WorkArgs&, cudaStream_t);

}  // namespace snap
