// snap_tables.cpp -- host-side index and coefficient tables of the library.
//
//  * bispectrum enumeration 0 <= 2j2 <= 2j1 <= 2j <= 2J (arXiv:2011.12875,
//    Sec. II-A) in canonical order, and the (t1 >= t2, t) triples of the
//    adjoint Y (Sec. III, Eq. y);
//  * Clebsch-Gordan coefficients, obtained here from Wigner 3j symbols
//    (Racah's sum for the 3j symbol, long double);
//  * the weighted beta of every Y triple, and the Y work list sorted by
//    output element with its balanced split into warp slices.
#include "snap_tables.h"

#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <map>
#include <unordered_map>

namespace snap {

namespace {

long double lfact(int n) {
  long double f = 1.0L;
  for (int k = 2; k <= n; ++k) f *= (long double)k;
  return f;
}

// Wigner 3j symbol (j1 j2 j3; m1 m2 m3) with doubled arguments.
long double wigner3j(int tj1, int tj2, int tj3, int tm1, int tm2, int tm3) {
  if (tm1 + tm2 + tm3 != 0) return 0.0L;
  if (tj3 < std::abs(tj1 - tj2) || tj3 > tj1 + tj2 || ((tj1 + tj2 + tj3) & 1)) return 0.0L;
  if (std::abs(tm1) > tj1 || std::abs(tm2) > tj2 || std::abs(tm3) > tj3) return 0.0L;
  // integer combinations
  const int j1pj2mj3 = (tj1 + tj2 - tj3) / 2;
  const int j1mj2pj3 = (tj1 - tj2 + tj3) / 2;
  const int mj1pj2pj3 = (-tj1 + tj2 + tj3) / 2;
  const int jsum1 = (tj1 + tj2 + tj3) / 2 + 1;
  const long double tri = lfact(j1pj2mj3) * lfact(j1mj2pj3) * lfact(mj1pj2pj3) / lfact(jsum1);
  const long double mf = lfact((tj1 + tm1) / 2) * lfact((tj1 - tm1) / 2) * lfact((tj2 + tm2) / 2) *
                         lfact((tj2 - tm2) / 2) * lfact((tj3 + tm3) / 2) * lfact((tj3 - tm3) / 2);
  // k runs where all of these are >= 0
  const int x1 = (tj3 - tj2 + tm1) / 2;  // j3 - j2 + m1 + k
  const int x2 = (tj3 - tj1 - tm2) / 2;  // j3 - j1 - m2 + k
  const int y1 = j1pj2mj3;               // j1 + j2 - j3 - k
  const int y2 = (tj1 - tm1) / 2;        // j1 - m1 - k
  const int y3 = (tj2 + tm2) / 2;        // j2 + m2 - k
  const int kmin = std::max(0, std::max(-x1, -x2));
  const int kmax = std::min(y1, std::min(y2, y3));
  long double sum = 0.0L;
  for (int k = kmin; k <= kmax; ++k) {
    const long double den =
        lfact(k) * lfact(x1 + k) * lfact(x2 + k) * lfact(y1 - k) * lfact(y2 - k) * lfact(y3 - k);
    sum += ((k & 1) ? -1.0L : 1.0L) / den;
  }
  // overall phase (-1)^(j1 - j2 - m3)
  const int ph = (tj1 - tj2 - tm3) / 2;
  const long double sign = (ph & 1) ? -1.0L : 1.0L;
  return sign * std::sqrt(tri) * std::sqrt(mf) * sum;
}

}  // namespace

// <j1 m1 j2 m2 | j m> = (-1)^(j1 - j2 + m) sqrt(2j+1) (j1 j2 j; m1 m2 -m)
double clebsch_gordan(int tj1, int tm1, int tj2, int tm2, int tj, int tm) {
  if (tm1 + tm2 != tm) return 0.0;
  const long double w = wigner3j(tj1, tj2, tj, tm1, tm2, -tm);
  const int ph = (tj1 - tj2 + tm) / 2;
  const long double s = (ph & 1) ? -1.0L : 1.0L;
  return (double)(s * std::sqrt((long double)(tj + 1)) * w);
}

int count_coeff(int twojmax) {
  if (twojmax < 0 || twojmax > kMaxTwoJ) return -1;
  int n = 0;
  for (int t1 = 0; t1 <= twojmax; ++t1)
    for (int t2 = 0; t2 <= t1; ++t2)
      for (int t = t1 - t2; t <= std::min(twojmax, t1 + t2); t += 2)
        if (t >= t1) ++n;
  return n;
}

namespace {

// Factor order of the terms [first, end) of one output.  A term's product is
// symmetric in its two factors, and compute_Y groups the terms of an output
// by their first factor (Y += U[e1] * sum_k c_k U[e2,k]), so fewer distinct
// first factors mean fewer groups.  Choosing them is a vertex cover of the
// graph whose vertices are the stored elements (index, conjugation) and
// whose edges are the terms; the greedy cover takes, again and again, the
// element with the most terms not yet covered (ties: the larger element) and
// makes it the first factor of those terms.
void orient_by_cover(std::vector<unsigned>& terms, size_t first) {
  const size_t n = terms.size() - first;
  if (n < 2) return;
  auto e1 = [](unsigned w) { return (w & 1023u) << 1 | ((w >> 20) & 1u); };
  auto e2 = [](unsigned w) { return ((w >> 10) & 1023u) << 1 | ((w >> 21) & 1u); };
  std::unordered_map<unsigned, std::vector<size_t>> inc;  // element -> its terms
  for (size_t k = first; k < terms.size(); ++k) {
    const unsigned a = e1(terms[k]), b = e2(terms[k]);
    inc[a].push_back(k);
    if (b != a) inc[b].push_back(k);
  }
  std::unordered_map<unsigned, int> deg;
  std::vector<std::pair<int, unsigned>> heap;  // (uncovered terms, element)
  for (const auto& kv : inc) {
    deg[kv.first] = (int)kv.second.size();
    heap.push_back({(int)kv.second.size(), kv.first});
  }
  std::make_heap(heap.begin(), heap.end());
  std::vector<char> covered(n, 0);
  while (!heap.empty()) {
    std::pop_heap(heap.begin(), heap.end());
    const auto top = heap.back();
    heap.pop_back();
    const unsigned v = top.second;
    if (top.first != deg[v]) {  // stale entry: push the current count back
      if (deg[v] > 0) {
        heap.push_back({deg[v], v});
        std::push_heap(heap.begin(), heap.end());
      }
      continue;
    }
    if (top.first == 0) break;
    for (size_t k : inc[v]) {
      if (covered[k - first]) continue;
      covered[k - first] = 1;
      unsigned& w = terms[k];
      const unsigned a = e1(w), b = e2(w);
      if (a != v) {  // v is the second factor: swap the two factors
        w = ((w >> 10) & 1023u) | ((w & 1023u) << 10) | (((w >> 21) & 1u) << 20) |
            (((w >> 20) & 1u) << 21) | (w & ~((1u << 22) - 1));
      }
      const unsigned o = (a == v) ? b : a;
      if (o != v) --deg[o];
    }
    deg[v] = 0;
  }
}

// Half-layout place of element (xa, xb) of layer tt: past the stored columns its
// mirror, conjugated, with the sign.
void half_elem(int tt, int xa, int xb, int& idx, int& conj, double& sgn) {
  if (2 * xb <= tt) {
    idx = half_base(tt) + xb * (tt + 1) + xa;
    conj = 0;
    sgn = 1.0;
  } else {
    idx = half_base(tt) + (tt - xb) * (tt + 1) + (tt - xa);
    conj = 1;
    sgn = ((xa + xb) & 1) ? -1.0 : 1.0;
  }
}

}  // namespace

void HostTables::build(int J2) {
  twojmax = J2;
  H = half_size(J2);
  half_tmm.clear();
  for (int t = 0; t <= J2; ++t)
    for (int mb = 0; 2 * mb <= t; ++mb)
      for (int ma = 0; ma <= t; ++ma) half_tmm.push_back(pack_tmm(t, ma, mb));

  // canonical bispectrum index
  std::map<long, int> bidx;
  ncoeff = 0;
  for (int t1 = 0; t1 <= J2; ++t1)
    for (int t2 = 0; t2 <= t1; ++t2)
      for (int t = t1 - t2; t <= std::min(J2, t1 + t2); t += 2)
        if (t >= t1) bidx[(long)t1 * 10000 + t2 * 100 + t] = ncoeff++;
  auto idx_of = [&](int a, int b, int c) { return bidx.at((long)a * 10000 + b * 100 + c); };

  // Y triples (t1 >= t2, any t) with their CG blocks and beta weights.
  ztrip.clear();
  cg.clear();
  for (int t1 = 0; t1 <= J2; ++t1)
    for (int t2 = 0; t2 <= t1; ++t2)
      for (int t = t1 - t2; t <= std::min(J2, t1 + t2); t += 2) {
        ZTrip z;
        z.t1 = t1;
        z.t2 = t2;
        z.t = t;
        z.cg_off = (int)cg.size();
        for (int x1 = 0; x1 <= t1; ++x1)
          for (int x2 = 0; x2 <= t2; ++x2) {
            const int m1 = 2 * x1 - t1, m2 = 2 * x2 - t2;
            cg.push_back(std::abs(m1 + m2) <= t ? clebsch_gordan(t1, m1, t2, m2, t, m1 + m2) : 0.0);
          }
        // The derivative of E_i = sum_l beta_l B_l with respect to U_t collects,
        // for every component l whose sorted triple contains t, the Z matrix
        // built from the other two U's.  Moving the conjugate of a triple
        // product from U_t to a U of larger rank scales it by
        // (t_big + 1)/(t + 1); coinciding ranks count once per occurrence.
        if (t >= t1) {  // t is the largest rank: component (t1, t2, t)
          z.bidx = idx_of(t1, t2, t);
          z.fac = (t1 == t) ? ((t2 == t) ? 3.0 : 2.0) : 1.0;
        } else if (t >= t2) {  // t1 > t >= t2: component (t, t2, t1)
          z.bidx = idx_of(t, t2, t1);
          z.fac = ((t2 == t) ? 2.0 : 1.0) * (double)(t1 + 1) / (double)(t + 1);
        } else {  // t < t2 <= t1: component (t2, t, t1)
          z.bidx = idx_of(t2, t, t1);
          z.fac = (double)(t1 + 1) / (double)(t + 1);
        }
        ztrip.push_back(z);
      }

  // Bispectrum term list (descriptor output, Eq. z): for every canonical
  // component l = (t1 >= t2, t >= t1), for every half-layout element (t, ma,
  // mb) with a nonzero half weight w,
  //   B_l += Re( conj(U_t[ma][mb]) * w * sum C(ma1,ma2) C(mb1,mb2) U_t1 U_t2 ),
  // so B_l = Re Z^t_{t1t2} : conj(U_t) over the full matrix.  The records
  // use the compute_Y format with w folded into the coefficient; bit 22 ends
  // an output element, bit 23 ends a component; bout holds the U_t element
  // index of every output group in order.
  bterms.clear();
  bterm_coef.clear();
  bout.clear();
  bcomp_first.clear();
  bgroup_first.clear();
  for (int q = 0; q < (int)ztrip.size(); ++q) {
    const ZTrip& z = ztrip[q];
    if (z.t < z.t1) continue;  // canonical components only
    bcomp_first.push_back((int)bterms.size());
    bgroup_first.push_back((int)bout.size());
    const int t = z.t, dl = (z.t1 + z.t2 - t) / 2;
    for (int mb = 0; 2 * mb <= t; ++mb)
      for (int ma = 0; ma <= t; ++ma) {
        const int wgt = (2 * mb < t) ? 2 : (ma < mb ? 2 : (ma == mb ? 1 : 0));
        if (wgt == 0) continue;
        const size_t first = bterms.size();
        for (int mb1 = std::max(0, mb + dl - z.t2); mb1 <= std::min(z.t1, mb + dl); ++mb1) {
          const int mb2 = mb + dl - mb1;
          const double cb = cg[z.cg_off + mb1 * (z.t2 + 1) + mb2];
          if (cb == 0.0) continue;
          for (int ma1 = std::max(0, ma + dl - z.t2); ma1 <= std::min(z.t1, ma + dl); ++ma1) {
            const int ma2 = ma + dl - ma1;
            const double ca = cg[z.cg_off + ma1 * (z.t2 + 1) + ma2];
            if (ca == 0.0) continue;
            int i1, c1, i2, c2;
            double s1, s2;
            half_elem(z.t1, ma1, mb1, i1, c1, s1);
            half_elem(z.t2, ma2, mb2, i2, c2, s2);
            bterms.push_back((unsigned)i1 | ((unsigned)i2 << 10) | ((unsigned)c1 << 20) |
                             ((unsigned)c2 << 21));
            bterm_coef.push_back(wgt * ca * cb * s1 * s2);
          }
        }
        if (bterms.size() > first) {
          bterms.back() |= (1u << 22);
          bout.push_back(half_base(t) + mb * (t + 1) + ma);
        }
      }
    bterms.back() |= (1u << 23);
  }
  bcomp_first.push_back((int)bterms.size());
  bgroup_first.push_back((int)bout.size());
  // chunks of whole groups, about kBChunk terms (more at large 2J, so that
  // there are at most about kBMaxChunks), within components
  const int chunk_len = std::max<int>(kBChunk, (int)((bterms.size() + kBMaxChunks - 1) / kBMaxChunks));
  bchunk_term.clear();
  bchunk_group.clear();
  bcomp_chunk.clear();
  for (int l = 0; l < ncoeff; ++l) {
    bcomp_chunk.push_back((int)bchunk_term.size());
    int q = bcomp_first[l], gq = bgroup_first[l];
    bchunk_term.push_back(q);
    bchunk_group.push_back(gq);
    int inchunk = 0;
    for (; q < bcomp_first[l + 1]; ++q) {
      ++inchunk;
      if (bterms[q] & (1u << 22)) {  // a group ends here
        ++gq;
        if (inchunk >= chunk_len && q + 1 < bcomp_first[l + 1]) {
          bchunk_term.push_back(q + 1);
          bchunk_group.push_back(gq);
          inchunk = 0;
        }
      }
    }
  }
  bcomp_chunk.push_back((int)bchunk_term.size());
  bchunk_term.push_back((int)bterms.size());
  bchunk_group.push_back((int)bout.size());
  // device order: every chunk's groups cut into pieces of at most kBGroupMax
  // terms (a group of n terms into ceil(n / kBGroupMax) pieces whose lengths
  // differ by at most one), pieces ordered by length, stably
  const int nchunks = (int)bchunk_term.size() - 1;
  bdev.assign(bterms.size(), 0u);
  bdev_coef.assign(bterms.size(), 0.0);
  bdev_o.assign(bterms.size(), -1);
  bchunk_runs.assign((size_t)nchunks * kBGroupMax, 0);
  struct Piece {
    int first, len, o;
  };
  std::vector<Piece> pieces;
  for (int ch = 0; ch < nchunks; ++ch) {
    pieces.clear();
    int g = bchunk_group[ch], gfirst = bchunk_term[ch];
    for (int q = bchunk_term[ch]; q < bchunk_term[ch + 1]; ++q) {
      if (!(bterms[q] & (1u << 22))) continue;
      const int n = q + 1 - gfirst, np = (n + kBGroupMax - 1) / kBGroupMax;
      for (int k = 0, at = gfirst; k < np; ++k) {
        const int len = n / np + (k < n % np ? 1 : 0);
        pieces.push_back({at, len, bout[g]});
        at += len;
      }
      gfirst = q + 1;
      ++g;
    }
    std::stable_sort(pieces.begin(), pieces.end(), [](const Piece& x, const Piece& y) { return x.len < y.len; });
    int at = bchunk_term[ch];
    for (const Piece& pc : pieces) {
      bchunk_runs[(size_t)ch * kBGroupMax + pc.len - 1] += 1;
      for (int k = 0; k < pc.len; ++k, ++at) {
        bdev[at] = bterms[pc.first + k] & 0x3FFFFFu;
        bdev_coef[at] = bterm_coef[pc.first + k];
        bdev_o[at] = k == 0 ? pc.o : -1;
      }
    }
  }

  half_scale.assign(H, 0.0);
  for (int e = 0; e < H; ++e) {
    const int t = tmm_t(half_tmm[e]), ma = tmm_ma(half_tmm[e]), mb = tmm_mb(half_tmm[e]);
    long double f = 1.0L;
    for (int k = 2; k <= t - ma; ++k) f *= k;
    for (int k = 2; k <= ma; ++k) f *= k;
    for (int k = 2; k <= t - mb; ++k) f /= k;
    half_scale[e] = (double)std::sqrt(f);
  }
  // closed form of u: see snap_pairs.cuh.  P_k^(q,p) monic has the recursion
  // pi_{k+1} = (x - b_k) pi_k - g_k pi_{k-1} (Jacobi polynomials, alpha = q,
  // beta = p); with pi_k = s_k P_k, s_{k+1} = g_k s_{k-1}, the last factor is 1.
  // The kernels hold alpha and beta rounded to FP32, so their polynomials are
  // others, PP_k, of the same degrees: P_k = PP_k + sum_{j <= k} d_kj PP_j.  From
  // the two recursions, with x PP_j = (PP_{j+1} + PP_{j-1} - bb_j PP_j) / aa_j,
  //   d_{k+1,j} = al_k (d_{k,j-1} / aa_{j-1} + d_{k,j+1} / aa_{j+1} - d_kj bb_j / aa_j) + be_k d_kj - d_{k-1,j}
  // and, for the PP_k in P_k itself, (al_k - aa_k) / aa_k at j = k + 1 and k - 1
  // and be_k - al_k bb_k / aa_k at j = k.  1 + d_kk goes into the norm.
  pair_idx.clear();
  pair_norm.clear();
  pair_norm_fix.clear();
  pair_weight.clear();
  pair_ab.clear();
  pair_fix.clear();
  std::array<long double, kMaxTwoJ + 2> fact;
  for (int k = 0; k < (int)fact.size(); ++k) fact[k] = lfact(k);
  for (int p = 0; p <= J2; ++p)
    for (int q = J2 - p; q >= 0; --q) {
      long double s0 = 1.0L, s1 = 1.0L, al = 0.0L, be = 0.0L;  // s_{k-1}, s_k and the coefficients to P_k
      long double aa[kPairFix] = {}, bb[kPairFix] = {}, d[kPairFix][kPairFix] = {};
      const size_t first = pair_idx.size();
      pair_fix.resize((first + (J2 - p - q) / 2 + 1) * kPairFix, 0.0);
      for (int k = 0; p + q + 2 * k <= J2; ++k) {
        const int t = p + q + 2 * k, c = 2 * k + p + q;
        if (k > 0) {  // s0 = s_{k-1}, s1 = s_k
          const long double b = k == 1 ? (long double)(p - q) / (p + q + 2)
                                       : (long double)(p * p - q * q) / ((long double)(c - 2) * c);
          al = s0 / s1;
          be = -al * b;
          const int m = k - 1;
          aa[m] = (float)al;
          bb[m] = (float)be;
          for (int j = 0; j <= k; ++j) {
            long double v = j > 0 ? al * d[m][j - 1] / aa[j - 1] : 0.0L;
            if (j <= m) v += (be - al * bb[j] / aa[j]) * d[m][j];
            if (j < m) v += al * d[m][j + 1] / aa[j + 1] - d[m - 1][j];
            if (j == k || j == m - 1) v += (al - aa[m]) / aa[m];
            if (j == m) v += be - al * bb[m] / aa[m];
            d[k][j] = v;
          }
          for (int j = 0; j < k; ++j)
            pair_fix[(first + j) * kPairFix + k - j] = (double)(d[k][j] / (1.0L + d[k][k]));
        }
        unsigned w;
        if (2 * (k + q) <= t) w = (unsigned)(half_base(t) + (k + q) * (t + 1) + k);
        else w = (unsigned)(half_base(t) + (t - k - q) * (t + 1) + (t - k)) | (1u << 10) | ((unsigned)(q & 1) << 11);
        if (p > 0 && q > 0) w |= ((unsigned)(half_base(t) + k * (t + 1) + k + q) << 12) | (1u << 22);
        pair_idx.push_back(w);
        const long double n = fact[t] / std::pow(2.0L, k) /
                              std::sqrt(fact[t - k] * fact[k] * fact[t - k - q] * fact[k + q]) * s1;
        pair_norm.push_back((double)n);
        pair_norm_fix.push_back((double)(n + n * d[k][k]));
        pair_weight.push_back(p == 0 && q == 0 ? 1.0 : 2.0);
        pair_ab.push_back((double)al);
        pair_ab.push_back((double)be);
        // s_{k+1}: s_1 = sqrt(g_1), s_{k+1} = g_k s_{k-1}
        const auto g = [&](int m) -> long double {
          const long double d = 2.0L * m + p + q;
          if (m == 1) return 4.0L * (1 + p) * (1 + q) / (d * d * (d + 1));
          return 4.0L * m * (m + p) * (m + q) * (m + p + q) / (d * d * (d + 1) * (d - 1));
        };
        const long double s2 = k == 0 ? std::sqrt(g(1)) : g(k) * s0;
        s0 = s1;
        s1 = s2;
      }
    }

  // classes of one length in units of about 50 multiply-adds a pair (the last
  // unit of a length repeats its last class), then the same classes one a unit
  u_units.clear();
  u_nunits = u_cost = 0;
  for (int fine = 0; fine < 2; ++fine) {
    if (fine) u_nunits = (int)u_units.size() / kUUnit;
    for (int K = J2 / 2 + 1; K >= 1; --K) {
      const int most = fine || K >= 5 ? 1 : K >= 3 ? 2 : K == 2 ? 3 : 5;
      std::vector<int> cls;
      int at = 0;
      for (int p = 0; p <= J2; ++p)
        for (int q = J2 - p; q >= 0; --q) {
          const int steps = (J2 - p - q) / 2 + 1;
          if (steps == K) cls.push_back(p | q << 4 | at << 8);
          at += steps;
        }
      for (size_t c = 0; c < cls.size(); c += most) {
        std::vector<int> u(kUUnit, 0);
        u[0] = K;
        u[1] = most;
        for (int k = 0; k < most; ++k) u[2 + k] = cls[std::min(c + k, cls.size() - 1)];
        u_units.insert(u_units.end(), u.begin(), u.end());
        if (fine) u_cost += 6 + 6 * K;
      }
    }
  }
}

std::vector<double> HostTables::pair_scales(bool fp64, bool weighted) const {
  std::vector<double> w;
  for (size_t k = 0; k < pair_norm.size(); ++k) {
    const double n = (fp64 ? pair_norm_fix[k] : pair_norm[k]) * (weighted ? pair_weight[k] : 1.0);
    w.push_back(fp64 ? n : (float)n);
    if (!fp64) w.push_back(n - (float)n);
  }
  return w;
}

std::vector<double> HostTables::pair_recursion(bool fp64) const {
  std::vector<double> ab;
  for (size_t k = 0; k < pair_ab.size(); k += 2) {
    const double al = (float)pair_ab[k], be = (float)pair_ab[k + 1];
    ab.insert(ab.end(), {al, be});
    if (!fp64) ab.insert(ab.end(), {pair_ab[k] - al, pair_ab[k + 1] - be});
  }
  return ab;
}

std::vector<int> HostTables::pair_classes() const {
  std::vector<int> cls;
  int st = 0;
  for (int p = 0; p <= twojmax; ++p)
    for (int q = twojmax - p; q >= 0; --q) {
      const int steps = (twojmax - p - q) / 2 + 1;
      if (steps > 1) cls.push_back(st | steps << 16);
      st += steps;
    }
  // longest first, those of a length together: a warp takes several, its lanes then
  // run the same code (fused dE, 128 atoms 2J14: 57 us, in the classes' own order 59)
  std::stable_sort(cls.begin(), cls.end(), [](int x, int y) { return x >> 16 > y >> 16; });
  return cls;
}

void HostTables::build_terms() {
  // For every half-layout output element (t, ma, mb)
  // of Y, in output order, every nonzero term of every triple (t1 >= t2)
  // with output rank t:
  //   Y_t[ma][mb] += betaw * C(ma1, ma2) C(mb1, mb2) U_t1[ma1][mb1] U_t2[ma2][mb2],
  // ma2 = ma + d - ma1, mb2 = mb + d - mb1, d = (t1+t2-t)/2.  An element of U
  // past the stored half columns is (-1)^(ma+mb) conj of its mirror, so each
  // term stores the two half-layout indices, two conjugation flags, and a
  // coefficient with the signs, the CG product and betaw folded in.
  terms.clear();
  term_cg.clear();
  term_trip.clear();
  term_out_first.clear();
  // triples grouped by output rank
  std::vector<std::vector<int>> by_t(twojmax + 1);
  std::unordered_map<unsigned long long, size_t> same_layer;  // (triple, word) -> term
  for (int q = 0; q < (int)ztrip.size(); ++q) by_t[ztrip[q].t].push_back(q);
  for (int t = 0; t <= twojmax; ++t)
    for (int mb = 0; 2 * mb <= t; ++mb)
      for (int ma = 0; ma <= t; ++ma) {
        const size_t first = terms.size();
        same_layer.clear();
        // Below the centre of the middle column (2 mb = t, ma > mb) Y is the
        // mirror of the element above it, and the contractions that read Y
        // (energy, dE/dr) give it weight 0: one zero term there (Y = 0), and
        // the host export fills in the mirror.
        const bool mirrored = 2 * mb == t && ma > mb;
        for (int q : by_t[t]) {
          if (mirrored) break;
          const ZTrip& z = ztrip[q];
          const int dl = (z.t1 + z.t2 - t) / 2;
          for (int mb1 = std::max(0, mb + dl - z.t2); mb1 <= std::min(z.t1, mb + dl); ++mb1) {
            const int mb2 = mb + dl - mb1;
            const double cb = cg[z.cg_off + mb1 * (z.t2 + 1) + mb2];
            if (cb == 0.0) continue;
            for (int ma1 = std::max(0, ma + dl - z.t2); ma1 <= std::min(z.t1, ma + dl); ++ma1) {
              const int ma2 = ma + dl - ma1;
              const double ca = cg[z.cg_off + ma1 * (z.t2 + 1) + ma2];
              if (ca == 0.0) continue;
              int i1, c1, i2, c2;
              double s1, s2;
              half_elem(z.t1, ma1, mb1, i1, c1, s1);
              half_elem(z.t2, ma2, mb2, i2, c2, s2);
              // t1 == t2: the term with the factors swapped, (ma2, mb2) as
              // the first, has the same coefficient and the same product, so
              // the two are kept as one term, the stored element with the
              // lower (index, conjugation) first, with the summed coefficient
              if (z.t1 == z.t2 && (i2 < i1 || (i2 == i1 && c2 < c1))) {
                std::swap(i1, i2);
                std::swap(c1, c2);
              }
              const unsigned w = (unsigned)i1 | ((unsigned)i2 << 10) | ((unsigned)c1 << 20) |
                                 ((unsigned)c2 << 21);
              const double cgp = ca * cb * s1 * s2;
              if (z.t1 == z.t2) {
                const auto ins = same_layer.emplace(((unsigned long long)q << 32) | w, terms.size());
                if (!ins.second) {
                  term_cg[ins.first->second] += cgp;
                  continue;
                }
              }
              terms.push_back(w);
              term_cg.push_back(cgp);
              term_trip.push_back(q);
            }
          }
        }
        {  // drop merged terms whose coefficients cancelled exactly
          size_t o = first;
          for (size_t k = first; k < terms.size(); ++k)
            if (term_cg[k] != 0.0) {
              terms[o] = terms[k];
              term_cg[o] = term_cg[k];
              term_trip[o] = term_trip[k];
              ++o;
            }
          terms.resize(o);
          term_cg.resize(o);
          term_trip.resize(o);
        }
        if (mirrored) {
          terms.push_back(0u);
          term_cg.push_back(0.0);
          term_trip.push_back(by_t[t].front());
        }
        orient_by_cover(terms, first);
        // Group the output's terms by their first factor (index and
        // conjugation flag, stable): compute_Y then forms
        //   Y += U_t1[..] * sum_k coef_k U_t2,k[..]
        // once per group.  Bit 23 ends a group, bit 22 the output; every output has at
        // least one term: the term of the (t, 0, t) triple, whose
        // Clebsch-Gordan product is 1, or the zero term of a mirrored output.
        const size_t cnt = terms.size() - first;
        if (cnt > 0) {
          std::vector<size_t> ord(cnt);
          for (size_t k = 0; k < cnt; ++k) ord[k] = k;
          auto key = [&](size_t k) { return terms[first + k] & ((1023u) | (1u << 20)); };
          std::stable_sort(ord.begin(), ord.end(), [&](size_t x, size_t y) { return key(x) < key(y); });
          std::vector<unsigned> tw(cnt);
          std::vector<double> tc(cnt);
          std::vector<int> tq(cnt);
          for (size_t k = 0; k < cnt; ++k) {
            tw[k] = terms[first + ord[k]];
            tc[k] = term_cg[first + ord[k]];
            tq[k] = term_trip[first + ord[k]];
          }
          const unsigned kmask = 1023u | (1u << 20);
          for (size_t k = 0; k < cnt; ++k) {
            const bool end = k + 1 == cnt || (tw[k + 1] & kmask) != (tw[k] & kmask);
            terms[first + k] = tw[k] | (end ? (1u << 23) : 0u);
            term_cg[first + k] = tc[k];
            term_trip[first + k] = tq[k];
          }
          terms.back() |= (1u << 22);
        }
        term_out_first.push_back((int)first);
      }
  term_out_first.push_back((int)terms.size());
}

// a vector's byte offset and conjugation (bit 31) in 16 bits
static unsigned yc_pack(unsigned w) { return (w & 0x7FFFFFFFu) >> 8 | (w >> 31) << 15; }

void HostTables::build_classes(bool wide) {
  yc_wide = wide;
  const int J = twojmax, cw = wide ? 2 : 1;
  // Output pairs of a task.  FP32: 4 where a block has hundreds of tasks (2J14,
  // 2000 atoms: 387 us, with 2: 404), 2 where the largest would hold up the
  // rest (2J8, 2000 atoms: 37 us, with 4: 43).
  const int maxnp = wide ? 1 : J > 9 ? kYcOuts / 2 : 2;
  // first slot of the vector of each stored m
  std::vector<int> start((size_t)(2 * J + 1) * (J + 1), -1);
  auto at = [&](int ma, int mb) -> int& { return start[(size_t)(ma + J) * (J + 1) - mb]; };  // mb <= 0
  auto low = [](int ma, int mb) { return std::max(std::abs(ma), std::abs(mb)); };
  yc_slot.assign(H, 0);
  int n = 0;
  for (int mb = -J; mb <= 0; ++mb)
    for (int ma = -J; ma <= J; ++ma) {
      if ((ma - mb) & 1) continue;
      at(ma, mb) = n;
      for (int t = low(ma, mb); t <= J; t += 2) yc_slot[half_base(t) + (mb + t) / 2 * (t + 1) + (ma + t) / 2] = n++;
    }
  std::vector<int> trip((size_t)(J + 1) * (J + 1) * (J + 1), -1);
  for (int q = 0; q < (int)ztrip.size(); ++q)
    trip[((size_t)ztrip[q].t1 * (J + 1) + ztrip[q].t2) * (J + 1) + ztrip[q].t] = q;
  struct M {
    int a, b;
  };
  // coefficient (without beta) of u_t1[m1] u_t2[m2] in Y_t of m1 + m2, and its triple
  auto coef = [&](int t1, M m1, int t2, M m2, int t, int& q) {
    const bool same = m1.a == m2.a && m1.b == m2.b;
    q = -1;
    if (t < std::abs(t1 - t2) || t > t1 + t2) return 0.0;
    // a pair of equal m has each unordered (t1, t2) once; of different m, a
    // triple with t1 = t2 has its two terms, equal ones, in one
    if (same && t1 < t2) return 0.0;
    double w = !same && t1 == t2 ? 2.0 : 1.0;
    if (t1 < t2) {
      std::swap(t1, t2);
      std::swap(m1, m2);
    }
    q = trip[((size_t)t1 * (J + 1) + t2) * (J + 1) + t];
    const ZTrip& z = ztrip[q];
    auto c = [&](int x, int y) { return cg[z.cg_off + (x + t1) / 2 * (t2 + 1) + (y + t2) / 2]; };
    w *= c(m1.a, m2.a) * c(m1.b, m2.b);
    // mirrored vectors: (-1)^(ma + mb), ma + mb = (m_a + m_b) / 2 + t
    if (m1.b > 0 && (((m1.a + m1.b) / 2 + t1) & 1)) w = -w;
    if (m2.b > 0 && (((m2.a + m2.b) / 2 + t2) & 1)) w = -w;
    return w;
  };
  auto place = [&](M m) {  // byte offset of its vector's [32] complex float, bit 31: conjugate
    return m.b > 0 ? (unsigned)at(-m.a, -m.b) * 256u | 0x80000000u : (unsigned)at(m.a, m.b) * 256u;
  };
  yc_task.clear();
  yc_trip.clear();
  yc_head.clear();
  yc_cg.clear();
  yc_cost.clear();
  struct Item {
    M m1, m2;  // u[m2] the longer one
    int l1, l2;
  };
  std::vector<Item> items;
  for (int Mb = -J; Mb <= 0; ++Mb)
    for (int Ma = -J; Ma <= (Mb < 0 ? J : 0); ++Ma) {
      if ((Ma - Mb) & 1) continue;
      items.clear();
      for (int a1 = std::max(-J, Ma - J); a1 <= std::min(J, Ma + J); ++a1)
        for (int b1 = std::max(-J, Mb - J); b1 <= std::min(J, Mb + J); ++b1) {
          if ((a1 - b1) & 1) continue;
          const M m1{a1, b1}, m2{Ma - a1, Mb - b1};
          if (m2.a < m1.a || (m2.a == m1.a && m2.b < m1.b)) continue;
          const int l1 = (J - low(m1.a, m1.b)) / 2 + 1, l2 = (J - low(m2.a, m2.b)) / 2 + 1;
          items.push_back(l1 <= l2 ? Item{m1, m2, l1, l2} : Item{m2, m1, l2, l1});
        }
      std::stable_sort(items.begin(), items.end(), [](const Item& x, const Item& y) {
        return x.l2 != y.l2 ? x.l2 > y.l2 : x.l1 > y.l1;
      });
      for (int tb = low(Ma, Mb); tb <= J; tb += 4 * maxnp) {
        const int nout = std::min(2 * maxnp, (J - tb) / 2 + 1), np = (nout + 1) / 2;
        // rows [r0, r1) of each item that have a coefficient, and its cost
        struct Part {
          int r0, r1;
          long cost;
        };
        std::vector<Part> rows;
        long total = 0;
        for (const Item& it : items) {
          const int lo1 = low(it.m1.a, it.m1.b), lo2 = low(it.m2.a, it.m2.b);
          auto live = [&](int r) {
            int q;
            for (int k = 0; k < nout; ++k)
              for (int c = 0; c < it.l2; ++c)
                if (coef(lo1 + 2 * r, it.m1, lo2 + 2 * c, it.m2, tb + 2 * k, q) != 0.0) return true;
            return false;
          };
          Part p{0, it.l1, 0};
          while (p.r0 < p.r1 && !live(p.r0)) ++p.r0;
          while (p.r1 > p.r0 && !live(p.r1 - 1)) --p.r1;
          if (p.r1 > p.r0) p.cost = 30 + 4 * it.l2 + (long)(p.r1 - p.r0) * (8 + np * (4 * it.l2 + 8));
          total += p.cost;
          rows.push_back(p);
        }
        // What a record holds: one pair (m1, m2), or (wide, a single output) two of
        // one shape, the second for the warp's other half
        struct Unit {
          int a, b;
        };
        std::vector<Unit> units;
        const bool split = wide && nout == 1;
        for (int k = 0; k < (int)items.size(); ++k) {
          if (rows[k].r1 <= rows[k].r0) continue;
          auto shape = [&](int x) { return items[x].l2 * 16 + rows[x].r1 - rows[x].r0; };
          if (split) {
            auto it = std::find_if(units.begin(), units.end(), [&](const Unit& u) { return u.b < 0 && shape(u.a) == shape(k); });
            if (it != units.end()) {
              it->b = k;
              total -= rows[k].cost;
              continue;
            }
          }
          units.push_back({k, split ? -1 : k});
        }
        // two tasks of about equal cost, each with half of the pairs
        size_t next = 0;
        const int parts = total >= kYcWhole ? 2 : 1;
        for (int part = 0; part < parts; ++part) {
          const int task = (int)yc_cost.size();
          std::vector<int> rec(kYcTask, -1);
          rec[0] = (int)(yc_head.size() / kYcChunk);
          rec[2] = nout;
          rec[3] = parts == 1 ? 0 : 2 * (task - part) + 2 + part;
          for (int k = 0; k < nout; ++k) {
            const int t = tb + 2 * k, ma = (Ma + t) / 2, mb = (Mb + t) / 2, o = half_base(t) + mb * (t + 1) + ma;
            rec[4 + k] = o;
            if (Mb == 0 && Ma < 0) rec[4 + kYcOuts + k] = o + t - 2 * ma;
          }
          size_t pos = kYcChunk;  // words used of the open chunk
          auto open = [&] {
            yc_head.resize(yc_head.size() + kYcChunk, 0u);
            yc_cg.resize(yc_head.size(), 0.0);
            yc_trip.resize(yc_head.size(), -1);
            unsigned* h = &yc_head[yc_head.size() - kYcChunk];
            h[0] = (unsigned)task;
            h[1] = (unsigned)np;
            pos = 4;
          };
          open();
          long cost = 200;
          for (; next < units.size() && (part + 1 == parts || cost - 200 < total / 2); ++next) {
            const Unit u = units[next];
            const Item& it = items[u.a];
            const int l2p = (it.l2 + 1) & ~1, r0 = rows[u.a].r0, nrows = rows[u.a].r1 - r0;
            const size_t row = (size_t)np * l2p * 2 * cw;
            for (int r = 0; r < nrows;) {
              // four words are left at a chunk's end for the head that ends it
              size_t fit = pos + 8 <= kYcChunk ? (kYcChunk - 8 - pos) / row : 0;
              if (fit == 0) {
                open();
                fit = (kYcChunk - 8 - pos) / row;
              }
              const int n = (int)std::min<size_t>(fit, nrows - r);
              const size_t w0 = yc_head.size() - kYcChunk + pos;
              for (int h = 0; h < 2; ++h) {
                const int k = h == 0 || u.b < 0 ? u.a : u.b;
                const unsigned o1 = place(items[k].m1) + (unsigned)(rows[k].r0 + r) * 256u, o2 = place(items[k].m2);
                if (wide) yc_head[w0 + h] = yc_pack(o1) | yc_pack(o2) << 16;
                else yc_head[w0 + h] = h == 0 ? o1 : o2;
              }
              yc_head[w0 + 2] = (unsigned)n | (unsigned)it.l2 << 8;
              for (size_t w = w0 + 4; w < w0 + 4 + n * row; w += row, ++r)
                for (int o = 0; o < (wide ? 2 : nout); ++o) {
                  const int k = split && o == 1 ? u.b : u.a, out = split ? 0 : o;
                  if (k < 0 || out >= nout) continue;
                  const Item& p = items[k];
                  const int t1 = low(p.m1.a, p.m1.b) + 2 * (rows[k].r0 + r), lo2 = low(p.m2.a, p.m2.b);
                  for (int c = 0; c < p.l2; ++c) {
                    const size_t x =
                        wide ? w + ((size_t)o * l2p + c) * 2 : w + ((size_t)(o / 2) * l2p + c) * 2 + (o & 1);
                    yc_cg[x] = coef(t1, p.m1, lo2 + 2 * c, p.m2, tb + 2 * out, yc_trip[x]);
                  }
                }
              pos += 4 + n * row;
            }
            cost += rows[u.a].cost;
          }
          yc_head[yc_head.size() - kYcChunk] |= 0x80000000u;
          rec[1] = (int)(yc_head.size() / kYcChunk) - rec[0];
          yc_task.insert(yc_task.end(), rec.begin(), rec.end());
          yc_cost.push_back(cost);
        }
      }
    }
}

void HostTables::yc_list(std::vector<YcCoef>& coef, std::vector<YcGroup>& group) const {
  coef.clear();
  group.clear();
  std::vector<std::vector<YcCoef>> part(2 * kYcOuts);
  const unsigned* last = nullptr;
  int last_task = 0, outs = 0;
  auto flush = [&] {
    for (int o = 0; o < outs; ++o) {
      // the output of a half: the same one in (wide) tasks of a single output
      group.push_back({(int)coef.size(), last_task * kYcOuts + (yc_wide && yc_task[(size_t)last_task * kYcTask + 2] == 1 ? 0 : o)});
      coef.insert(coef.end(), part[o].begin(), part[o].end());
      part[o].clear();
    }
    outs = 0;
  };
  yc_rows([&](int k, const unsigned* head, int, size_t w, int o, int len) {
    if (head != last) flush();
    last = head;
    last_task = k;
    outs = std::max(outs, o + 1);
    for (int c = 0; c < len; ++c)
      if (yc_trip[w + 2 * c] >= 0) part[o].push_back({yc_cg[w + 2 * c], (int)(w + 2 * c), yc_trip[w + 2 * c]});
  });
  flush();
  group.push_back({(int)coef.size(), 0});
}

std::vector<unsigned> HostTables::yc_fixed(const double* beta) const {
  const std::vector<double> bw = beta_weights(beta);
  auto coef = [&](size_t x) { return yc_trip[x] < 0 ? 0.0 : yc_cg[x] * bw[yc_trip[x]]; };
  // the output of a half: the same one in tasks of a single output
  auto out_of = [&](size_t k, int h) { return yc_task[k * kYcTask + 2] == 1 ? 0 : h; };
  std::vector<double> top(yc_cost.size() * kYcOuts, 0.0);  // largest sum over a record of each output
  const unsigned* last[2] = {nullptr, nullptr};
  double sum[2] = {0.0, 0.0};
  yc_rows([&](int k, const unsigned* head, int, size_t w, int o, int len) {
    if (last[o] != head) sum[o] = 0.0;
    last[o] = head;
    for (int c = 0; c < len; ++c) sum[o] += std::fabs(coef(w + 2 * c));
    double& t = top[(size_t)k * kYcOuts + out_of(k, o)];
    if (!std::isnan(t) && !(sum[o] <= t)) t = sum[o];  // a NaN enters, and stays
  });
  std::vector<int> ex(top.size(), 0);  // top < 2^ex
  for (size_t k = 0; k < top.size(); ++k) {
    if (!std::isfinite(top[k])) ex[k] = kYcNan;
    else if (top[k] > 0.0) std::frexp(top[k], &ex[k]);
  }
  std::vector<unsigned> w(yc_head);
  for (size_t k = 0; k < yc_cost.size(); ++k)
    for (int ch = yc_task[k * kYcTask]; ch < yc_task[k * kYcTask] + yc_task[k * kYcTask + 1]; ++ch)
      for (int o = 0; o < 2; ++o) w[(size_t)ch * kYcChunk + 2 + o] = (unsigned)ex[k * kYcOuts + out_of(k, o)];
  yc_rows([&](int k, const unsigned*, int, size_t p, int o, int len) {
    const int e = ex[(size_t)k * kYcOuts + out_of(k, o)];
    for (int c = 0; c < len; ++c) {
      const long long v = e == kYcNan ? 0 : std::llrint(std::ldexp(coef(p + 2 * c), 60 - e));
      const int hi = (int)((v + (1LL << 29)) >> 30);
      w[p + 2 * c] = (unsigned)hi;
      w[p + 2 * c + 1] = (unsigned)(int)(v - hi * (1LL << 30));
    }
  });
  return w;
}

std::vector<int> HostTables::yc_bins(int nbins) const {
  // units: a task, or the two halves of a sum (they meet in one CTA)
  std::vector<std::array<int, 2>> unit;
  auto cost = [&](const std::array<int, 2>& u) { return yc_cost[u[0]] + (u[1] < 0 ? 0 : yc_cost[u[1]]); };
  for (int k = 0; k < (int)yc_cost.size(); ++k) {
    const bool two = yc_task[(size_t)k * kYcTask + 3] != 0;
    unit.push_back({k, two ? k + 1 : -1});
    if (two) ++k;
  }
  std::stable_sort(unit.begin(), unit.end(), [&](const auto& x, const auto& y) { return cost(x) > cost(y); });
  std::vector<std::vector<int>> bin(nbins);
  std::vector<long> load(nbins, 0);
  for (const auto& u : unit) {  // the next largest to the least loaded CTA
    const int b = (int)(std::min_element(load.begin(), load.end()) - load.begin());
    bin[b].push_back(u[0]);
    if (u[1] >= 0) bin[b].push_back(u[1]);
    load[b] += cost(u);
  }
  std::vector<int> out(1, 0);
  for (auto& b : bin) {
    std::stable_sort(b.begin(), b.end(), [&](int x, int y) { return yc_cost[x] > yc_cost[y]; });
    out.push_back(out.back() + (int)b.size());
  }
  for (const auto& b : bin) out.insert(out.end(), b.begin(), b.end());
  return out;
}

std::vector<double> HostTables::beta_weights(const double* beta) const {
  std::vector<double> w(ztrip.size());
  for (size_t q = 0; q < ztrip.size(); ++q) w[q] = ztrip[q].fac * beta[1 + ztrip[q].bidx];
  return w;
}

std::vector<double> HostTables::term_coef(const double* beta) const {
  const std::vector<double> bw = beta_weights(beta);
  std::vector<double> c(terms.size());
  for (size_t k = 0; k < terms.size(); ++k) c[k] = term_cg[k] * bw[term_trip[k]];
  return c;
}

std::vector<int> HostTables::bslices(int nslices) const {
  // contiguous runs of components with about equal term counts
  const long total = (long)bterms.size();
  std::vector<int> b(1, 0);
  int k = 1;
  for (int l = 0; l < ncoeff; ++l) {
    if (k < nslices && (long)bcomp_first[l + 1] * nslices >= total * k) {
      b.push_back(l + 1);
      ++k;
    }
  }
  while ((int)b.size() < nslices + 1) b.push_back(ncoeff);
  b[nslices] = ncoeff;
  return b;
}

std::vector<int> HostTables::bparts(int nparts, int* maxchunks, int* maxterms) const {
  const std::vector<int> b = bslices(nparts);
  int mx = 0, mt = 0;
  for (int k = 0; k < nparts; ++k) {
    const int c0 = bcomp_chunk[b[k]], c1 = bcomp_chunk[b[k + 1]];
    mx = std::max(mx, c1 - c0);
    mt = std::max(mt, bchunk_term[c1] - bchunk_term[c0]);
  }
  *maxchunks = mx;
  *maxterms = mt;
  return b;
}

std::vector<int> HostTables::lane_outputs(int lanes, int* m) const {
  std::vector<int> ord(H);
  for (int o = 0; o < H; ++o) ord[o] = o;
  auto nterm = [&](int o) { return term_out_first[o + 1] - term_out_first[o]; };
  std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) { return nterm(x) > nterm(y); });
  const int mm = (H + lanes - 1) / lanes;
  std::vector<int> t((size_t)lanes * mm, -1);
  for (int k = 0; k < H; ++k) {
    const int round = k / lanes, pos = k % lanes;
    const int lane = (round & 1) ? lanes - 1 - pos : pos;
    t[(size_t)lane * mm + round] = ord[k];
  }
  *m = mm;
  return t;
}

std::vector<unsigned> HostTables::bwords(bool cp) const {
  std::vector<unsigned> w(bdev.size(), 0u);
  for (size_t q = 0; q < bdev.size(); ++q) {
    const unsigned t = bdev[q];
    const unsigned i1 = t & 1023u, i2 = (t >> 10) & 1023u, c1 = (t >> 20) & 1u, c2 = (t >> 21) & 1u;
    unsigned x = cp ? (((i2 + c2 * (unsigned)H) << 8) | ((i1 + c1 * (unsigned)H) << 19))
                    : ((i2 << 8) | (i1 << 18) | (c1 << 30) | (c2 << 31));
    if (bdev_o[q] >= 0) {
      const unsigned o = (unsigned)bdev_o[q];
      if (o > 1023u) return {};  // not reached for 2J <= 14 (H = 652)
      x |= (o & 0xFFu) | ((o >> 8) << (cp ? 30 : 28));
    }
    w[q] = x;
  }
  return w;
}

}  // namespace snap
