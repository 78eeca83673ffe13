// snap_tables.h -- host-side tables of the library (see snap_tables.cpp).
#pragma once
#include <vector>

#include "snap_internal.h"

namespace snap {

struct ZTrip {
  int t1, t2, t;  // Y triple: Z^t_{t1 t2} with t1 >= t2
  int cg_off;     // offset of its cg[x1][x2] block
  int bidx;       // canonical bispectrum component it belongs to
  double fac;     // multiplicity / rank factor of the derivative
};

struct HostTables {
  int twojmax = 0, H = 0, ncoeff = 0;
  std::vector<int> half_tmm;
  std::vector<ZTrip> ztrip;
  std::vector<double> cg;
  // compute_Y terms: packed indices/flags, CG product with signs, triple
  std::vector<unsigned> terms;
  std::vector<double> term_cg;
  std::vector<int> term_trip;
  std::vector<int> term_out_first;  // [H+1] first term of every output
  // bispectrum terms (records as above, coefficient without beta), the U
  // element of each output group, and the first term of each component
  std::vector<unsigned> bterms;
  std::vector<double> bterm_coef;
  std::vector<int> bout;
  std::vector<int> bcomp_first;
  std::vector<int> bgroup_first;  // [ncoeff+1] first output group of each component
  // the bispectrum term list cut into chunks of whole output groups (about
  // kBChunk terms, never across a component): first term and first group of
  // every chunk (+1 end entry each) and the first chunk of every component
  std::vector<int> bchunk_term, bchunk_group, bcomp_chunk;
  // The device order of the bispectrum terms: within every chunk each output
  // group cut into pieces of at most kBGroupMax terms (near-equal lengths),
  // the pieces ordered by length (stably), so that the device walks runs of
  // equal-length pieces with branch-free bodies.  Chunks keep their term
  // ranges.  bdev: the table words (as bterms, without the end bits);
  // bdev_coef: their coefficients; bdev_o: the U element of each term's
  // piece, -1 on all but a piece's first term; bchunk_runs [nchunks]
  // [kBGroupMax]: the number of pieces of 1, 2, ... terms of every chunk.
  std::vector<unsigned> bdev;
  std::vector<double> bdev_coef;
  std::vector<int> bdev_o;
  std::vector<unsigned short> bchunk_runs;
  // [H]: S_t(ma, mb) = sqrt((t - ma)! ma! / (t - mb)!) of every half-layout
  // element, the factor between the scaled recursion's v and u
  std::vector<double> half_scale;

  // The closed form of u (snap_pairs.cuh): the steps (p, q, k) of the classes
  // (p, q), p + q <= 2J, in the order p rising, q falling, k rising.
  // pair_idx: the half-layout elements of the step, bits 0-9 (ma, mb) = (k,
  //   k + q), bit 10 conjugated and bit 11 negated when it is read through its
  //   mirror, bits 12-21 (k + q, k) with bit 22 set when it is another element
  //   (p, q > 0);
  // pair_norm: n s_k, u = n s_k monomial P_k(x);
  // pair_weight: the step's weight in a full-matrix contraction (2; 1 for p =
  //   q = 0);
  // pair_ab: alpha_{k-1}, beta_{k-1} of the recursion to P_k (0, 0 at k = 0);
  // with alpha and beta rounded to FP32 the recursion gives other polynomials PP:
  // P_k = (1 + d_kk) (PP_k + sum_{j < k} f_kj PP_j).  pair_fix: [kPairFix] a step
  //   j, f_kj at k - j (0 at 0 and past the class); pair_norm_fix: pair_norm (1 +
  //   d_kk).
  std::vector<unsigned> pair_idx;
  std::vector<double> pair_norm, pair_norm_fix, pair_weight, pair_ab, pair_fix;
  // What the kernels take of these.  pair_scales: a step's step_scale, norm (x
  // weight), and pair_recursion: its rec_ab (snap_closed.cuh), in FP32 with what
  // the rounding leaves off; pair_classes: the classes of several steps, longest
  // first, first step | steps << 16.
  std::vector<double> pair_scales(bool fp64, bool weighted) const;
  std::vector<double> pair_recursion(bool fp64) const;
  std::vector<int> pair_classes() const;
  // compute_U's units (snap_u.cu): [nunits][kUUnit] the steps K of its classes,
  // their number M, and per class p | q << 4 | first step << 8; longest first:
  // u_nunits of about equal work, then each class by itself.  u_cost: about the
  // multiply-adds of all classes for a pair.
  std::vector<int> u_units;
  int u_nunits = 0, u_cost = 0;

  // compute_Y (yc_kernel, snap_kernels.cu).  With m = (2 ma -
  // t, 2 mb - t) the doubled projections of an element, the elements of every
  // rank t with one m are its vector u[m]; the outputs with one M are a class,
  // and its Y is a sum over the unordered pairs m1 + m2 = M of bilinear forms
  //   Y_t[M] += sum_t1 u_t1[m1] sum_t2 c[t][t1][t2] u_t2[m2].
  // yc_slot: [H] position of each half-layout element when the vectors are
  //   stored one after the other, t rising (a vector with m_b > 0 is the mirror
  //   of a stored one: conjugated, its sign folded into c);
  // yc_task: [ntask][kYcTask] first chunk, chunks, outputs, half, the output
  //   elements (up to kYcOuts), and the element each zeroes (the mirror below
  //   the centre of the middle column) or -1; a task has outputs of one class,
  //   at most kYcOuts (wide: 2) of them, and all pairs m1 + m2 = M (half = 0) or
  //   half of them (two tasks k, k + 1 with half = 2 k + 2 and 2 k + 3);
  // the stream, kYcChunk words a chunk: word 0 the task (bit 31: its last
  //   chunk), word 1 the output pairs np of the task, words 2-3 zero, then
  //   records: a head {byte offset of u[m1] (bit 31: conjugate), the same of
  //   u[m2], rows | length of u[m2] << 8, 0} and per row (t1) np x (length
  //   rounded up to even) coefficient pairs (outputs 2k, 2k + 1); a head with
  //   no rows ends the chunk.  yc_head holds the words that are not
  //   coefficients, yc_cg / yc_trip the coefficients without beta and their
  //   triples (-1: not one);
  // yc_cost: about the instructions of each task.
  // wide (the FP64 path): a coefficient is two words (yc_cg / yc_trip at the
  // first), a row 2 halves x (length rounded up to even), np = 1, words 2-3 of a
  // chunk are the exponents of its task's outputs (yc_fixed), and words 0-1 of a
  // head are for a warp's two halves, u[m1] in the lower and u[m2] in the upper 16
  // bits (slot, bit 15: conjugate).  The halves take the two outputs of a task,
  // from one pair (m1, m2), or, in a task of one output, two pairs of one shape.
  std::vector<int> yc_slot, yc_task, yc_trip;
  std::vector<unsigned> yc_head;
  std::vector<double> yc_cg;
  std::vector<long> yc_cost;
  bool yc_wide = false;
  void build_classes(bool wide);
  // frees yc_head, yc_cg and yc_trip (once they are on the device)
  void drop_stream() {
    std::vector<unsigned>().swap(yc_head);
    std::vector<double>().swap(yc_cg);
    std::vector<int>().swap(yc_trip);
  }
  // f(task, word, output, rows' elements) over every row of every output: the
  // coefficient of element c is at word + c * stride
  template <typename F>
  void yc_rows(F&& f) const {
    const int cw = yc_wide ? 2 : 1;
    for (size_t k = 0; k < yc_cost.size(); ++k) {
      const int* rec = &yc_task[k * kYcTask];
      for (int ch = rec[0]; ch < rec[0] + rec[1]; ++ch) {
        const size_t base = (size_t)ch * kYcChunk;
        const int np = (int)yc_head[base + 1];
        for (size_t p = base + 4; (yc_head[p + 2] & 255u) != 0;) {
          const unsigned* head = &yc_head[p];
          const int len = (int)(head[2] >> 8), lp = (len + 1) & ~1;
          p += 4;
          for (int r = 0; r < (int)(head[2] & 255u); ++r, p += (size_t)np * lp * 2 * cw)
            for (int o = 0; o < 2 * np; ++o)
              f((int)k, head, r, yc_wide ? p + (size_t)o * lp * 2 : p + (size_t)(o / 2) * lp * 2 + (o & 1), o, len);
        }
      }
    }
  }
  // The stream's coefficients in the order of their records and outputs (output
  // after output, row after row), and the groups of a record and an output; a
  // last group with first = their number ends the list.
  void yc_list(std::vector<YcCoef>& coef, std::vector<YcGroup>& group) const;
  // The stream's words of the FP64 path with the coefficients of beta in 60-bit
  // fixed point, scaled by the power of two above each output's largest sum of
  // their sizes over a record (kYcNan: not finite, the output is not a number):
  // what launch_yc_coefs does on the device.
  std::vector<unsigned> yc_fixed(const double* beta) const;
  // The tasks dealt to nbins CTAs of about equal cost, decreasing in each:
  // nbins + 1 offsets, then the tasks
  std::vector<int> yc_bins(int nbins) const;

  void build(int twojmax);
  // the list of terms (terms, term_*), which only the warp-per-atom compute_Y walks
  void build_terms();
  std::vector<double> beta_weights(const double* beta) const;
  std::vector<double> term_coef(const double* beta) const;
  // outputs dealt to `lanes` lanes in decreasing term count, snake order:
  // [lanes][m] output indices, -1 past a lane's last; m returned in *m
  std::vector<int> lane_outputs(int lanes, int* m) const;
  std::vector<int> bslices(int nslices) const;
  // nparts contiguous runs of components with about equal term counts (entry
  // k = first component of run k, entry nparts = ncoeff); *maxchunks = the
  // most chunks of one run
  // and *maxterms = the most terms of one run
  std::vector<int> bparts(int nparts, int* maxchunks, int* maxterms) const;
  // The bispectrum records' words as the device reads them (one per term of
  // the device order):
  //   cp = false (factors' stored elements, imaginary parts flipped by flag):
  //     bits 8-17 second factor, 18-27 first factor, 30 conjugate the first
  //     factor, 31 conjugate the second; a piece's U element in bits 0-7
  //     (low) and 28-29 (high) of its first word
  //   cp = true (factors in a [2][H] plane, conjugates in the second half):
  //     bits 8-18 second factor, 19-29 first factor; the piece's U element in
  //     bits 0-7 and 30-31 of its first word
  // Empty if an element does not fit in 10 bits.
  std::vector<unsigned> bwords(bool cp) const;
};

double clebsch_gordan(int tj1, int tm1, int tj2, int tm2, int tj, int tm);
int count_coeff(int twojmax);

// One atom's pairs in the fused dE's arithmetic, on the host (snap_col_*.cu).
template <typename R>
int pair_host(const HostTables& tab, int npairs, const double* par, const double* y, double* out);

}  // namespace snap
