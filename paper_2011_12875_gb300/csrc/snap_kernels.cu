// snap_kernels.cu -- compute_Y, the bispectrum and the force gather.
//
// Notation follows arXiv:2011.12875: t = 2j, U_t = Ulisttot, Y_t = adjoint
// (Eq. y), dE_i/dr_ik = Re sum_t Y_t : conj(dU_t/dr_ik) (Eq. snapforce2).
// R is the working precision of the recursions: float (mixed) or double.
// Every CTA works on a fixed set of atoms and writes each output once, so the
// results are deterministic; there are no global atomics in the data path.
#include <math.h>

#include <algorithm>
#include <utility>

#include "snap_geom.cuh"
#include "snap_internal.h"

namespace snap {

namespace {

constexpr unsigned kFull = 0xffffffffu;

template <typename R>
struct __align__(2 * sizeof(R)) cx {
  R re, im;
};

template <typename R>
__device__ __forceinline__ cx<R> mk(R re, R im) {
  cx<R> c;
  c.re = re;
  c.im = im;
  return c;
}
// x * y + z with one rounding (complex multiply-adds are written as chains
// of these, two a component)
template <typename R>
__device__ __forceinline__ R fmr(R x, R y, R z) {
  if constexpr (sizeof(R) == 4) return fmaf(x, y, z);
  else return fma(x, y, z);
}

template <typename R>
__device__ __forceinline__ R warp_sum(R v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Weight of a half-layout element in a full-matrix contraction M : N* of two
// matrices with the inversion symmetry: 2 for mb < t/2; on the middle column
// (2 mb = t) 2 above the centre, 1 at the centre, 0 below.
__device__ __forceinline__ int half_weight(int t, int ma, int mb) {
  if (2 * mb < t) return 2;
  return ma < mb ? 2 : (ma == mb ? 1 : 0);
}

// ------------------------------------------- staging (bulk copies, waits)

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
// Orders this thread's ordinary accesses to shared memory before bulk copies
// into it (the async proxy) that are issued after the next barrier: a barrier by
// itself does not order the two.
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned phase) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(phase)
      : "memory");
  return ok != 0;
}

// Bounded waits.  A wait gives up after kWaitNs of the global timer (or
// kSpinCap polls, whichever comes first), so a copy that never completes
// cannot hang the GPU: the kernel raises an error flag and returns, and the
// call reports SNAP_ERR_TIMEOUT.
constexpr unsigned long long kWaitNs = 1000000000ull;  // 1 s
constexpr unsigned kSpinCap = 1u << 28;

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, unsigned phase, unsigned long long limit_ns) {
  const unsigned long long t0 = global_ns();
  for (unsigned it = 0; it < kSpinCap; ++it) {
    if (mbar_try_wait(bar, phase)) return true;
    if ((it & 63u) == 63u && global_ns() - t0 > limit_ns) return false;
  }
  return false;
}

// Stage `bytes` from global `src` into shared `dst` with one bulk (TMA) copy
// completed on the mbarrier `bar`, issued by thread 0; every thread of the
// CTA waits, bounded.  The outcome is made CTA-uniform.  On a timeout the CTA
// raises flags[3] and waits once more, again bounded, for the copy it issued
// (if that second wait runs out too, the copy may still land in the exiting
// CTA's shared memory).  skip_copy registers the bytes without issuing the
// copy: a test hook under which the wait runs out with nothing in flight.
// `overlap()` runs on every thread while the copy is in flight.
// With src2 given, a second block of `bytes` from src2 lands at dst + off2
// (right after the first when off2 is 0) on the same barrier.
// With src3 given, bytes3 from src3 land at dst + off3, on the same barrier.
template <typename F>
__device__ bool stage_bulk(void* dst, const void* src, unsigned bytes, uint64_t* bar, int* flags,
                           bool skip_copy, F&& overlap, const void* src2 = nullptr, unsigned off2 = 0,
                           const void* src3 = nullptr, unsigned bytes3 = 0, unsigned off3 = 0) {
  if (threadIdx.x == 0) mbar_init(bar, 1);
  __syncthreads();
  if (threadIdx.x == 0) {
    mbar_expect_tx(bar, (src2 ? 2 * bytes : bytes) + (src3 ? bytes3 : 0u));
    if (!skip_copy) {
      bulk_g2s(dst, src, bytes, bar);
      if (src2) bulk_g2s(static_cast<char*>(dst) + (off2 ? off2 : bytes), src2, bytes, bar);
      if (src3) bulk_g2s(static_cast<char*>(dst) + off3, src3, bytes3, bar);
    }
  }
  overlap();
  const bool ok = __syncthreads_and(mbar_wait_bounded(bar, 0, kWaitNs));
  if (!ok) {
    if (threadIdx.x == 0) atomicMax(&flags[3], 1);
    mbar_wait_bounded(bar, 0, kWaitNs / 4);
  }
  return ok;
}

// v with its sign bit XORed with bit 31 of m
__device__ __forceinline__ float flip_sign(float v, unsigned m) {
  return __int_as_float(__float_as_int(v) ^ (int)m);
}
__device__ __forceinline__ double flip_sign(double v, unsigned m) {
  return __longlong_as_double(__double_as_longlong(v) ^ ((long long)m << 32));
}

template <typename R>
struct YAcc {
  R re, im;  // the output element
  R ar, ai;  // sum of coef * second factor over the current group
};

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ------------------------------------------- compute_Y by classes
// The terms of Eq. (y) ordered for registers.  An element's doubled
// projections m = (2 ma - t, 2 mb - t) add up in a product, so the outputs of
// all ranks t with one M are a sum over the pairs m1 + m2 = M of bilinear forms
//   Y_t[M] += sum_t1 u_t1[m1] sum_t2 c[t][t1][t2] u_t2[m2]
// of two short vectors (at most J + 1 ranks): both are loaded once, and up to
// 8 x 8 x 8 coefficients used on them (HostTables::build_classes, whose stream
// of heads and coefficients a warp walks).  Lanes are the 32 atoms of a block;
// a warp takes a class (a task) at a time and keeps its outputs in registers.
//
// The arithmetic is packed (fma.rn.f32x2) over two outputs t, t + 2: the
// coefficients come in such pairs, so nothing but u has to be duplicated.
//
// The list of terms it replaces took three 128-byte wavefronts of shared memory
// a term (its record and 8 bytes a lane of the factor) for two FMAs, and was
// bound by them; here a term takes a quarter of a wavefront (coefficients, four
// a load) and the vectors about 0.4.  The dense forms hold 7% of zero
// coefficients at 2J14.  What bounds it now is issue: a packed FMA (two cycles of
// its pipe) comes with 1.6 other instructions (unpacking the vectors, heads,
// loops), on 16 warps an SM (2J14, 2000 atoms: issue slots 62% used, shared
// memory 59%, FMA pipe 52%).
// Measured, list of terms -> now: FP32, 2000 atoms, 2J8 41 -> 34 us, 2J11 199 ->
// 119, 2J14 845 -> 388; 16000 atoms, 2J8 218 -> 178, 2J14 6005 -> 2809; FP64 (in
// fixed point, below), 2000 atoms, 2J8 404 -> 170, 2J11 2390 -> 821, 2J14 9344 ->
// 3042; 128 atoms, 2J8 119 -> 28.
// Chunks of a warp's ring
__host__ __device__ constexpr int yc_slots(int rsize) { return rsize == 8 ? 2 : 3; }
// Warps of a CTA: one CTA an SM above 2J = 9 (the block's U fills its shared
// memory), two up to there, with the registers that FP32 and fixed point (96)
// need.  FP32 up to 2J = 8: with sixteen warps the tasks left most of them waiting
// for the largest, and their rings took half of the shared memory; sixteen /
// eight, us: 2J4 2000 atoms 14.2 / 10.0, 5488 22.5 / 18.2; 2J6 22.3 / 16.3, 39.0 / 32.4;
// 2J8 35.1 / 33.8, 75.7 / 71.4, 16000 atoms 178.3 / 178.0; but 2J9 49.1 / 54.5, 113 / 121.
__host__ __device__ constexpr int yc_warps(int rsize, int H) {
  return rsize == 4 ? (H <= half_size(8) ? 8 : 16) : H <= half_size(9) ? 10 : 20;
}

typedef unsigned long long f2;  // two FP32

__device__ __forceinline__ f2 f2_pack(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 f2_get(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// A record's head, unpacked
struct YcHead {
  uint4 h;
  __device__ __forceinline__ explicit YcHead(const unsigned* p) : h(*reinterpret_cast<const uint4*>(p)) {}
  __device__ __forceinline__ int rows() const { return (int)(h.z & 255u); }
  __device__ __forceinline__ int len() const { return (int)(h.z >> 8); }
};

// The records of one length L from p on (h: the first one's head): NP output
// pairs, rows (t1) of L elements of u[m2].  The next head and the next row's
// factor are read ahead.
template <int NP, int L>
__device__ __forceinline__ void yc_run(const unsigned* __restrict__& p, YcHead& h, const char* __restrict__ ul,
                                       f2 (&yr)[NP], f2 (&yi)[NP]) {
  constexpr int LP = (L + 1) & ~1, ROW = NP * LP * 2;
  do {
    const int rows = h.rows();
    const char* u1 = ul + (h.h.x & 0x7FFFFFFFu);
    const char* u2 = ul + (h.h.y & 0x7FFFFFFFu);
    const unsigned c1 = h.h.x & 0x80000000u, c2 = h.h.y & 0x80000000u;
    const unsigned* q = p + 4;
    p = q + rows * ROW;
    h = YcHead(p);
    float2 v = *reinterpret_cast<const float2*>(u1);
    f2 ar[L], ai[L];
#pragma unroll
    for (int c = 0; c < L; ++c) {
      const float2 w = *reinterpret_cast<const float2*>(u2 + c * 256);
      const float im = flip_sign(w.y, c2);
      ar[c] = f2_pack(w.x, w.x);
      ai[c] = f2_pack(im, im);
    }
#pragma unroll 1
    for (const unsigned* end = p; q != end; q += ROW) {
      const float im = flip_sign(v.y, c1);
      const f2 x = f2_pack(v.x, v.x), y = f2_pack(im, im), ny = f2_pack(-im, -im);
      u1 += 256;  // one row past the vector at the end, inside the CTA's shared memory
      v = *reinterpret_cast<const float2*>(u1);
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        f2 br, bi;
#pragma unroll
        for (int c = 0; c < L; c += 2) {
          const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(q + (k * LP + c) * 2);
          br = c == 0 ? f2_mul(w.x, ar[c]) : f2_fma(w.x, ar[c], br);
          bi = c == 0 ? f2_mul(w.x, ai[c]) : f2_fma(w.x, ai[c], bi);
          if (c + 1 < L) {
            br = f2_fma(w.y, ar[c + 1], br);
            bi = f2_fma(w.y, ai[c + 1], bi);
          }
        }
        yr[k] = f2_fma(x, br, yr[k]);
        yi[k] = f2_fma(x, bi, yi[k]);
        yr[k] = f2_fma(ny, bi, yr[k]);
        yi[k] = f2_fma(y, br, yi[k]);
      }
    }
  } while (h.len() == L);
}

// Running sums of a task's output pairs, and (long sums, 2J > 9) what their
// roundings lost.
template <int NPM, bool COMP>
struct YcSum {
  f2 r[NPM], i[NPM], er[COMP ? NPM : 1], ei[COMP ? NPM : 1];
};
// s += x (COMP: Kahan's sum, e the part of s that is too much)
template <bool COMP>
__device__ __forceinline__ void yc_add(f2& s, f2& e, f2 x) {
  if constexpr (COMP) {
    const f2 minus = f2_pack(-1.f, -1.f);
    const f2 y = f2_fma(minus, e, x), t = f2_add(s, y);
    e = f2_fma(minus, y, f2_fma(minus, s, t));
    s = t;
  } else {
    s = f2_add(s, x);
  }
}

// The records of a chunk (from word 4) of a task with NP output pairs.  A
// chunk's terms are summed by themselves and then added to the outputs.  The
// list of terms summed each output in one go; its largest error in Y, relative
// to the largest Y, was 1.2e-6 at 2J8 and 3.3e-6 at 2J14, here 4e-7 and 6e-7
// (one long sum in this order: 1.4e-6 and 1.9e-6).
template <int NP, int LM, int NPM, bool COMP>
__device__ __forceinline__ void yc_chunk(const unsigned* __restrict__ p, const char* __restrict__ ul,
                                         YcSum<NPM, COMP>& s) {
  f2 yr[NP], yi[NP];
#pragma unroll
  for (int k = 0; k < NP; ++k) yr[k] = yi[k] = 0;
  YcHead h(p);
  while (h.rows() != 0) {
    switch (h.len()) {
#define SNAP_YC(L) \
  case L: \
    if constexpr (L <= LM) yc_run<NP, L>(p, h, ul, yr, yi); \
    break;
      SNAP_YC(1) SNAP_YC(2) SNAP_YC(3) SNAP_YC(4) SNAP_YC(5) SNAP_YC(6) SNAP_YC(7) SNAP_YC(8)
#undef SNAP_YC
      default: return;
    }
  }
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    yc_add<COMP>(s.r[k], s.er[COMP ? k : 0], yr[k]);
    yc_add<COMP>(s.i[k], s.ei[COMP ? k : 0], yi[k]);
  }
}

// The two precisions of the walk below: what a task's outputs are held in, how
// a chunk adds to them and how they are stored.
template <int LM, int WARPS>
struct YcSingle {
  static constexpr int kAtoms = 32;  // of a block; a row is their [32] of an element
  static constexpr int kWarps = WARPS;  // of a CTA
  static constexpr int kSlots = yc_slots(4);
  static constexpr int NPM = LM > 5 ? 4 : 2;
  static constexpr bool COMP = LM > 5;
  YcSum<NPM, COMP> y;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < NPM; ++k) y.r[k] = y.i[k] = y.er[COMP ? k : 0] = y.ei[COMP ? k : 0] = 0;
  }
  __device__ __forceinline__ void chunk(unsigned np, const unsigned* __restrict__ p, const char* __restrict__ ul, int) {
    switch (np) {
#define SNAP_YC(NP) \
  case NP: \
    if constexpr (NP <= NPM) yc_chunk<NP, LM, NPM, COMP>(p, ul, y); \
    break;
      SNAP_YC(1) SNAP_YC(2) SNAP_YC(3) SNAP_YC(4)
#undef SNAP_YC
      default: break;
    }
  }
  // the outputs, plus those at `other` if it is given, to Yb
  __device__ __forceinline__ void store(const int* __restrict__ rec, uint4, char* Yb, const char* other, int lane,
                                        int) const {
    cx<float>* Yg = reinterpret_cast<cx<float>*>(Yb) + lane;
    const int nout = __ldg(rec + 2);
#pragma unroll
    for (int k = 0; k < NPM; ++k) {
      const float2 r = f2_get(y.r[k]), i = f2_get(y.i[k]);
#pragma unroll
      for (int o = 0; o < 2; ++o)
        if (2 * k + o < nout) {
          const int at = __ldg(rec + 4 + 2 * k + o) * 32;
          cx<float> v = o == 0 ? mk<float>(r.x, i.x) : mk<float>(r.y, i.y);
          if (other) {
            const cx<float> w = reinterpret_cast<const cx<float>*>(other)[at + lane];
            v = mk<float>(v.re + w.re, v.im + w.im);
          }
          Yg[at] = v;
          // the mirror below the centre of the middle column, which no
          // contraction reads
          const int z = __ldg(rec + 4 + kYcOuts + 2 * k + o);
          if (z >= 0) Yg[z * 32] = mk<float>(0.f, 0.f);
        }
    }
  }
};

// FP64 in fixed point.  The FP64 pipe does a warp's multiply-add in 15 cycles
// of an SM; the integer pipe a 32 x 32 + 64 bit one in half a cycle.  So the
// block's U and the coefficients are held as two limbs (59 bits and a sign,
// more than the 53 of a double) and a product is three integer multiply-adds,
// hi hi and the two cross ones; the fourth is below the last bit.
//   u = (h 2^30 + l) 2^(s - 59), |h| <= 2^29, |l| <= 2^29, 2^s above the atom's
//     largest component of U (yc_limbs; rounded to nearest, exact for components
//     above 2^-6 of the largest: of a thermal BCC atom's at 2J14, about half);
//   c = (h 2^30 + l) 2^(e - 60), |l| <= 2^29, 2^e above the largest sum of |c|
//     over a record (m1, m2) of its output;
//   a row's sum A = sum_t2 c u is rounded at 2^-59 and split into h, l again,
//     and u A, formed in the same way and summed over the record, is added to
//     the output's 96-bit sum, which is exact.
// Sums of a record stay below 2^63: with sum |h(c)| <= 2^30 and |A| <= 2^59,
//   hi hi: 2^59, 2 x 2^59; cross: 2^59 + 8 2^58, 2 (8 2^58 + 2^59).
// A rounding here is 2^-59 of the largest |U| (twice in a product) times the
// largest sum of |c|, where FP64 rounds at 2^-53 of each partial sum: what is
// large in Y is closer than in FP64, an element far below the rest of its atom's
// Y, or one that only coefficients far below an output's largest feed, has fewer
// correct bits than its own size would allow.  dE/dr and the energy sum over
// all of Y, so they are as close as in FP64.  Error of a step's energies /
// forces against 64 bits (root mean square over that of the exact ones, eight
// inputs), FP64 list of terms and layer recursion -> fixed point and closed forms:
// 2J8 2000 atoms 9.2e-16 / 5.8e-15 -> 7.9e-16 / 5.4e-15, 2J14 2.6e-15 / 6.5e-15 ->
// 2.1e-15 / 6.3e-15, 2J4 250 atoms 6.5e-16 / 5.5e-15 -> 6.0e-16 / 5.0e-15.
//
// A block is 16 atoms (a row of 16 x 16 bytes is then 256, as in FP32, and the
// whole of 2J14 stays in shared memory); a warp's halves take the two outputs
// of a task, or halves of the pairs of a single one (the classes' odd outputs:
// with a half idle there, 2J8 took 197 us and 2J14 3390).
__device__ __forceinline__ void wide_add(long long& s, int x, int y) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s) : "r"(x), "r"(y));
}

struct Acc96 {
  unsigned lo, mid, hi;
  __device__ __forceinline__ void add(long long v) {
    const unsigned l = (unsigned)v, h = (unsigned)(v >> 32), s = (unsigned)((int)h >> 31);
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(lo), "+r"(mid), "+r"(hi)
        : "r"(l), "r"(h), "r"(s));
  }
  __device__ __forceinline__ void add(const Acc96& v) {
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(lo), "+r"(mid), "+r"(hi)
        : "r"(v.lo), "r"(v.mid), "r"(v.hi));
  }
  __device__ __forceinline__ double value() const {
    return fma((double)(long long)(((unsigned long long)hi << 32) | mid), 4294967296.0, (double)lo);
  }
};

// the sum of the lane in the warp's other half
__device__ __forceinline__ Acc96 shfl16(const Acc96& v) {
  return Acc96{__shfl_xor_sync(kFull, v.lo, 16), __shfl_xor_sync(kFull, v.mid, 16), __shfl_xor_sync(kFull, v.hi, 16)};
}

// hi hi and cross sums to one number, rounded (the cross sum starts at half
// of 2^30), plus 2^29
constexpr long long kYcRound = 1LL << 29, kYcSplit = kYcRound + (1LL << 59);

// yc_run in fixed point: one output a lane
template <int L>
__device__ __forceinline__ void yf_run(const unsigned* __restrict__& p, YcHead& h, const char* __restrict__ ul, int half,
                                       Acc96& yr, Acc96& yi) {
  constexpr int LP = (L + 1) & ~1, ROW = LP * 4;
  do {
    const unsigned at = half ? h.h.y : h.h.x;
    const char* u1 = ul + ((at & 0x7FFFu) << 8);
    const char* u2 = ul + ((at >> 8) & 0x7FFF00u);
    // conj(u1) v = conj(u1 conj(v)): u[m1] is taken as it is
    const int c1 = (int)(at << 16) >> 31, c2 = c1 ^ ((int)at >> 31);  // -1: conjugate
    const unsigned* q = p + 4 + half * LP * 2;
    p += 4 + h.rows() * ROW;
    const unsigned* end = p + half * LP * 2;
    h = YcHead(p);
    int4 v = *reinterpret_cast<const int4*>(u1);
    int4 a[L];
#pragma unroll
    for (int c = 0; c < L; ++c) {
      a[c] = *reinterpret_cast<const int4*>(u2 + c * 256);
      a[c].z = (a[c].z ^ c2) - c2;
      a[c].w = (a[c].w ^ c2) - c2;
    }
    long long ph = 0, qh = 0, pc = kYcRound, qc = kYcRound;
#pragma unroll 1
    for (; q != end; q += ROW) {
      const int4 x = v;
      u1 += 256;  // one row past the vector at the end, inside the CTA's shared memory
      v = *reinterpret_cast<const int4*>(u1);
      long long rh = 0, rc = kYcSplit, ih = 0, ic = kYcSplit;
#pragma unroll
      for (int c = 0; c < L; c += 2) {
        const int4 w = *reinterpret_cast<const int4*>(q + c * 2);
        wide_add(rh, w.x, a[c].x);
        wide_add(ih, w.x, a[c].z);
        wide_add(rc, w.x, a[c].y);
        wide_add(ic, w.x, a[c].w);
        wide_add(rc, w.y, a[c].x);
        wide_add(ic, w.y, a[c].z);
        if (c + 1 < L) {
          wide_add(rh, w.z, a[c + 1].x);
          wide_add(ih, w.z, a[c + 1].z);
          wide_add(rc, w.z, a[c + 1].y);
          wide_add(ic, w.z, a[c + 1].w);
          wide_add(rc, w.w, a[c + 1].x);
          wide_add(ic, w.w, a[c + 1].z);
        }
      }
      int Ah, Al, Bh, Bl;
      split30(rh + (rc >> 30), Ah, Al);
      split30(ih + (ic >> 30), Bh, Bl);
      const int nz = -x.z, nw = -x.w;
      wide_add(ph, x.x, Ah);
      wide_add(qh, x.x, Bh);
      wide_add(pc, x.x, Al);
      wide_add(qc, x.x, Bl);
      wide_add(ph, nz, Bh);
      wide_add(qh, x.z, Ah);
      wide_add(pc, x.y, Ah);
      wide_add(qc, x.y, Bh);
      wide_add(pc, nz, Bl);
      wide_add(qc, x.z, Al);
      wide_add(pc, nw, Bh);
      wide_add(qc, x.w, Ah);
    }
    yr.add(ph + (pc >> 30));
    const long long q2 = qh + (qc >> 30);
    yi.add((q2 ^ c1) - c1);
  } while (h.len() == L);
}

constexpr int kYcBad = 1 << 20;
template <int LM, int WARPS>
struct YcFixed {
  static constexpr int kAtoms = 16;
  static constexpr int kWarps = WARPS;
  static constexpr int kSlots = yc_slots(8);
  Acc96 yr, yi;
  __device__ __forceinline__ void clear() { yr = yi = Acc96{0u, 0u, 0u}; }
  __device__ __forceinline__ void chunk(unsigned, const unsigned* __restrict__ p, const char* __restrict__ ul, int half) {
    YcHead h(p);
    while (h.rows() != 0) {
      switch (h.len()) {
#define SNAP_YC(L) \
  case L: \
    if constexpr (L <= LM) yf_run<L>(p, h, ul, half, yr, yi); \
    break;
        SNAP_YC(1) SNAP_YC(2) SNAP_YC(3) SNAP_YC(4) SNAP_YC(5) SNAP_YC(6) SNAP_YC(7) SNAP_YC(8)
#undef SNAP_YC
        default: return;
      }
    }
  }
  // `ex`: the exponent of the lane's atom, or kYcBad
  __device__ __forceinline__ void store(const int* __restrict__ rec, uint4 h, char* Yb, const char* other, int lane,
                                        int ex) const {
    const int o = lane >> 4, nout = __ldg(rec + 2);
    Acc96 r = yr, i = yi;
    if (nout == 1) {  // the halves are parts of one sum
      r.add(shfl16(yr));
      i.add(shfl16(yi));
    }
    if (o >= nout) return;
    const int ec = (int)(o ? h.w : h.z), n = 2 * ex + ec - 58;
    // 2^n in two factors (a coefficient may be as small or large as a double)
    const int n1 = n >> 1, n2 = n - n1;
    double f1 = __hiloint2double((n1 + 1023) << 20, 0);
    const double f2 = __hiloint2double((n2 + 1023) << 20, 0);
    if (ex == kYcBad || ec == kYcNan) f1 = __longlong_as_double(0x7FF8000000000000LL);
    const int at = __ldg(rec + 4 + o) * 32 + (lane & 15);
    cx<double> v = mk<double>(r.value() * f1 * f2, i.value() * f1 * f2);
    if (other) {
      const cx<double> w = reinterpret_cast<const cx<double>*>(other)[at];
      v = mk<double>(v.re + w.re, v.im + w.im);
    }
    reinterpret_cast<cx<double>*>(Yb)[at] = v;
    const int z = __ldg(rec + 4 + kYcOuts + o);
    if (z >= 0) reinterpret_cast<cx<double>*>(Yb)[z * 32 + (lane & 15)] = mk<double>(0.0, 0.0);
  }
};

// The staged block of U, [H][16] complex double, to fixed point in place;
// returns the exponent of the lane's atom (kYcBad if its U is not finite).
__device__ int yf_prepare(unsigned char* su, int H, int* top) {
  // top: [16] in shared memory.  A thread has one atom throughout.
  const int al = threadIdx.x & 15, n = H * 16;
  if (threadIdx.x < 16) top[threadIdx.x] = 0;
  __syncthreads();
  int m = 0;  // the larger of two magnitudes has the larger high word
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int4 v = *reinterpret_cast<const int4*>(su + (size_t)e * 16);
    m = max(m, max(v.y & 0x7FFFFFFF, v.w & 0x7FFFFFFF));
  }
  atomicMax(top + al, m);
  __syncthreads();
  const int E = yc_scale(top[al]);
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    int4* x = reinterpret_cast<int4*>(su + (size_t)e * 16);
    const int4 v = *x;
    int4 w;
    yc_limbs(v.x, v.y, E, w.x, w.y);
    yc_limbs(v.z, v.w, E, w.z, w.w);
    *x = w;
  }
  return E == 0x7FF ? kYcBad : E - 1022;
}

// One warp's share of a CTA's tasks (tl: first chunk and chunks of each),
// taken from a counter in shared memory: a task's outputs have one warp, so
// nothing depends on which.  Chunks come through the warp's ring, the next
// task's behind the last of the one before.
template <class P>
__device__ __forceinline__ void yc_tasks(const WorkArgs& a, const char* __restrict__ ul, unsigned* __restrict__ ring,
                                         const int2* __restrict__ tl, int nt, int* next, int* met, size_t at, int lane,
                                         int ex) {
  P y;
  y.clear();
  int pc = 0, left = 0, live = 0, slot = 0;
  bool more = true;
  auto issue = [&](int s) {
    if (left == 0 && more) {
      int k = 0;
      if (lane == 0) k = atomicAdd(next, 1);
      k = __shfl_sync(kFull, k, 0);
      more = k < nt;
      if (more) {
        pc = tl[k].x;
        left = tl[k].y;
      }
    }
    if (left > 0) {
      const unsigned* g = a.yc_stream + (size_t)pc * kYcChunk + lane * 4;
      unsigned* d = ring + s * kYcChunk + lane * 4;
      cp_async16(d, g);
      cp_async16(d + kYcChunk / 2, g + kYcChunk / 2);
      ++pc;
      --left;
      ++live;
    }
    cp_async_commit();
  };
  static_assert(kYcChunk == 256, "two 16-byte copies a lane");
#pragma unroll
  for (int s = 0; s < P::kSlots - 1; ++s) issue(s);
  while (live > 0) {
    cp_async_wait<P::kSlots - 2>();
    __syncwarp();
    issue(slot == 0 ? P::kSlots - 1 : slot - 1);  // the slot of the chunk before
    const unsigned* ch = ring + slot * kYcChunk;
    const uint4 h = *reinterpret_cast<const uint4*>(ch);
    y.chunk(h.y, ch + 4, ul, lane >> 4);
    if (h.x >> 31) {  // the task's last chunk
      const int* rec = a.yc_task + (size_t)(h.x & 0x7FFFFFFFu) * kYcTask;
      const int half = __ldg(rec + 3);
      char* Y = static_cast<char*>(a.Y) + at;
      if (half == 0) {
        y.store(rec, h, Y, nullptr, lane, ex);
      } else {
        // The sum's other half may be another warp's: each leaves its own (the
        // first in Y, the second in Y2), and the one that comes second adds the
        // two (a sum of two, so their order does not matter).
        char* Y2 = static_cast<char*>(a.Y2) + at;
        y.store(rec, h, (half & 1) ? Y2 : Y, nullptr, lane, ex);
        __threadfence_block();
        __syncwarp();
        int first = 0;
        if (lane == 0) first = atomicAdd(met + (half >> 1) - 1, 1) == 0;
        first = __shfl_sync(kFull, first, 0);
        if (!first) {
          __threadfence_block();
          y.store(rec, h, Y, (half & 1) ? Y : Y2, lane, ex);
        }
      }
      y.clear();
    }
    --live;
    slot = slot == P::kSlots - 1 ? 0 : slot + 1;
  }
  cp_async_wait<0>();  // no copy outlives the warp's tasks
}

// Shared memory: the block's U in class-major order (256 bytes an element),
// the barrier, the rings, the CTA's tasks, and per split sum how many halves
// are done.
__host__ __device__ constexpr size_t yc_ring_offset(int H) { return (size_t)H * 256 + 16; }
__host__ __device__ constexpr size_t yc_smem(int rsize, int H, int ntasks, int warps) {
  return yc_ring_offset(H) + (size_t)warps * yc_slots(rsize) * kYcChunk * 4 + (size_t)ntasks * (sizeof(int2) + sizeof(int));
}

// CTA = one block of atoms x one ysplit-th of the tasks; U of the block staged
// by TMA bulk copies, one an element (256 bytes), which put it in class-major
// order.  QUEUE: a persistent launch, (block, split) items from a device
// counter (flags[5], zeroed with the flags by every evaluation); the staging
// barrier is reused item after item (its phase flips per completed copy), and a
// proxy fence stands between an item's accesses to the block and the copies of
// the next.
template <class P, int LM, bool QUEUE>
__global__ void __launch_bounds__(P::kWarps * 32, LM <= 5 ? 2 : 1) yc_kernel(WorkArgs a, int ysplit) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int item_s, next_s, top_s[16];
  constexpr bool FIXED = P::kAtoms == 16;
  constexpr int kRow = FIXED ? 512 : 256;  // bytes of an element's 32 atoms in global memory
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int H = a.H;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + (size_t)H * 256);
  unsigned* ring = reinterpret_cast<unsigned*>(smem + yc_ring_offset(H)) + warp * P::kSlots * kYcChunk;
  int2* tl = reinterpret_cast<int2*>(smem + yc_ring_offset(H) + (size_t)P::kWarps * P::kSlots * kYcChunk * 4);
  int* met = reinterpret_cast<int*>(tl + a.yc_ntask);
  const long nitems = (long)((a.n + P::kAtoms - 1) / P::kAtoms) * ysplit;
  if (threadIdx.x == 0) mbar_init(bar, 1);
  unsigned phase = 0;
  for (long item = blockIdx.x;;) {
    if (QUEUE) {
      if (threadIdx.x == 0) item_s = atomicAdd(&a.flags[5], 1);
      __syncthreads();  // also: every warp is done with the previous block
      item = item_s;
      if (item >= nitems) break;
    }
    const long blk = item / ysplit;
    const int part = (int)(item - blk * ysplit);
    // the block's first atom in the [ceil(N / 32)][H][32] buffers
    const size_t at = FIXED ? (size_t)(blk >> 1) * H * kRow + (blk & 1) * 256 : (size_t)blk * H * kRow;
    if (threadIdx.x == 0) {
      next_s = 0;
      mbar_expect_tx(bar, (unsigned)(H * 256));
    }
    __syncthreads();
    if (!a.test_skip_stage) {
      const char* ug = static_cast<const char*>(a.U) + at;
      for (int e = threadIdx.x; e < H; e += blockDim.x)
        bulk_g2s(smem + (size_t)__ldg(a.yc_slot + e) * 256, ug + (size_t)e * kRow, 256, bar);
    }
    const int b0 = a.yc_bins[part], nt = a.yc_bins[part + 1] - b0;
    for (int k = threadIdx.x; k < nt; k += blockDim.x) {
      const int* rec = a.yc_task + (size_t)a.yc_bins[ysplit + 1 + b0 + k] * kYcTask;
      tl[k] = make_int2(__ldg(rec), __ldg(rec + 1));
    }
    for (int k = threadIdx.x; k < a.yc_ntask; k += blockDim.x) met[k] = 0;
    const bool ok = __syncthreads_and(mbar_wait_bounded(bar, phase, kWaitNs));
    if (!ok) {
      if (threadIdx.x == 0) atomicMax(&a.flags[3], 1);
      mbar_wait_bounded(bar, phase, kWaitNs / 4);
      return;
    }
    phase ^= 1u;
    int ex = 0;
    if (FIXED) {
      ex = yf_prepare(smem, H, top_s);
      __syncthreads();
    }
    yc_tasks<P>(a, reinterpret_cast<const char*>(smem) + (FIXED ? (lane & 15) * 16 : lane * 8), ring, tl, nt, &next_s,
                met, at, lane, ex);
    if (!QUEUE) break;
    fence_proxy_async();  // this thread's accesses to the staged block (yf_prepare stores to it) come first
    __syncthreads();      // item_s and the staged block are rewritten next
  }
}

// ------------------------------------------- compute_Y's coefficients
// The stream of a new beta, on the device: on the host it took, with the upload
// of 6 and 11 MB, 2.1 ms at 2J14 in FP32 and 7.5 in fixed point (the list of terms
// before it 1.9); all of snap_set_beta takes 27 and 77 us now, at 2J8 22 and 38 (83).
__global__ void __launch_bounds__(256) yc_coef_kernel(const YcCoef* __restrict__ coef, int n, const double* __restrict__ bw,
                                                      float* __restrict__ stream) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (k < n) stream[coef[k].at] = (float)(coef[k].cg * bw[coef[k].trip]);
}

// Fixed point, first pass: the largest sum of sizes of every output (a thread a
// group; of two numbers that are not negative the larger has the larger bits, and
// a NaN the largest).
__global__ void __launch_bounds__(128) yc_top_kernel(const YcCoef* __restrict__ coef, const YcGroup* __restrict__ group, int n,
                                                     const double* __restrict__ bw, unsigned long long* __restrict__ top) {
  const int g = blockIdx.x * 128 + threadIdx.x;
  if (g >= n) return;
  double s = 0.0;
  for (int k = group[g].first; k < group[g + 1].first; ++k) s += fabs(coef[k].cg * bw[coef[k].trip]);
  atomicMax(top + group[g].out, (unsigned long long)__double_as_longlong(s));
}

// the exponent above it, or kYcNan
__device__ __forceinline__ int yc_exponent(unsigned long long top) {
  const double t = __longlong_as_double((long long)top);
  int e = 0;
  if (t > 0.0) frexp(t, &e);
  return isfinite(t) ? e : kYcNan;
}

// Second pass: a thread a group's coefficients, or (past the groups) the
// exponents in a chunk's head.
__global__ void __launch_bounds__(128) yc_fixed_kernel(const YcCoef* __restrict__ coef, const YcGroup* __restrict__ group, int n,
                                                       const double* __restrict__ bw, const int* __restrict__ task, int nchunk,
                                                       const unsigned long long* __restrict__ top, unsigned* __restrict__ stream) {
  const int g = blockIdx.x * 128 + threadIdx.x;
  if (g < n) {
    const int e = yc_exponent(top[group[g].out]);
    for (int k = group[g].first; k < group[g + 1].first; ++k) {
      const YcCoef c = coef[k];
      const long long v = e == kYcNan ? 0 : __double2ll_rn(ldexp(c.cg * bw[c.trip], 60 - e));
      const int hi = (int)((v + (1LL << 29)) >> 30);
      stream[c.at] = (unsigned)hi;
      stream[c.at + 1] = (unsigned)(int)(v - hi * (1LL << 30));
    }
  } else if (g < n + nchunk) {
    unsigned* ch = stream + (size_t)(g - n) * kYcChunk;
    const int k = (int)(ch[0] & 0x7FFFFFFFu), nout = task[k * kYcTask + 2];
    for (int o = 0; o < 2; ++o) ch[2 + o] = (unsigned)yc_exponent(top[k * kYcOuts + (nout == 1 ? 0 : o)]);
  }
}

// ------------------------------------------- compute_Y, one atom per warp
// The alternative layout to the warp of atoms (the paper compares the two,
// Sec. V-B): warp = one atom, its Ulisttot and conj(Ulisttot) staged in shared
// memory as a [2][H] block, lanes over output elements (dealt to the lanes in
// decreasing term count, snake order, so their loads balance); each lane walks
// its outputs' term records, grouped by their first factor:
//   Y += U_e1 * sum_k coef_k U_e2,k
// (a word: the two elements' places in the [2][H] block, the first factor's in
// bits 0-10 and the second's in 11-21, and kYaGroup where a group ends; and the
// coefficient).
constexpr int kYaWarps = 8;
constexpr int kYaSum = 4;

template <typename R>
__global__ void __launch_bounds__(kYaWarps * 32) yi_atom_kernel(WorkArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long i = (long)blockIdx.x * kYaWarps + warp;
  if (i >= a.n) return;  // whole warp
  const int H = a.H;
  cx<R>* ua = reinterpret_cast<cx<R>*>(smem) + (size_t)warp * 2 * H;
  const long base = (i >> 5) * (long)H * 32 + (i & 31);
  const cx<R>* Ug = reinterpret_cast<const cx<R>*>(a.U) + base;
  for (int e = lane; e < H; e += 32) {
    const cx<R> v = Ug[(long)e * 32];
    ua[e] = v;
    ua[H + e] = mk<R>(v.re, -v.im);
  }
  __syncwarp();
  cx<R>* Yg = reinterpret_cast<cx<R>*>(a.Y) + base;
  const YRec<R>* __restrict__ rec = reinterpret_cast<const YRec<R>*>(a.yrec);
  const int m = a.ysched_m;
  for (int k = 0; k < m; ++k) {
    const int o = a.ysched[lane * m + k];
    if (o < 0) break;
    YAcc<R> y;
    y.re = y.im = y.ar = y.ai = R(0);
    // FP32: what every 4 kYaSum = 16 records have added is put into a compensated sum
    // (a long FP32 sum is further off), on all lanes at the same record, and the
    // records are taken four at a time, their loads together.  Bound by the loads'
    // latency; compute_Y, 54 atoms, 2J8 / 2J14: 98 / 2430 us in FP32 (one long sum,
    // record by record: 90 / 2530; compensated at each lane's own groups' ends: 186 /
    // 4880), 455 / 12100 in FP64.
    R sr = R(0), si = R(0), er = R(0), ei = R(0);
    auto add = [](R& s, R& e, R x) {
      const R v = x - e, t = s + v;
      e = (t - s) - v;
      s = t;
    };
    auto term = [&](unsigned w, R c, cx<R> u2) {
      y.ar += c * u2.re;
      y.ai += c * u2.im;
      if (w & kYaGroup) {
        const cx<R> u1 = ua[w & 2047u];
        y.re = fmr(-u1.im, y.ai, fmr(u1.re, y.ar, y.re));
        y.im = fmr(u1.im, y.ar, fmr(u1.re, y.ai, y.im));
        y.ar = R(0);
        y.ai = R(0);
      }
    };
    int q = a.yfirst[o], n = 0;
    const int q1 = a.yfirst[o + 1];
    for (; q + 4 <= q1; q += 4) {
      unsigned w[4];
      R c[4];
      cx<R> u2[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        w[j] = rec[q + j].w;
        c[j] = rec[q + j].c;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) u2[j] = ua[(w[j] >> 11) & 2047u];
#pragma unroll
      for (int j = 0; j < 4; ++j) term(w[j], c[j], u2[j]);
      if (sizeof(R) == 4 && ++n == kYaSum) {
        n = 0;
        add(sr, er, y.re);
        add(si, ei, y.im);
        y.re = y.im = R(0);
      }
    }
    for (; q < q1; ++q) term(rec[q].w, rec[q].c, ua[(rec[q].w >> 11) & 2047u]);
    if (sizeof(R) == 4) {
      add(sr, er, y.re);
      add(si, ei, y.im);
    } else {
      sr = y.re;
      si = y.im;
    }
    Yg[(long)o * 32] = mk<R>(sr, si);
  }
}

// ------------------------------------------------------- bispectrum B_l
// Descriptor output (Sec. II-A, Eq. z): B_l = Re Z^t_{t1t2} : conj(U_t) for
// every canonical component l, 32 atoms a CTA (lanes = atoms; the block's U
// staged in shared memory by a TMA bulk copy, as in compute_Y), and, with
// DERIV, its directional derivative along the tangent dU of Ulisttot
// (Eqs. z and dbidrk): B_l is trilinear in (U_t1, U_t2, conj U_t), so
//   dB_l = Re [ (Z(dU_t1, U_t2) + Z(U_t1, dU_t2)) : conj(U_t) + Z : conj(dU_t) ]
// (dU has the inversion symmetry of U, so the records' conjugation flags hold
// for it too).
// The term list is cut into chunks of whole output groups (never across a
// component).  CTA (block, part) takes the components of its part; its
// warps take the part's chunks in turn, each leaving one partial sum per atom
// (in shared memory, or in a global scratch where the part has too many
// chunks), and the partials of a component are added in chunk order: a fixed
// order, whatever the launch shape, and no warp waits on the largest
// component.
//
// Records (snap_tables.h, bwords): the factors' byte offsets sit in the word
// already scaled to the plane's element stride (one mask each).  Each output
// group is cut into pieces of at most kBGroupMax terms, and a chunk's pieces
// are stored by length, so a chunk is runs of equal-length pieces walked by
// branch-free bodies (records, factors and output elements loaded ahead of
// the arithmetic); a piece's first word holds its output element.  The
// contraction is linear in Z, so each piece is contracted on its own.  CP:
// the staged block is [2][H][32] with the conjugates in its second half (no
// sign flips); with DERIV the tangent's planes follow, [U | conj U | dU |
// conj dU].
template <typename R, bool CP>
__device__ __forceinline__ unsigned b_off1(unsigned w) {
  const unsigned o = CP ? ((w >> 11) & 0x7FF00u) : ((w >> 10) & 0x3FF00u);
  return sizeof(R) == 4 ? o : o << 1;
}
template <typename R, bool CP>
__device__ __forceinline__ unsigned b_off2(unsigned w) {
  const unsigned o = CP ? (w & 0x7FF00u) : (w & 0x3FF00u);
  return sizeof(R) == 4 ? o : o << 1;
}
// byte offset of a piece's output element, from the piece's first word
template <typename R, bool CP>
__device__ __forceinline__ unsigned b_out(unsigned w) {
  const unsigned o = (w & 0xFFu) | (((w >> (CP ? 30 : 28)) & 3u) << 8);
  return o * (unsigned)(32 * sizeof(cx<R>));
}

// one record: from the CTA's staged copy (RS) or through the read-only path
template <typename R, bool RS>
__device__ __forceinline__ void b_load(const YRec<R>* __restrict__ rec, int q, unsigned& w, R& c) {
  if constexpr (RS) {
    if constexpr (sizeof(R) == 4) {
      const uint2 r = *reinterpret_cast<const uint2*>(rec + q);
      w = r.x;
      c = __uint_as_float(r.y);
    } else {
      const uint4 r = *reinterpret_cast<const uint4*>(rec + q);
      w = r.x;
      c = (R)__hiloint2double((int)r.w, (int)r.z);
    }
  } else if constexpr (sizeof(R) == 4) {
    const uint2 r = __ldg(reinterpret_cast<const uint2*>(rec + q));
    w = r.x;
    c = __uint_as_float(r.y);
  } else {
    const uint4 r = __ldg(reinterpret_cast<const uint4*>(rec + q));
    w = r.x;
    c = (R)__hiloint2double((int)r.w, (int)r.z);
  }
}

// G pieces of K terms from record q: per piece Z = sum c u1 u2 (and dZ),
// then acc += Re(Z conj U_o) (DERIV: Re(dZ conj U_o + Z conj dU_o)).
template <typename R, bool CP, bool DERIV, bool RS, int K, int G>
__device__ __forceinline__ void b_pieces(const YRec<R>* __restrict__ rec, int q, const char* __restrict__ ul,
                                         const char* __restrict__ dl, R& acc) {
  constexpr int N = G * K;
  unsigned w[N];
  R c[N];
#pragma unroll
  for (int j = 0; j < N; ++j) b_load<R, RS>(rec, q + j, w[j], c[j]);
  cx<R> u1[N], u2[N], d1[DERIV ? N : 1], d2[DERIV ? N : 1], uo[G], duo[DERIV ? G : 1];
#pragma unroll
  for (int j = 0; j < N; ++j) {
    u1[j] = *reinterpret_cast<const cx<R>*>(ul + b_off1<R, CP>(w[j]));
    u2[j] = *reinterpret_cast<const cx<R>*>(ul + b_off2<R, CP>(w[j]));
    if constexpr (DERIV) {
      d1[j] = *reinterpret_cast<const cx<R>*>(dl + b_off1<R, CP>(w[j]));
      d2[j] = *reinterpret_cast<const cx<R>*>(dl + b_off2<R, CP>(w[j]));
    }
  }
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const unsigned ob = b_out<R, CP>(w[g * K]);
    uo[g] = *reinterpret_cast<const cx<R>*>(ul + ob);
    if constexpr (DERIV) duo[g] = *reinterpret_cast<const cx<R>*>(dl + ob);
  }
#pragma unroll
  for (int g = 0; g < G; ++g) {
    R zr, zi, dzr = R(0), dzi = R(0);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int j = g * K + k;
      const unsigned m1 = (w[j] << 1) & 0x80000000u, m2 = w[j] & 0x80000000u;
      const R b1 = CP ? u1[j].im : flip_sign(u1[j].im, m1), b2 = CP ? u2[j].im : flip_sign(u2[j].im, m2);
      // c u1 u2 = (p + i q)(u2.re + i b2), p + i q = c u1
      const R p = c[j] * u1[j].re, qq = c[j] * b1;
      if (k == 0) {
        zr = p * u2[j].re;
        zi = p * b2;
      } else {
        zr = fmr(p, u2[j].re, zr);
        zi = fmr(p, b2, zi);
      }
      zr = fmr(-qq, b2, zr);
      zi = fmr(qq, u2[j].re, zi);
      if constexpr (DERIV) {
        // d(c u1 u2) = c du1 u2 + c u1 du2
        const R db1 = CP ? d1[j].im : flip_sign(d1[j].im, m1), db2 = CP ? d2[j].im : flip_sign(d2[j].im, m2);
        const R dp = c[j] * d1[j].re, dq = c[j] * db1;
        dzr = fmr(dp, u2[j].re, dzr);
        dzr = fmr(-dq, b2, dzr);
        dzr = fmr(p, d2[j].re, dzr);
        dzr = fmr(-qq, db2, dzr);
        dzi = fmr(dp, b2, dzi);
        dzi = fmr(dq, u2[j].re, dzi);
        dzi = fmr(p, db2, dzi);
        dzi = fmr(qq, d2[j].re, dzi);
      }
    }
    if constexpr (DERIV) {
      acc = fmr(uo[g].re, dzr, acc);
      acc = fmr(uo[g].im, dzi, acc);
      acc = fmr(duo[g].re, zr, acc);
      acc = fmr(duo[g].im, zi, acc);
    } else {
      acc = fmr(uo[g].re, zr, acc);
      acc = fmr(uo[g].im, zi, acc);
    }
  }
}

// All ng pieces of K terms from record q (advanced past them): about kStep
// records a body.
template <typename R, bool CP, bool DERIV, bool RS, int K>
__device__ __forceinline__ void b_run(const YRec<R>* __restrict__ rec, int& q, int ng, const char* __restrict__ ul,
                                      const char* __restrict__ dl, R& acc) {
  constexpr int kStep = DERIV ? 4 : 8;
  constexpr int G = K >= kStep ? 1 : kStep / K;
  for (; ng >= G; ng -= G, q += G * K) b_pieces<R, CP, DERIV, RS, K, G>(rec, q, ul, dl, acc);
  for (; ng > 0; --ng, q += K) b_pieces<R, CP, DERIV, RS, K, 1>(rec, q, ul, dl, acc);
}

// gpart: the partial sums' scratch in global memory ([CTA][maxchunks][32]),
// or null for shared memory.  RS: the run's records staged beside the planes
// (rec_bytes of shared memory) by the same bulk copy.
// DS (DERIV): the tangent's block is staged too; without it (two blocks do not
// fit, 2J = 14) U alone is staged and dU is read through L1.
template <typename R, bool STAGED, bool CP, bool DERIV, bool RS, bool DS>
__global__ void __launch_bounds__(kBiThreads, kBiCtasPerSm)
    bi_kernel(WorkArgs a, const cx<R>* __restrict__ dUg, double* __restrict__ out, R* __restrict__ gpart,
              unsigned rec_bytes) {
  extern __shared__ __align__(128) unsigned char smem[];
  static_assert(STAGED || (!CP && !RS), "the conjugate plane and the records are staged");
  static_assert(!DS || (STAGED && DERIV), "the tangent is staged with U");
  static_assert(!(CP && DERIV && !DS), "the conjugate plane of dU needs dU staged");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const long blk = blockIdx.x;
  const int H = a.H;
  const size_t plane = (size_t)H * 32 * sizeof(cx<R>);
  constexpr int NP = (CP ? 2 : 1) * (DS ? 2 : 1);
  const cx<R>* ug = reinterpret_cast<const cx<R>*>(a.U) + blk * H * 32;
  const cx<R>* dg = DERIV ? dUg + blk * H * 32 : nullptr;
  const char* ul = reinterpret_cast<const char*>(ug + lane);
  const char* dl = DERIV ? reinterpret_cast<const char*>(dg + lane) : nullptr;
  const size_t roff = STAGED ? NP * plane + 16 : 0;  // records, then partials
  R* part = gpart ? gpart + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * a.bmaxchunks * 32
                  : reinterpret_cast<R*>(smem + roff + (RS ? rec_bytes : 0u));  // [maxchunks][32]
  const int l0 = a.bpart[blockIdx.y], l1 = a.bpart[blockIdx.y + 1];
  const int c0 = a.bcomp_chunk[l0], c1 = a.bcomp_chunk[l1];
  const YRec<R>* __restrict__ grec = reinterpret_cast<const YRec<R>*>(CP ? a.brec_cp : a.brec);
  // records [qb, q1) of the run; FP32 records start on a 16-byte boundary
  const int qb = RS ? (sizeof(R) == 4 ? a.bchunk_term[c0] & ~1 : a.bchunk_term[c0]) : 0;
  const unsigned rbytes =
      RS ? (unsigned)(((a.bchunk_term[c1] - qb) * sizeof(YRec<R>) + 15) / 16 * 16) : 0u;
  if (STAGED) {
    cx<R>* su = reinterpret_cast<cx<R>*>(smem);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + NP * plane);
    if (!stage_bulk(su, ug, (unsigned)plane, bar, a.flags, a.test_skip_stage != 0, [] {},
                    DS ? reinterpret_cast<const void*>(dg) : nullptr, (unsigned)((CP ? 2 : 1) * plane),
                    RS ? reinterpret_cast<const void*>(grec + qb) : nullptr, rbytes, (unsigned)roff))
      return;
    if (CP) {
      const int he = H * 32;
      for (int e = threadIdx.x; e < he; e += blockDim.x) {
        const cx<R> v = su[e];
        su[he + e] = mk<R>(v.re, -v.im);
        if (DS) {
          const cx<R> d = su[2 * he + e];
          su[3 * he + e] = mk<R>(d.re, -d.im);
        }
      }
      __syncthreads();
    }
    ul = reinterpret_cast<const char*>(su + lane);
    if (DS) dl = ul + (CP ? 2 : 1) * plane;
  }
  const YRec<R>* __restrict__ rec = RS ? reinterpret_cast<const YRec<R>*>(smem + roff) : grec;
  static_assert(kBGroupMax == 8, "one 16-byte run header per chunk");
  const uint4* __restrict__ runs = reinterpret_cast<const uint4*>(a.bchunk_runs);
  for (int ch = c0 + warp; ch < c1; ch += nw) {
    const uint4 h = __ldg(runs + ch);
    int q = a.bchunk_term[ch] - qb;
    R acc = R(0);
    b_run<R, CP, DERIV, RS, 1>(rec, q, (int)(h.x & 0xffffu), ul, dl, acc);
    b_run<R, CP, DERIV, RS, 2>(rec, q, (int)(h.x >> 16), ul, dl, acc);
    b_run<R, CP, DERIV, RS, 3>(rec, q, (int)(h.y & 0xffffu), ul, dl, acc);
    b_run<R, CP, DERIV, RS, 4>(rec, q, (int)(h.y >> 16), ul, dl, acc);
    b_run<R, CP, DERIV, RS, 5>(rec, q, (int)(h.z & 0xffffu), ul, dl, acc);
    b_run<R, CP, DERIV, RS, 6>(rec, q, (int)(h.z >> 16), ul, dl, acc);
    b_run<R, CP, DERIV, RS, 7>(rec, q, (int)(h.w & 0xffffu), ul, dl, acc);
    b_run<R, CP, DERIV, RS, 8>(rec, q, (int)(h.w >> 16), ul, dl, acc);
    part[(ch - c0) * 32 + lane] = acc;
  }
  __syncthreads();
  const long i = blk * 32 + lane;
  for (int l = l0 + warp; l < l1; l += nw) {
    R v = R(0);
    for (int ch = a.bcomp_chunk[l]; ch < a.bcomp_chunk[l + 1]; ++ch) v += part[(ch - c0) * 32 + lane];
    if (i < a.n) out[i * a.ncoeff + l] = (double)v;
  }
}

// ------------------------------------------- weighted force (autograd)
// grad_k = sum_i w_i dE_i/dr_k = -( w_k sum_s dE_k/dr_ks - sum_s w_{k_s} dE_{k_s}/dr_{k_s,k} ),
// gathered through the reverse-slot map like the forces (w = 1 gives -F).
__global__ void __launch_bounds__(256) force_weighted_kernel(WorkArgs a, const double* __restrict__ wt,
                                                             double* __restrict__ grad) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long k = (long)blockIdx.x * 8 + warp;
  if (k >= a.n) return;
  const double wk = wt[k];
  double f[3] = {0, 0, 0};
  const int cnt = a.cnt[k];
  for (int s = lane; s < cnt; s += 32) {
    const long q = k * a.K + s;
    const int j = a.nbr[q];
    const int r = a.rev[q];
    const double* d = a.dedr + q * 3;
    for (int c = 0; c < 3; ++c) f[c] += wk * d[c];
    if (r >= 0) {
      const double wj = wt[j];
      const double* dj = a.dedr + ((long)j * a.K + r) * 3;
      for (int c = 0; c < 3; ++c) f[c] -= wj * dj[c];
    }
  }
  for (int c = 0; c < 3; ++c) f[c] = warp_sum(f[c]);
  if (lane == 0)
    for (int c = 0; c < 3; ++c) grad[3 * k + c] = -f[c];
}

// --------------------------------------------- energy, forces and virial
// CTA = kFAtoms consecutive atoms, kFThreads threads (a warp per two atoms).
// FP64 runs at 1/64 of the FP32 rate on this part and a warp FP64
// instruction costs the same whatever its active lanes, so the FP64 sums are
// short trees on full warps instead of long chains on a few threads:
//  * energy: E_i - beta_0 is a cubic form in U, so by Euler's relation
//    E_i = beta_0 + (1/3) Re sum_t Y_t : conj(U_t) (full matrices; half layout
//    with half_weight).  kFSlices slices per atom take every kFSlices-th
//    element in the working precision (lanes over atoms: the U and Y reads
//    are coalesced); the slices are added in FP64 by a fixed tree;
//  * forces: lane l of an atom's kFLanes takes slots l, l + kFLanes, ...: it
//    forms g = dE_i/dr_ik - dE_k/dr_ki (the second term through the
//    reverse-slot map, no atomics), adds its g in slot order and accumulates
//    the virial products -dE_i/dr_ik,a r_ik,b; the lane sums are then added
//    by a fixed butterfly;
//  * virial: W_ab is reduced per CTA by the same kind of tree and the last
//    CTA to finish adds the CTA partials in a fixed order (batch mode: per
//    atom, reduced per configuration afterwards).
// Every sum has an order fixed by the slot and element indices alone, so the
// per-atom results do not depend on launch shape or batching.
constexpr int kFAtoms = 8;
constexpr int kFThreads = 128;
constexpr int kFWarps = kFThreads / 32;
constexpr int kFSlices = kFThreads / kFAtoms;  // energy slices per atom
constexpr int kFLanes = 16;                    // lanes per atom in the force sums
static_assert(kFWarps * 32 / kFLanes == kFAtoms, "a warp per two atoms");

// Sum of x[0..N) over each aligned group of G lanes (N <= G, both powers of
// two).  A level with mask m first halves the components a lane carries (the
// lane with bit m clear keeps the lower half and receives its partner's
// lower half), so N components take N - 1 + log2(G / N) additions instead of
// N log2(G).  Returns the total of component (lane mod G) / (G / N).
template <int N, int G>
__device__ __forceinline__ double tree_sum(double (&x)[N], int lane) {
  static_assert(N >= 1 && N <= G && G <= 32 && (N & (N - 1)) == 0 && (G & (G - 1)) == 0, "");
  int n = N;
#pragma unroll
  for (int m = G / 2; m >= 1; m >>= 1) {
    if (n > 1) {
      const bool up = lane & m;
      const int h = n / 2;
#pragma unroll
      for (int j = 0; j < N / 2; ++j) {
        if (j < h) {
          const double send = up ? x[j] : x[j + h];
          const double keep = up ? x[j + h] : x[j];
          x[j] = keep + __shfl_xor_sync(kFull, send, m);
        }
      }
      n = h;
    } else {
      x[0] += __shfl_xor_sync(kFull, x[0], m);
    }
  }
  return x[0];
}

inline size_t force_smem(int, bool) { return 0; }

template <typename R>
__global__ void __launch_bounds__(kFThreads) force_kernel(WorkArgs a) {
  __shared__ double ew[kFWarps][kFAtoms];  // energy: per warp, per atom
  __shared__ double wv[kFWarps][8];        // virial: per warp, per component
  __shared__ bool last;
  const int K = a.K, H = a.H;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const long i0 = (long)blockIdx.x * kFAtoms;
  const int na = (int)min((long)kFAtoms, a.n - i0);
  // forces: lanes 16h .. 16h + 15 of warp w take atom 2w + h.  The first
  // pass's slot loads go out before the count and the energy loads (every
  // slot below K is in bounds; those at or past the count are discarded).
  const int l = lane % kFLanes;
  const int ai = 2 * w + lane / kFLanes;
  const bool have = ai < na;
  const long i = i0 + ai;
  bool ok[2];
  int rv[2], kn[2], ky[2];
  double d[2][3], r[2][3], dk[2][3];
  auto load_slots = [&](int s0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int s = s0 + u * kFLanes + l;
      rv[u] = -1;
      kn[u] = 0;
      ky[u] = -1;
#pragma unroll
      for (int c = 0; c < 3; ++c) d[u][c] = r[u][c] = dk[u][c] = 0.0;
      if (have && s < K) {
        const long q = i * K + s;
        kn[u] = a.nbr[q];
        ky[u] = a.key[q];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          d[u][c] = a.dedr[q * 3 + c];
          r[u][c] = a.rij[q * 3 + c];
        }
      }
    }
  };
  const int cnt_raw = have ? a.cnt[i] : 0;
  load_slots(0);
  // energy partials: lane = atom (8) x slice (4) of the warp's 4 slices
  if (a.energy) {
    const int ae = lane % kFAtoms, sl = (kFSlices / kFWarps) * w + lane / kFAtoms;
    R e = R(0);
    if (ae < na) {
      const long ie = i0 + ae;
      const long blk = ie >> 5;
      const int li = (int)(ie & 31);
      const cx<R>* Ug = reinterpret_cast<const cx<R>*>(a.U) + blk * H * 32 + li;
      const cx<R>* Yg = reinterpret_cast<const cx<R>*>(a.Y) + blk * H * 32 + li;
#pragma unroll 8
      for (int el = sl; el < H; el += kFSlices) {
        const int p = __ldg(a.half_tmm + el);
        const R w8 = (R)half_weight(tmm_t(p), tmm_ma(p), tmm_mb(p));
        const cx<R> u = Ug[el * 32], y = Yg[el * 32];
        e += w8 * (y.re * u.re + y.im * u.im);
      }
    }
    double de = (double)e;
    de += __shfl_xor_sync(kFull, de, 8);
    de += __shfl_xor_sync(kFull, de, 16);
    if (lane < kFAtoms) ew[w][lane] = de;
  }
  const int cnt = min(cnt_raw, K);
  double f[4] = {0.0, 0.0, 0.0, 0.0};
  double v[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int s0 = 0; s0 < cnt; s0 += 2 * kFLanes) {
    // two slots per pass: the reverse slot (a pass over the neighbour's row
    // of pair keys, kept for the weighted gather) after the first-level
    // loads, then its dE/dr
    if (s0 > 0) load_slots(s0);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      ok[u] = s0 + u * kFLanes + l < cnt;
      if (ok[u]) {
        const long q = i * K + s0 + u * kFLanes + l;
        rv[u] = geo::find_rev_key(a, (int)i, q, kn[u], ky[u]);
        a.rev_out[q] = rv[u];
        if (rv[u] < 0) atomicMax(&a.flags[1], 1);
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (ok[u] && rv[u] >= 0)
#pragma unroll
        for (int c = 0; c < 3; ++c) dk[u][c] = a.dedr[((long)kn[u] * K + rv[u]) * 3 + c];
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (!ok[u]) continue;
#pragma unroll
      for (int c = 0; c < 3; ++c) f[c] += d[u][c] - dk[u][c];
      v[0] = fma(-d[u][0], r[u][0], v[0]);
      v[1] = fma(-d[u][1], r[u][1], v[1]);
      v[2] = fma(-d[u][2], r[u][2], v[2]);
      v[3] = fma(-d[u][0], r[u][1], v[3]);
      v[4] = fma(-d[u][0], r[u][2], v[4]);
      v[5] = fma(-d[u][1], r[u][2], v[5]);
    }
  }
  const double fsum = tree_sum<4, kFLanes>(f, lane);  // component l / 4
  if (have && l % 4 == 0 && l / 4 < 3) a.forces[3 * i + l / 4] = fsum;
  if (a.vatom) {  // batch mode: per-atom virial, reduced per configuration later
    const double vs = tree_sum<8, kFLanes>(v, lane);  // component l / 2
    if (have && l % 2 == 0 && l / 2 < 6) a.vatom[6 * i + l / 2] = vs;
  } else if (a.virial) {
    const double vs = tree_sum<8, 32>(v, lane);  // component lane / 4
    if (lane % 4 == 0) wv[w][lane / 4] = vs;
  }
  __syncthreads();
  if (a.energy && tid < na) {
    const double e = (ew[0][tid] + ew[1][tid]) + (ew[2][tid] + ew[3][tid]);
    a.energy[i0 + tid] = a.beta0 + e * (1.0 / 3.0);
  }
  const bool vir = !a.vatom && a.virial;
  if (!vir && !a.hflags) return;
  const int cta = blockIdx.x, ncta = gridDim.x;
  if (vir && tid < 6) a.vpart[6 * cta + tid] = (wv[0][tid] + wv[1][tid]) + (wv[2][tid] + wv[3][tid]);
  __syncthreads();
  // the fence after the barrier makes every write and flag update of this
  // CTA (the reverse-slot check's included) visible before its count
  if (tid == 0) {
    __threadfence();
    last = (atomicAdd(&a.flags[4], 1) == ncta - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (a.hflags) {
    // the evaluation's end: the status words to the host-mapped copy and all
    // flags zeroed for the next evaluation (no other CTA touches them now)
    __syncthreads();  // every thread of this CTA is past its own flag reads
    if (tid < 8) {
      const int v = __ldcg(a.flags + tid);
      if (tid < 4) a.hflags[tid] = v;
      a.flags[tid] = 0;
    }
  }
  if (!vir) return;
  // last CTA: thread t adds the CTA partials t, t + kFThreads, ... in order
  // (loads issued four at a time), then the same trees: a fixed order, so
  // the virial is deterministic
  double x[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int b0 = tid; b0 < ncta; b0 += 4 * kFThreads) {
    double y[4][6];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int b = b0 + k * kFThreads;
#pragma unroll
      for (int c = 0; c < 6; ++c) y[k][c] = b < ncta ? __ldcg(a.vpart + 6 * b + c) : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int c = 0; c < 6; ++c) x[c] += y[k][c];
  }
  const double xs = tree_sum<8, 32>(x, lane);
  if (lane % 4 == 0) wv[w][lane / 4] = xs;
  __syncthreads();
  if (tid < 6) a.virial[tid] = (wv[0][tid] + wv[1][tid]) + (wv[2][tid] + wv[3][tid]);
}

}  // namespace


// Split of each block's outputs into ysplit CTAs.  CTAs of one launch take
// about equal time, so the launch lasts ceil(CTAs / per) CTA lifetimes; the
// split minimises
//   ceil(nblk ysplit / per) (1 / ysplit + c),
// c = the fixed cost of a CTA (staging U) relative to a whole block's terms.
static int yi_split(int nblk, long per, double c) {
  double best = 1e300;
  int split = 1;
  for (int ys = 1; ys <= 64; ++ys) {
    const long w = ((long)nblk * ys + per - 1) / per;
    const double t = (double)w * (1.0 / ys + c);
    if (t < best - 1e-12) {
      best = t;
      split = ys;
    }
  }
  return split;
}

YiGeometry yi_geometry(int rsize, int H, int n, int nsm, int waves, int ntasks) {
  YiGeometry g;
  g.nblk = rsize == 4 ? (n + 31) / 32 : (n + 15) / 16;
  // The CTAs an SM holds share its pipes, so the launch lasts as long as the
  // SM with the most CTAs.  c = 0.02 / waves (the tunable: more waves, finer
  // splits).
  const int warps = yc_warps(rsize, H);
  g.threads = warps * 32;
  g.smem = yc_smem(rsize, H, ntasks, warps);
  g.split = yi_split(g.nblk, nsm, 0.02 / std::max(1, waves));
  return g;
}

cudaError_t launch_yc_coefs(bool fixed, const YcCoef* coef, int ncoef, const YcGroup* group, int ngroup, const double* bw,
                            const int* task, int ntask, int nchunk, unsigned long long* top, unsigned* stream,
                            cudaStream_t s) {
  if (!fixed)
    return launch_k(yc_coef_kernel, dim3((ncoef + 255) / 256), dim3(256), 0, s, coef, ncoef, bw,
                    reinterpret_cast<float*>(stream));
  cudaError_t e = cudaMemsetAsync(top, 0, sizeof(*top) * ntask * kYcOuts, s);
  if (e == cudaSuccess) e = launch_k(yc_top_kernel, dim3((ngroup + 127) / 128), dim3(128), 0, s, coef, group, ngroup, bw, top);
  if (e != cudaSuccess) return e;
  return launch_k(yc_fixed_kernel, dim3((ngroup + nchunk + 127) / 128), dim3(128), 0, s, coef, group, ngroup, bw, task, nchunk,
                  top, stream);
}

template <typename K>
cudaError_t launch_yq(K kq, const YiGeometry& g, const WorkArgs& a, cudaStream_t s) {
  // persistent: as many CTAs as stay resident, (block, split) items from the queue
  cudaError_t e = allow_smem(kq, g.smem);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kq, g.threads, g.smem);
  if (e != cudaSuccess) return e;
  const long nitems = (long)g.nblk * g.split;
  const long grid = std::min<long>(nitems, (long)a.nsm * std::max(1, occ));
  return launch_k(kq, dim3((unsigned)grid), dim3(g.threads), g.smem, s, a, g.split);
}

template <class P, int LM>
cudaError_t launch_yc(const YiGeometry& g, const WorkArgs& a, cudaStream_t s) {
  if (a.persist & 1) return launch_yq(yc_kernel<P, LM, true>, g, a, s);
  cudaError_t e = allow_smem(yc_kernel<P, LM, false>, g.smem);
  if (e != cudaSuccess) return e;
  return launch_k(yc_kernel<P, LM, false>, dim3((unsigned)(g.nblk * g.split)), dim3(g.threads), g.smem, s, a,
                  g.split);
}

template <typename R>
cudaError_t launch_yi(const WorkArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  if (a.yi_layout == 1) {
    const size_t sm = sizeof(cx<R>) * 2 * (size_t)a.H * kYaWarps;
    cudaError_t e = allow_smem(yi_atom_kernel<R>, sm);
    if (e != cudaSuccess) return e;
    return launch_k(yi_atom_kernel<R>, dim3((unsigned)((a.n + kYaWarps - 1) / kYaWarps)),
                    dim3(kYaWarps * 32), sm, s, a);
  }
  const YiGeometry g = yi_geometry(sizeof(R), a.H, a.n, a.nsm, a.yi_waves, a.yc_ntask);
  if (g.split != a.yc_split) return cudaErrorInvalidValue;
  constexpr int RS = sizeof(R), W8 = yc_warps(RS, half_size(8)), W9 = yc_warps(RS, half_size(9)),
                W14 = yc_warps(RS, half_size(14));
  if constexpr (RS == 4)
    return a.twojmax <= 8   ? launch_yc<YcSingle<5, W8>, 5>(g, a, s)
           : a.twojmax <= 9 ? launch_yc<YcSingle<5, W9>, 5>(g, a, s)
                            : launch_yc<YcSingle<8, W14>, 8>(g, a, s);
  else
    return a.twojmax <= 9 ? launch_yc<YcFixed<5, W9>, 5>(g, a, s) : launch_yc<YcFixed<8, W14>, 8>(g, a, s);
}

template <typename R>
cudaError_t launch_force(const WorkArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  const size_t sm = force_smem(a.K, a.vatom != nullptr);
  cudaError_t e = allow_smem(force_kernel<R>, sm);
  if (e != cudaSuccess) return e;
  return launch_k(force_kernel<R>, dim3((unsigned)((a.n + kFAtoms - 1) / kFAtoms)), dim3(kFThreads), sm, s, a);
}

// Bispectrum (dU == nullptr) or its derivative along dU into out [N][N_B]:
// grid (32-atom blocks, component runs a.nbparts), 8 warps a CTA.
BiPlan bi_plan(int rsize, int H, bool deriv, int maxchunks, int maxterms, int layout, bool have_cp) {
  BiPlan p;
  const size_t plane = (size_t)H * 32 * 2 * rsize;
  const size_t np = deriv ? 2 : 1;
  const size_t part = (size_t)maxchunks * 32 * rsize;
  p.staged = plane + 16 <= kBiSmemMax;              // U's block
  p.ds = deriv && np * plane + 16 <= kBiSmemMax;    // and the tangent's beside it
  const size_t ns = p.ds ? 2 : 1;                    // staged blocks
  // the conjugate plane when asked for, or (planned) when two CTAs still fit an SM
  p.cp = p.staged && (!deriv || p.ds) && have_cp && layout != 1 && 2 * ns * plane + 16 <= kBiSmemMax &&
         (layout == 2 || 2 * ns * plane + 16 + part <= kBiSmemPair);
  const size_t planes = p.staged ? (p.cp ? 2 : 1) * ns * plane + 16 : 0;
  p.gpart = planes + part > kBiSmemMax;
  const size_t base = planes + (p.gpart ? 0 : part);
  // a run's records (one more for the 16-byte-aligned start of FP32 records)
  // when they fit without losing the second CTA of an SM
  const size_t rec = (((size_t)maxterms + 1) * (rsize == 4 ? 8 : 16) + 15) / 16 * 16;
  p.rs = p.staged && base + rec <= (base <= kBiSmemPair ? kBiSmemPair : kBiSmemMax);
  p.rec_bytes = p.rs ? rec : 0;
  p.smem = base + p.rec_bytes;
  return p;
}

bool bi_plane_fits(int rsize, int H) { return 2 * (size_t)H * 32 * 2 * rsize + 16 <= kBiSmemMax; }

template <typename R, bool DERIV>
cudaError_t launch_bi_t(const WorkArgs& a, const void* dU, double* out, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  const long nblk = (a.n + 31) / 32;
  const BiPlan p = bi_plan((int)sizeof(R), a.H, DERIV, a.bmaxchunks, a.bmaxterms, a.bi_layout, a.brec_cp != nullptr);
  R* gpart = p.gpart ? reinterpret_cast<R*>(a.bscratch) : nullptr;
  if (p.gpart && !gpart) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)nblk, (unsigned)a.nbparts);
  const cx<R>* d = reinterpret_cast<const cx<R>*>(dU);
  const unsigned rb = (unsigned)p.rec_bytes;
  auto go = [&](auto kern) -> cudaError_t {
    cudaError_t e = allow_smem(kern, p.smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, grid, dim3(kBiThreads), p.smem, s, a, d, out, gpart, rb);
  };
  if (!p.staged) return go(bi_kernel<R, false, false, DERIV, false, false>);
  if (DERIV && !p.ds)  // U staged, dU through L1
    return p.rs ? go(bi_kernel<R, true, false, DERIV, true, false>) : go(bi_kernel<R, true, false, DERIV, false, false>);
  if (p.cp)
    return p.rs ? go(bi_kernel<R, true, true, DERIV, true, DERIV>) : go(bi_kernel<R, true, true, DERIV, false, DERIV>);
  return p.rs ? go(bi_kernel<R, true, false, DERIV, true, DERIV>) : go(bi_kernel<R, true, false, DERIV, false, DERIV>);
}

template <typename R>
cudaError_t launch_bi(const WorkArgs& a, cudaStream_t s) {
  return launch_bi_t<R, false>(a, nullptr, a.B, s);
}
template cudaError_t launch_bi<float>(const WorkArgs&, cudaStream_t);
template cudaError_t launch_bi<double>(const WorkArgs&, cudaStream_t);

template <typename R>
cudaError_t launch_dbi(const WorkArgs& a, const void* dU, double* dB, cudaStream_t s) {
  return launch_bi_t<R, true>(a, dU, dB, s);
}
template cudaError_t launch_dbi<float>(const WorkArgs&, const void*, double*, cudaStream_t);
template cudaError_t launch_dbi<double>(const WorkArgs&, const void*, double*, cudaStream_t);

cudaError_t launch_force_weighted(const WorkArgs& a, const double* w, double* grad, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  return launch_k(force_weighted_kernel, dim3((a.n + 7) / 8), dim3(256), 0, s, a, w, grad);
}

// End of an evaluation: the status words (flags 0-3) go to the host-mapped
// copy, and every flag, counters included, is zeroed for the next
// evaluation (the kernels before it in the stream have completed).
__global__ void flags_out_kernel(int* __restrict__ flags, int* __restrict__ hflags) {
  const int t = threadIdx.x;
  if (t < 8) {
    const int v = flags[t];
    if (t < 4) hflags[t] = v;
    flags[t] = 0;
  }
}

cudaError_t launch_flags_out(int* flags, int* hflags, cudaStream_t s) {
  return launch_k(flags_out_kernel, dim3(1), dim3(32), 0, s, flags, hflags);
}

// Per-configuration virial: one CTA per configuration sums its atoms in a
// fixed order (strided partial sums, then a tree).
__global__ void __launch_bounds__(256) virial_conf_kernel(const double* __restrict__ vatom,
                                                          const NeighConf* __restrict__ confs,
                                                          double* __restrict__ virial) {
  __shared__ double red[256];
  const NeighConf c = confs[blockIdx.x];
  for (int k = 0; k < 6; ++k) {
    double t = 0.0;
    for (int i = threadIdx.x; i < c.n; i += blockDim.x) t += vatom[6 * (long)(c.start + i) + k];
    red[threadIdx.x] = t;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
      if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) virial[6 * blockIdx.x + k] = red[0];
    __syncthreads();
  }
}

cudaError_t launch_virial_conf(const double* vatom, const NeighConf* confs, int nconf, double* virial,
                               cudaStream_t s) {
  if (nconf <= 0) return cudaSuccess;
  return launch_k(virial_conf_kernel, dim3(nconf), dim3(256), 0, s, vatom, confs, virial);
}

template cudaError_t launch_yi<float>(const WorkArgs&, cudaStream_t);
template cudaError_t launch_yi<double>(const WorkArgs&, cudaStream_t);
template cudaError_t launch_force<float>(const WorkArgs&, cudaStream_t);
template cudaError_t launch_force<double>(const WorkArgs&, cudaStream_t);

// ------------------------------------------------- FMA throughput probe
// Peak FMA rate of the working precision, for the roofline denominators:
// every thread runs kProbeChains independent multiply-add chains (enough to
// cover the pipeline latency) for `iters` rounds.  The chains' operands come
// from the arguments, and the sums are stored only under a condition the host
// never meets, so nothing is folded away.
constexpr int kProbeChains = 8;

template <typename R>
__global__ void __launch_bounds__(256) fma_probe_kernel(int iters, R b, R c, R* sink) {
  R x[kProbeChains];
#pragma unroll
  for (int k = 0; k < kProbeChains; ++k) x[k] = R(threadIdx.x + k);
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int k = 0; k < kProbeChains; ++k) x[k] = fma(x[k], b, c);
  }
  R t = R(0);
#pragma unroll
  for (int k = 0; k < kProbeChains; ++k) t += x[k];
  if (t == R(-12345.0)) sink[threadIdx.x] = t;
}

template <typename R>
cudaError_t fma_probe(int nsm, int iters, double* flops, float* ms, R* sink, cudaStream_t s) {
  const int blocks = nsm * 8, threads = 256;
  cudaEvent_t e0, e1;
  cudaError_t e = cudaEventCreate(&e0);
  if (e != cudaSuccess) return e;
  e = cudaEventCreate(&e1);
  if (e != cudaSuccess) return e;
  // warm-up launch, then the timed one
  e = launch_k(fma_probe_kernel<R>, dim3(blocks), dim3(threads), 0, s, iters / 8, R(0.999), R(1e-3), sink);
  if (e == cudaSuccess) e = cudaEventRecord(e0, s);
  if (e == cudaSuccess) e = launch_k(fma_probe_kernel<R>, dim3(blocks), dim3(threads), 0, s, iters, R(0.999), R(1e-3), sink);
  if (e == cudaSuccess) e = cudaEventRecord(e1, s);
  if (e == cudaSuccess) e = cudaEventSynchronize(e1);
  if (e == cudaSuccess) e = cudaEventElapsedTime(ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  *flops = 2.0 * kProbeChains * 4 * (double)iters * blocks * threads;
  return e;
}
template cudaError_t fma_probe<float>(int, int, double*, float*, float*, cudaStream_t);
template cudaError_t fma_probe<double>(int, int, double*, float*, double*, cudaStream_t);

}  // namespace snap
