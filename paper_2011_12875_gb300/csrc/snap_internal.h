// snap_internal.h -- device-side layouts and launcher prototypes shared by the
// library's translation units (not part of the public C ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <mutex>
#include <unordered_map>

namespace snap {

// Kernel launch with the configuration as arguments (one place to change how
// the library launches).
#ifdef __CUDACC__
template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                            cudaStream_t s, Args... args) {
  kernel<<<grid, block, smem, s>>>(static_cast<KArgs>(args)...);
  return cudaGetLastError();
}
#endif

// Shared memory of a CTA: the most there is, and what a launch may use without
// being allowed to.
constexpr size_t kSmemMax = 227 * 1024, kSmemFree = 48 * 1024;

// Allows a launch of `kernel` with `bytes` of dynamic shared memory.  The limit
// is an attribute of the function, which every context and host thread shares,
// so it is always set to the same value, the most the kernel can have: set to a
// launch's own bytes, one thread could lower it between another's setting it
// and launching.
inline cudaError_t allow_smem_of(const void* kernel, size_t bytes) {
  size_t fixed;  // static shared memory, looked up once
  {
    static std::mutex mu;
    static std::unordered_map<const void*, size_t> seen;
    std::lock_guard<std::mutex> lock(mu);
    auto it = seen.find(kernel);
    if (it == seen.end()) {
      cudaFuncAttributes fa;
      const cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
      if (e != cudaSuccess) return e;
      it = seen.emplace(kernel, fa.sharedSizeBytes).first;
    }
    fixed = it->second;
  }
  if (bytes + fixed <= kSmemFree) return cudaSuccess;
  if (bytes + fixed > kSmemMax) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kSmemMax - fixed));
}
template <typename K>
inline cudaError_t allow_smem(K kernel, size_t bytes) {
  return allow_smem_of(reinterpret_cast<const void*>(kernel), bytes);
}

constexpr int kMaxTwoJ = 14;
constexpr int kYcChunk = 256;  // words of a compute_Y stream chunk (snap_tables.h)
constexpr int kYcOuts = 8;     // most outputs of a compute_Y task
constexpr int kYcTask = 4 + 2 * kYcOuts;
// Cost from which a task's sum is split in two.  compute_Y, 2000 atoms, us, from 300 /
// 1000 / 3000 / never: FP32 2J8 34.1 / 33.8 / 32.6 / 36.3, 2J14 388 / 388 / 388 / 491; FP64 2J6
// 60 / 61 / 70 / 72, 2J8 170 / 170 / 171 / 174.
constexpr long kYcWhole = 1000;
constexpr int kPairFix = 8;  // most steps of a class (HostTables::pair_fix)
constexpr int kUUnit = 8;  // words of a compute_U unit (HostTables::u_units)
constexpr int kYcNan = 0x7FFF;  // exponent of an output whose coefficients are not finite
constexpr int kBChunk = 96;    // bispectrum terms a warp takes at a time (whole groups)
constexpr int kBMaxChunks = 1024;  // chunks are lengthened past this count
constexpr int kBGroupMax = 8;      // longest bispectrum term piece (longer groups are cut)
constexpr int kMaxNeighCap = 64;
constexpr int kGeomStride = 20;  // doubles per neighbour slot, see PairGeom

// A coefficient of compute_Y's stream: without beta, its word and its triple
// (HostTables::yc_list).
struct __align__(16) YcCoef {
  double cg;
  int at, trip;
};
// The coefficients of a record for one output, coef[first ..) to the next one's.
struct YcGroup {
  int first, out;  // out: task x kYcOuts + output
};

// compute_Y's fixed point (snap_kernels.cu), on the device and in its host walk.
// limbs of v, |v| < 2^59, given v + 2^29: v = h 2^30 + l, -2^29 <= l < 2^29
__host__ __device__ inline void split30(long long v, int& h, int& l) {
  h = (int)(v >> 30);
  l = (int)((unsigned)v & 0x3FFFFFFFu) - (1 << 29);
}
// An atom's scale, the biased exponent E of its largest component of U (top: the
// high word of that magnitude): components are held in units of 2^(E - 1022 -
// 59).  U below 2^-150 has that scale; 0x7FF: not finite.
__host__ __device__ inline int yc_scale(int top) { return top >> 20 > 1022 - 150 ? top >> 20 : 1022 - 150; }
// The limbs of a component (low and high word) at scale E, rounded to nearest,
// halves away from zero; subnormals count as zero.
__host__ __device__ inline void yc_limbs(int lo, int hi, int E, int& h, int& l) {
  const int e = (hi >> 20) & 0x7FF;
  // |x| = M 2^(e - 1075) = v 2^(E - 1022 - 59)
  const unsigned long long M = ((unsigned long long)((hi & 0xFFFFF) | 0x100000) << 32) | (unsigned)lo;
  const int sh = e - E + 6;
  unsigned long long v = 0;
  if (sh >= 0) v = M << (sh & 7);
  else if (sh > -55) v = (M + (1ull << (-sh - 1))) >> -sh;
  if (e == 0) v = 0;
  split30((hi < 0 ? -(long long)v : (long long)v) + (1LL << 29), h, l);
}

// Half-matrix layout (Sec. V-A: u_j only needs floor(j)+1 of its columns):
// layer t = 2j holds columns mb = 0..t/2, each column ma = 0..t.
__host__ __device__ constexpr int half_layer_size(int t) { return (t + 1) * (t / 2 + 1); }
__host__ __device__ constexpr int half_base(int t) {
  int n = 0;
  for (int s = 0; s < t; ++s) n += half_layer_size(s);
  return n;
}
__host__ __device__ constexpr int half_size(int twojmax) { return half_base(twojmax + 1); }

// Packed (t, ma, mb) of a half-layout element.
__host__ __device__ constexpr int pack_tmm(int t, int ma, int mb) { return t | (ma << 8) | (mb << 16); }
__host__ __device__ constexpr int tmm_t(int p) { return p & 0xff; }
__host__ __device__ constexpr int tmm_ma(int p) { return (p >> 8) & 0xff; }
__host__ __device__ constexpr int tmm_mb(int p) { return (p >> 16) & 0xff; }

// compute_Y term record: w = index of U_t1 element (10 bits) | index of the
// U_t2 element << 10 | conj U_t1 << 20 | conj U_t2 << 21 | last term of the
// output << 22; c = coefficient in the working precision.
template <typename R>
struct YRec;
template <>
struct __align__(8) YRec<float> {
  unsigned w;
  float c;
};
template <>
struct __align__(16) YRec<double> {
  unsigned w, pad;
  double c;
};

// Per neighbour slot geometry (Cayley-Klein parameters, Sec. II-A), computed
// in FP64 and stored in the working precision R:
//  [0..1] a, [2..3] b, [4] f_c, [5..7] d f_c / d r_d,
//  [8..13] d a / d r_d (re, im per d), [14..19] d b / d r_d.
// A slot with r >= rcut has f_c = 0 and zero derivatives.

// One configuration of a batch: atoms [start, start + n), box L, image
// shifts S enumerated beyond the nearest image.
struct NeighConf {
  int start, n;
  double L[3];
  int S[3];
};

// Image shifts the device neighbour build enumerates beyond the nearest
// image, per axis: none when the box is longer than 2 (rcut + 0.05 A), else
// ceil(rcut / L) + 1.  The build loops over (2 Sx + 1)(2 Sy + 1)(2 Sz + 1)
// images for every 32 candidates and stores shifts as signed bytes, so a box
// that needs more than kMaxImageLoop images in all, or more than kMaxImageShift
// along one axis, is refused (false): such a box holds more images of a
// single atom within rcut than any neighbour capacity.  rcut and the box
// lengths must be finite and positive.
constexpr int kMaxImageLoop = 4096;
constexpr int kMaxImageShift = 100;
inline bool image_shifts(const double* L, double rcut, int S[3]) {
  if (!(rcut > 0.0 && rcut < 1e30)) return false;
  long loop = 1;
  for (int d = 0; d < 3; ++d) {
    if (!(L[d] > 0.0 && L[d] < 1e300)) return false;
    const double q = rcut / L[d];
    if (!(q < (double)kMaxImageShift)) return false;
    S[d] = (L[d] > 2.0 * (rcut + 0.05)) ? 0 : (int)std::ceil(q) + 1;
    if (S[d] > kMaxImageShift) return false;
    loop *= 2L * S[d] + 1;
  }
  return loop <= kMaxImageLoop;
}

// centre atoms per CTA of the device neighbour build
constexpr int kNeighAtomsPerCta = 2;

struct NeighArgs {
  int n, K;
  // batch mode: confs != nullptr; CTA b builds atoms
  // cta_map[b].y + 0..kNeighAtomsPerCta-1 of configuration cta_map[b].x
  const NeighConf* confs;
  const int2* cta_map;
  const double* pos;     // [n][3]
  const float4* pos4;    // [n] FP32 copy for the coarse test
  // [ceil(n/32)][2]: FP32 centre and half extent of each 32-atom tile, for
  // skipping far tiles in the single-configuration build; nullptr: no skipping
  const float4* tiles = nullptr;
  double Lx, Ly, Lz;
  int Sx, Sy, Sz;        // image shifts enumerated beyond the nearest image
  double rcut;
  int* cnt;
  int* nbr;
  signed char* img;
  double* rij;
  int* key;  // [n][K] pair_key of every stored slot, or nullptr
  int* flags;
};

// Search key of a stored pair (k, image s): k * 32 + the image's code
// (s_d + 1 in base 3) when every |s_d| <= 1 (and the atoms index below 2^26),
// else -1.  The opposite pair (i, -s) has code 26 - code, so the force gather
// finds the reverse slot with one pass over k's row of keys.
__host__ __device__ constexpr int pair_key(int k, int ix, int iy, int iz, long n) {
  return (ix >= -1 && ix <= 1 && iy >= -1 && iy <= 1 && iz >= -1 && iz <= 1 && n < (1L << 26))
             ? k * 32 + (ix + 1) * 9 + (iy + 1) * 3 + (iz + 1)
             : -1;
}

// What a kernel reads stands together: every CTA fetches its lines of it.
struct WorkArgs {
  int n, K, twojmax, H;
  double rcut, rfac0, rmin0, wself, beta0;
  double inv_span;  // 1 / (rcut - rmin0)
  double th_scale;  // rfac0 / (rcut - rmin0): theta0 / pi = th_scale (r - rmin0)
  // FP32 copies for the mixed path's slot gradients (no FP64 work per slot):
  // th_scale, d theta0 / d r = pi th_scale, 1 / (rcut - rmin0), rmin0 and
  // the switching derivative's factor -pi / (2 (rcut - rmin0))
  float th_scale_f, dth_f, inv_span_f, rmin0_f, dfc_f;
  int switchflag;
  const int* cnt;
  const int* nbr;
  const signed char* img;
  const int* rev;
  int* rev_out;  // the same table, written by the force kernel
  const int* key;  // [N][K] pair_key of every slot
  double* rij;
  void* geom;  // R [N][K][kGeomStride]: Cayley-Klein geometry in the working precision
  // Ulisttot and Y: complex (re, im interleaved), AoSoA [ceil(N/32)][H][32]
  void* U;
  void* Y;
  double* dedr;
  double* vatom;   // per-atom virial [N][6] (batch mode) or nullptr
  double* energy;
  double* forces;
  double* vpart;
  double* virial;
  int* flags;
  // non-null on the kernel that ends an evaluation (the force kernel): its
  // last CTA writes flags[0..3] to this host-mapped copy and zeroes the flags
  int* hflags;
  const int* half_tmm;
  const void* hscale;  // R [H]: S_t(ma, mb) of the scaled recursion (u = S v)
  int nsm;
  int col_warps;  // fused dE: an SM with few batches shares them (tunable, de_plan)
  int de_maxcnt;  // neighbour count the fused dE launch is planned for (last seen maximum, else K)
  int yi_waves;   // compute_Y waves per SM (tunable)
  int persist;    // tunable: bit 0 persistent compute_Y, bit 1 persistent fused dE (work queues)
  int de_atoms;   // tunable: atoms per fused dE CTA (0: planned)
  int test_skip_stage;  // test hook: TMA staging registers its bytes but issues no copy
  // bispectrum output
  int ncoeff;
  const void* brec;       // YRec<R> records of the bispectrum terms (sign-flip words)
  const void* brec_cp;    // the same records in the conjugate-plane words (null: unused)
  const int* bchunk_term;   // chunks of the bispectrum term list (snap_tables.h)
  const void* bchunk_runs;  // [nchunks][kBGroupMax] u16: pieces of 1, 2, ... terms of every chunk
  const int* bcomp_chunk;
  int bi_layout;            // tunable: 0 planned, 1 sign flips, 2 conjugate plane
  void* bscratch;           // partial sums of the bispectrum chunks when shared memory is short
  const int* bpart;         // [nbparts+1] first component of each CTA's run
  int nbparts, bmaxchunks, bmaxterms;  // runs, most chunks and most terms of one run
  double* B;              // [N][ncoeff]
  // compute_Y's tables (HostTables::yc_*); yc_bins for yc_split CTAs a block
  void* Y2;  // the second halves of split sums (as Y; the tangent's buffer)
  const int* yc_bins;
  const int* yc_slot;
  const int* yc_task;
  const unsigned* yc_stream;
  int yc_split, yc_ntask;
  int yi_layout;          // 0: warp of 32 atoms (AoSoA), 1: warp per atom
  // warp-per-atom layout: term records (snap_tables.cpp), [H+1] first term of
  // each output element, [32][ysched_m] outputs of each lane
  int ysched_m;
  const void* yrec;
  const int* yfirst;
  const int* ysched;
  // closed-form u of a pair (snap_pairs.cuh, HostTables::pair_*), per step
  const unsigned* pair_idx;
  const void* pair_scale;  // step_scale<R>: norm x weight
  const void* pair_norm;   // step_scale<R>
  const void* pair_ab;     // rec_ab<R>
  const double* pair_fix;  // FP64: [step][kPairFix], the polynomials' rounding (HostTables::pair_fix)
  const int* pair_cls;     // FP64: the classes of several steps, first step | steps << 16
  int npair_steps, npair_cls;
  // compute_U's units, [u_nunits + u_nfine][kUUnit] (HostTables::u_units)
  const int* u_units;
  int u_nunits, u_nfine, u_cost;
};

// Launchers (snap_neigh.cu)
cudaError_t launch_pos4(int n, const double* pos, float4* pos4, cudaStream_t s, float4* tiles = nullptr,
                        double* copy = nullptr);
cudaError_t launch_neigh_build(const NeighArgs& a, cudaStream_t s);
// Caller-supplied list to the internal tables, with (geom) the slots' geometry.
template <typename R>
cudaError_t launch_neigh_ingest(const WorkArgs& a, bool geom, const double* pos, double Lx, double Ly, double Lz,
                                const int* ucnt, const int* uidx, const signed char* uimg, int ucap, int* cnt, int* nbr,
                                signed char* img, double* rij, int* key, int* flags, cudaStream_t s);

// Launchers (snap_u.cu): the neighbour build with the slots' geometry, one
// configuration (ncta = 0) or a batch of ncta CTAs (na.confs); compute_U.
template <typename R>
cudaError_t launch_neigh_geom(const NeighArgs& na, const WorkArgs& a, int ncta, cudaStream_t s);
template <typename R> cudaError_t launch_u(const WorkArgs& a, cudaStream_t s);

// Launchers (snap_kernels.cu), R = float (mixed) or double (FP64)
template <typename R> cudaError_t launch_yi(const WorkArgs& a, cudaStream_t s);

// The stream's words that depend on beta (bw: HostTables::beta_weights, device).
// fixed: the FP64 path's fixed point, top [tasks x kYcOuts] scratch.
cudaError_t launch_yc_coefs(bool fixed, const YcCoef* coef, int ncoef, const YcGroup* group, int ngroup, const double* bw,
                            const int* task, int ntask, int nchunk, unsigned long long* top, unsigned* stream,
                            cudaStream_t s);

// Launch shape of compute_Y for N atoms: nblk blocks of atoms x split CTAs of
// `threads`, with `smem` bytes of shared memory.
struct YiGeometry {
  int nblk, split, threads;
  size_t smem;
};
// The warp-per-atom layout's term record word ends a group (the rest of the
// word: yi_atom_kernel).
constexpr unsigned kYaGroup = 1u << 28;
YiGeometry yi_geometry(int rsize, int H, int n, int nsm, int waves, int ntasks);

// End of an evaluation: flags[0..3] into the host-mapped status words
// (device pointer hflags), all eight flags zeroed.
cudaError_t launch_flags_out(int* flags, int* hflags, cudaStream_t s);

// Per-configuration virial: sum of vatom over each configuration's atoms.
cudaError_t launch_virial_conf(const double* vatom, const NeighConf* confs, int nconf, double* virial,
                               cudaStream_t s);
template <typename R> cudaError_t launch_force(const WorkArgs& a, cudaStream_t s);
template <typename R> cudaError_t launch_bi(const WorkArgs& a, cudaStream_t s);

// Launch plan of the bispectrum kernels (B and dB) for the precision's size
// (4 or 8 bytes), H, and the most chunks and terms of a CTA's run: the
// block's planes staged (U's, and dU's when both fit) or read from global memory, the conjugate plane or
// sign flips, the run's term records staged or read through L1 (rs), the
// partial sums in shared memory or in the global scratch (gpart, then CTAs x
// maxchunks x 32 x rsize bytes), and the dynamic shared memory.  Layout:
// [planes][barrier, 16 B][records, rec_bytes][partials].
constexpr int kBiThreads = 512;
constexpr int kBiCtasPerSm = 2;  // register budget of the kernels (64 a thread)
constexpr size_t kBiSmemMax = 200 * 1024;   // one CTA an SM
constexpr size_t kBiSmemPair = 112 * 1024;  // two CTAs an SM
struct BiPlan {
  bool staged, ds, cp, rs, gpart;  // ds: the tangent's block staged beside U (dB)
  size_t smem, rec_bytes;
};
BiPlan bi_plan(int rsize, int H, bool deriv, int maxchunks, int maxterms, int layout, bool have_cp);
// whether the conjugate-plane records can ever be used for this size and H
bool bi_plane_fits(int rsize, int H);

// compute_U by the layer recursion (snap_col_*.cu), 2J <= u_col_max: for caller
// lists, and fused with the neighbour build, one configuration (ncta = 0) or a
// batch.
constexpr int u_col_max(size_t rsize) { return rsize == 4 ? 9 : 5; }
template <typename R> cudaError_t launch_ui_col(const WorkArgs& a, cudaStream_t s);
template <typename R> cudaError_t launch_neigh_u(const NeighArgs& na, const WorkArgs& a, int ncta, cudaStream_t s);
// Tangent of Ulisttot along the displacement field g ([N][3], device); 0..14.
template <typename R>
cudaError_t launch_tan_col(const WorkArgs& a, const double* g, void* dU, cudaStream_t s);

// Fused dU + dE/dr in closed form (snap_pairs.cuh), 0 <= twojmax <= 14.
template <typename R> cudaError_t launch_de(const WorkArgs& a, cudaStream_t s);

// d B_l along the tangent dU (snap_kernels.cu) and the weighted force gather.
template <typename R> cudaError_t launch_dbi(const WorkArgs& a, const void* dU, double* dB, cudaStream_t s);
cudaError_t launch_force_weighted(const WorkArgs& a, const double* w, double* grad, cudaStream_t s);

// FMA throughput probe (synchronous): flops and milliseconds of one timed launch
template <typename R>
cudaError_t fma_probe(int nsm, int iters, double* flops, float* ms, R* sink, cudaStream_t s);

}  // namespace snap
