// Internal definitions of the GB300 J/K builder: constants, index helpers,
// device-side data layout and the shell-pair handle.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "../../include/fock.h"
#include "streams.h"

namespace fk {

// Whether a handle's quartets below the cutoff run in FP32.
inline bool mixed_opts(const fock_opts &o) {
  return (o.precision & ~FOCK_NO_TWO_FLOAT) == FOCK_MIXED && o.fp32_cutoff > 0.0;
}

constexpr int LMAX = 3;             // f functions
constexpr int LTOT = 4 * LMAX;      // largest total angular momentum of a quartet
constexpr int NCLASS = 10;          // pair classes (la >= lb)
constexpr int MAXPRIM = 8;          // primitives per shell
constexpr int MAXCP = 100;          // Cartesian pairs of an (f,f) pair
constexpr int NHMAX = 455;          // Hermite functions with t+u+v <= 12

// Boys table: F_k(T_i), T_i = i*h, k = 0..BOYS_NORD-1, Taylor expansion of
// order BOYS_TAYLOR about the nearest grid point; T >= BOYS_TMAX uses the
// asymptotic form F_0 = sqrt(pi/T)/2 with upward recursion.
constexpr int BOYS_TAYLOR = 8;                 // terms k = 0..7
constexpr int BOYS_NORD = LTOT + BOYS_TAYLOR;  // orders 0..19
constexpr double BOYS_H = 1.0 / 16.0;
constexpr double BOYS_INVH = 16.0;
constexpr double BOYS_TMAX = 64.0;
constexpr int BOYS_NGRID = 1025;               // T_i for i = 0..1024
// Two-float table: F_n(T_i), n = 0..BOYSFF_NORD-1, T_i = i/64 up to BOYS_TMAX
constexpr float BOYSFF_INVH = 64.0f;
constexpr int BOYSFF_NGRID = 4097;
constexpr int BOYSFF_NORD = LTOT + 6;          // a row is 144 bytes (16-byte aligned)

__host__ __device__ constexpr int ncart(int l) { return (l + 1) * (l + 2) / 2; }
__host__ __device__ constexpr int nherm(int L) { return (L + 1) * (L + 2) * (L + 3) / 6; }
__host__ __device__ constexpr int pair_class(int la, int lb) { return la * (la + 1) / 2 + lb; }

// Compact index of the Hermite (or Cartesian) exponent vector (t,u,v):
// ordered by degree t+u+v, then t descending, then u descending.
__host__ __device__ inline int hidx(int t, int u, int v) {
  int d = t + u + v, r = d - t;
  return d * (d + 1) * (d + 2) / 6 + r * (r + 1) / 2 + (r - u);
}

// Cartesian component i (0..ncart(l)-1) of a shell of angular momentum l.
__host__ __device__ inline void cart_comp(int l, int i, int &x, int &y, int &z) {
  int k = 0;
  while (i > k) {
    i -= k + 1;
    ++k;
  }
  x = l - k;
  y = k - i;
  z = i;
}

// Primitive-pair centre and exponent (Px, Py, Pz, zeta), one 32-byte load.
struct __align__(32) PZ {
  double x, y, z, w;
};

// Per-class constant tables, copied into shared memory by the kernels
// (16-byte aligned so its size is a whole number of 16-byte words).
struct alignas(16) ClassTables {
  int16_t eoff[NCLASS][MAXCP + 1];   // E offset of Cartesian pair k within a primitive pair block
  int16_t nE[NCLASS];                // E doubles per primitive pair
  uint8_t comp[LMAX + 1][10][3];     // Cartesian components per shell
  uint8_t hvec[NHMAX][3];            // (t,u,v) of compact Hermite index
};

// Device view of a handle's pair data (plain pointers, passed by value).
struct DevPairs {
  // shells
  const double *sxyz;  // [3*nshell]
  const int *sbf;      // first basis function
  const int *sl;       // angular momentum
  // contracted pairs, sorted (class, contraction bucket, G descending)
  const int2 *ab;      // canonical shells (la >= lb; a >= b when la == lb)
  const double *G;     // Schwarz factor G_ab
  const int2 *prim;    // (first primitive pair, count)
  const int *cls;      // pair class
  // primitive pairs
  const PZ *pz;        // (Px, Py, Pz, zeta)
  const float4 *pf;    // the same in FP32 (grid indices, seeds)
  const int *eoff;     // offset of the primitive pair's E block
  const double *E;     // Hermite coefficients (Cartesian normalisation and U folded in)
  const double *Gp;    // primitive Schwarz factor G_[ab]; each pair's primitives sorted by it, descending
  const float *Gpf;    // the same rounded to FP32
  // FP32 copies for the mixed-precision path and the FP32 screening pre-test
  const float *Gf;     // G_ab rounded to FP32
  const float *shl;    // shell centres as FP32 hi/lo pairs: [6*s] = hx hy hz lx ly lz
  const float4 *paf;   // (P - A, zeta) with A the first shell of the canonical pair
  const float4 *pal;   // remainders of paf (two-float path): P - A and zeta less their FP32 values
  const float2 *E2;    // Hermite coefficients as two floats (null without the two-float path)
  const float *Ef;     // Hermite coefficients, FP32 (null without an FP32 path)
  const int *smol;     // shell -> molecule of a batch (null for one molecule)
  const int *satom;    // shell -> atom (shells on one atom share an index)
  const float *Gn;     // nshell^2: n_z G_xz for kept pairs (x, z), else 0 (GDG bound)
  const float2 *sRG;   // per shell: radius R_s and largest Schwarz factor G_s of its kept pairs
  int nshell, nbf, npair;
  int nprim_total;
  long long nE_total;
};

// Per-molecule entry of a batched build (device table, rewritten per call).
struct MolEntry {
  const double *D;
  double *J;
  double *K;
  const float *Df;     // FP32 copy of D (mixed path) or null
  long long dsh_off;   // offset of the molecule's nshell^2 block maxima
  long long n2_off;    // offset of the molecule's N^2 block in packed per-call arrays
  int N, s0, ns;       // functions, first shell, shells
  float gmax2;         // largest G_ab^2 of the molecule
};

// Host arrays mirroring DevPairs (the compact, sorted data of a handle).
struct Staging {
  std::vector<double> sxyz;
  std::vector<int> sbf, sl;
  std::vector<int2> ab;
  std::vector<double> G;
  std::vector<int2> prim;
  std::vector<int> cls;
  std::vector<PZ> pz;
  std::vector<float4> pf;
  std::vector<int> eoff;
  std::vector<double> E;
  std::vector<double> Gp;
  std::vector<float> Gpf;
  std::vector<float4> paf, pal;
  std::vector<float> Ef, Gf, shl;
  std::vector<int> smol;
  std::vector<int> satom;
  std::vector<float2> sRG;
  std::vector<float> Gn;
};

// One unit of work: bra pair index, ket pair index range [k0, k1).
struct Unit {
  int bra, k0, k1, pad;
};

// Launch shape of a group kernel (kernels_group.cu).
struct GroupConfig {
  int G = 0, warps = 0, blocks = 0;  // lanes per quartet (0 = not used), warps per block, grid
  size_t smem = 0;
};

// All work units of one (bra class, ket class) pair and their launches.
struct Tier {
  int cb = 0, ck = 0;   // bra class, ket class
  bool reg = false;     // on the per-class register kernels (else the group kernels)
  bool r32 = false;     // group tier whose FP32 part runs on the FP32 register kernel
  bool in_range = true;  // seeds within the FP32 exponent range, see seeds_in_range
  int tag = 0;          // class pair + 1 when class pairs are timed apart (tuning)
  int G = 1;            // lanes per quartet (group kernels)
  GroupConfig grp, g32;  // group kernels: FP64 and two-float lists; FP32 list (mixed)
  int blocks = 0;       // grid of the register kernel (all lists, or FP64 and FP32)
  int blocks_hi = 0;    // the same for FP64 alone beside the two-float kernels
  int blocks_ff = 0;    // grid of the two-float register kernel (0: all lists in one)
  int blocks32 = 0;     // grid of the FP32 register kernel of a group tier
  long long quartets = 0;  // Schwarz-passing quartets
  int maxprim = 1;      // most primitive quartets of one quartet
  int nsplit = 1;       // shares of a quartet's primitive quartets
  double cost = 0.0;    // modelled work, for the order of the launches
  bool queued = false;  // its launches wait for those of the other tiers, see set_queued
  int nunits;
  Unit *d_units;
};

// Whether the seeds pref (-2 alpha)^m F_m(T), pref = 1/sqrt(zeta + eta), m = 0..L,
// of a class pair fit the FP32 exponent range for all exponents zeta in
// [z0, z1], eta in [e0, e1] (sums of two primitive exponents), alpha = zeta eta /
// (zeta + eta).  The powers pref (2 alpha)^m are formed before they meet F_m, and
// the recursion makes nothing larger of them, so 2^120 leaves it room below
// 2^128.  At the lower end F_m(0) = 1/(2m+1) counts, and the remainder of a value
// (2^-48 of it) has to be a multiple of 2^-149: 2^-100.  With equal exponents
// that admits f shells of 1.7e-3 .. 690, (fd|fd) of 5e-4 .. 3e3, (dd|dd) of 8e-5 ..
// 3e4; outside a class pair runs in FP64 alone.
inline bool seeds_in_range(int L, double z0, double z1, double e0, double e1) {
  const double a0 = 2.0 * z0 / (z0 + e0) * e0, a1 = 2.0 * z1 / (z1 + e1) * e1;
  const double hi = -0.5 * log2(z0 + e0) + L * std::max(0.0, log2(a1));
  const double lo = -0.5 * log2(z1 + e1) + L * std::min(0.0, log2(a0)) - log2(2.0 * L + 1.0);
  return hi < 120.0 && lo > -100.0;
}

// Threads that keep the chip busy: 152 SMs x 16 warps.
constexpr long long kFillThreads = 152 * 16 * 32;

// A tier that would leave most of the chip's threads without a quartet shares
// each quartet's primitive quartets between up to 8 threads (groups), as far as
// every share keeps at least two; large tiers keep whole quartets, which are
// digested once.
inline void set_split(Tier &t) {
  const int lanes = t.reg ? 1 : t.G;
  t.nsplit = 1;
  while (t.nsplit < 8 && 4 * t.nsplit <= t.maxprim && t.quartets * lanes * t.nsplit < kFillThreads / 2) t.nsplit *= 2;
}

// Whether a build's launches run side by side or (FP64 ones of larger classes
// apart) one after the other.  Side by side they hide one another's beginnings and
// ends; but bodies that share an SM also evict one another's instructions, and in
// a build large enough for the ends not to matter that costs more.  Measured, one
// after the other against side by side, modelled operations of the build in
// brackets: mixed C12H26 (0.3e11) 22.5 against 17.9 ms, C20H42 (1.2e11) 55.4
// against 54.3, (H2O)20 (1.7e11) 69 against 74, (H2O)32 (7e11) 222 against 284,
// (H2O)40 (13e11) 403 against 549; FP64 C20H42 100 against 97, C31H64 (3.1e11)
// 248 against 249, (H2O)32 416 against 462, (H2O)40 771 against 882.
inline void set_queued(std::vector<Tier> &tiers, bool mixed) {
  double cost = 0.0;
  for (const Tier &t : tiers) cost += t.cost;
  for (Tier &t : tiers) t.queued = cost >= (mixed ? 1.5e11 : 6e11);
}
}  // namespace fk

struct fock_shellpairs {
  int device = 0;
  int nshell = 0, nbf = 0;
  double tau_build = 0.0, prune_eps = 1e-3;
  fock_opts opts{};
  // host copies (for statistics and tests)
  std::vector<double> h_sxyz;
  std::vector<int> h_sbf, h_sl;
  std::vector<int2> h_ab;
  std::vector<double> h_G;
  std::vector<int2> h_prim;
  std::vector<int> h_cls;
  std::vector<fk::Unit> h_units;      // all tiers, concatenated
  std::vector<int> h_unit_tier;
  fk::Staging host;                   // compact pair data (merged into batch plans)
  std::vector<double> h_R, h_Gs;      // per-shell radius and Schwarz maximum (decay bound)
  int decay_nbins = 0;                // 0.5-bohr distance bins of the decay fit
  unsigned long long serial = 0;      // unique id (batch plan cache key)
  float gmax2 = 0.0f;                 // largest G_ab^2
  bool ff_ok = false;                 // two floats wanted; exponents, centres and integrals within their range
  // device allocations
  void *d_block = nullptr;            // one allocation holding all pair arrays
  fk::DevPairs dev{};
  std::vector<fk::Tier> tiers;
  std::vector<int> order;             // tiers by modelled work, descending
  size_t bytes = 0;
};

namespace fk {
// Byte offsets of the per-call scratch of a J/K build in one buffer (256-byte
// aligned parts): shell-block maxima (FP64) at 0, work counters, the FP32
// copy of D (mixed precision), FP32 block maxima, and in the decay-bound
// exchange mode the bounds W, the distance bins and H, Lambda.  (api.cu)
struct ScratchLayout {
  size_t cnt_off = 0, df_off = 0, dshf_off = 0, w_off = 0, bins_off = 0, hl_off = 0, t_off = 0, gdg_off = 0,
         total = 0;
};
ScratchLayout scratch_layout(const fock_shellpairs *sp);
// FOCK_OK, or what a build answers to its arguments.  (api.cu)
fock_status check_build_args(const fock_shellpairs *sp, const double *D, double schwarz_thresh, const double *J,
                             const double *K);
// The work of one build with its scratch in place, whatever it holds; ev (may be
// null): tiers + 1 events, recorded around the tiers, which then run one after
// the other.  Under a RelaxedCaptureMode.  (api.cu)
fock_status enqueue_build(const fock_shellpairs *sp, const double *D, double schwarz_thresh, double *J, double *K,
                          char *scratch, cudaStream_t stream, const cudaEvent_t *ev);

// Status of a CUDA runtime result; a failure also sets the text returned by
// fock_last_error ("where: error name (description)").  (api.cu)
fock_status cuda_status(cudaError_t e, const char *where);

// host helpers (host_pairs.cpp)
const ClassTables &class_tables();
const std::vector<double> &boys_table();
const std::vector<float2> &boys_table_ff();
void boys_eval_host(int mmax, double T, double *F);
void hermite_1d(int la, int lb, double p, double xpa, double xpb, double *E /*[4][4][7]*/);
int hermite_count(int la, int lb);
void hermite_pair(int la, int lb, double alpha, const double *A, double beta, const double *B,
                  bool cart_norm, double *out);

// Per-call choices of a J/K build besides precision: which matrices are built
// (1 = J, 2 = K, 3 = both) and the decay-bound exchange test (Wsh null: the
// exact test).
struct CallParts {
  int parts = 3;
  const float *Wsh = nullptr;  // nshell^2 decay bounds of the density blocks
  double k_thresh = 0.0;       // tau*
  const unsigned *dmax = nullptr;  // bits of max|D| (null: FP64 only)
  float gmax2 = 0.0f;
};

// device entry points (kernels.cu)
cudaError_t upload_tables(cudaStream_t st);
const double *dev_boys();
const float *dev_boys_f();
const float2 *dev_boys_ff();
const ClassTables *dev_class_tables();
cudaError_t launch_schwarz(const DevPairs &dp, const int2 *rows, const int *nrows, double *part, double *Gpair,
                           double *Gprim, cudaStream_t st);  // schwarz.cu
// dmax (may be null): receives the FP32 bits of max|D| by atomicMax (zeroed by the caller)
cudaError_t launch_dprep(const double *D, int nbf, const int *sbf, const int *sl, int nshell,
                         double *Dsh, cudaStream_t st, float *Df = nullptr, float *Dshf = nullptr,
                         unsigned *dmax = nullptr);
// E2[i] = E[i] as two floats
cudaError_t launch_split_e(const double *E, long long n, float2 *E2, cudaStream_t st);
// prim_eps: primitive-quartet screening factor (the handle's prune_eps; 0 = off)
// counters: kCounters work counters of this tier (one per part), zero
constexpr int kCounters = 3;
// par (may be null): the launches go to a stream of this set instead of st, by
// index, the place of the tier among the build's
cudaError_t launch_jk_tier(const Tier &t, const DevPairs &dp, const double *D, const double *Dsh,
                           double tau, double prim_eps, double *J, double *K, int *counters,
                           cudaStream_t st, StreamSet *par, int index, const float *Df = nullptr, double fp32_cutoff = 0.0,
                           const float *Dshf = nullptr, const CallParts &cp = CallParts());
// Decay bound of Sec. 4.3.1 for one density: bins (nbins doubles, zeroed
// here) of the block maxima Dsh of shells on different atoms by centre
// distance (0.5 bohr), the fit into HL[0] = H, HL[1] = Lambda, and the
// per-shell-pair bounds W (nshell^2 floats; null = fit only).  With Gn
// (nshell^2 floats, n_z G_xz over kept pairs), the FP32 block maxima Dshf and
// two nshell^2 float buffers T, GDG, blocks whose GDG bound is below
// k_thresh get W = 0.
cudaError_t launch_decay_bound(const DevPairs &dp, const double *Dsh, int nbins, double *bins, double *HL, float *W,
                               cudaStream_t st, const float *Gn = nullptr, const float *Dshf = nullptr,
                               float *T = nullptr, float *GDG = nullptr, double k_thresh = 0.0);
// bits of the streams that the launches of the index-th tier may use
unsigned tier_streams(int index);
cudaError_t launch_symmetrize(double *J, double *K, int n, cudaStream_t st);
// batched variants (one launch over every molecule of a batch)
cudaError_t launch_zero_batch(const MolEntry *mt, const long long *n2_prefix, int nmol, long long total,
                              cudaStream_t st);
cudaError_t launch_dprep_batch(const MolEntry *mt, const long long *dsh_prefix, int nmol, long long total,
                               const int *sbf, const int *sl, double *Dsh, float *Dshf, unsigned *dmax,
                               cudaStream_t st);
cudaError_t launch_symmetrize_batch(const MolEntry *mt, const long long *n2_prefix, int nmol, long long total,
                                    cudaStream_t st);
cudaError_t launch_jk_tier_batch(const Tier &t, const DevPairs &dp, const MolEntry *mt, const double *Dsh,
                                 const float *Dshf, const unsigned *dmax, double tau, double prim_eps,
                                 int *counters, cudaStream_t st, StreamSet *par, int index, double fp32_cutoff);
// Launch shapes of a tier's kernels; ff: the two-float path is on, mixed: the FP32
// path (both only for a tier in range).
cudaError_t configure_tier(Tier &t, bool ff, bool mixed);
int read_and_clear_status(cudaStream_t st, int *status);
int read_bounds(long long out[2]);
}  // namespace fk
