// GB300 (sm_103a) kernels around the J/K quartet kernels: density preparation and
// decay bound, symmetrisation, and the launches of a class pair's quartet kernels
// (kernels_reg.cuh, kernels_group.cu).
//
// Integral scheme: McMurchie-Davidson (arXiv:2407.21445 Sec. 4.1, Eqs. MD
// def, EabP def1-3): a primitive quartet is
//   [ab|cd] = sum_p sum_q E^{ab}_p (-1)^{|q|} R_{p+q} E^{cd}_q ,
// R_{tuv} from the Hermite recursion R^{(n)}_{t+1,u,v} = t R^{(n+1)}_{t-1,u,v}
// + X_PQ R^{(n+1)}_{tuv} seeded by R^{(n)}_{000} = pref (-2 alpha)^n F_n(T),
// pref = U_P U_Q 2 sqrt(alpha/pi), alpha = zeta eta / (zeta + eta),
// T = alpha |P-Q|^2 (the paper's garbled seed read this way).  For each bra
// primitive pair the ket primitive pairs are accumulated into the
// half-transformed Y[p][cd] = sum_q (-1)^{|q|} E^{cd}_q R_{p+q}, then
// ERI[ab][cd] += sum_p E^{ab}_p Y[p][cd]; the contracted ERIs are digested with
// the density into the six J/K blocks of the 8-fold permutational symmetry
// (Sec. 2.3, Sec. 3.2 "six Fock matrix blocks").
//
// GB300 executes FP64 at 1/64 of the FP32 rate: only the primitive quartets
// whose contribution needs 53 bits run on the FP64 pipe (kargs.cuh, kHiFrac),
// beside the others on the FP32 units.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <mutex>

#include "device_common.cuh"
#include "group.h"
#include "kargs.cuh"
#include "prec.cuh"
#include "reg_dispatch.h"

namespace fk {

__device__ int g_status = 0;  // sticky device status word (fock_status)

static double *s_boys[64];
static float *s_boysf[64];
static float2 *s_boysff[64];
static ClassTables *s_tabs[64];

// Shell-block maxima |D| (Sec. 3.2 density screening) and a finiteness check.
__global__ void k_dprep(const double *__restrict__ D, int N, const int *__restrict__ sbf,
                        const int *__restrict__ sl, int ns, double *__restrict__ Dsh, float *__restrict__ Df,
                        float *__restrict__ Dshf, unsigned *__restrict__ dmax) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= ns * ns) return;
  const int a = idx / ns, b = idx - a * ns;
  const int fa = sbf[a], fb = sbf[b], na = ncart(sl[a]), nb = ncart(sl[b]);
  double mx = 0.0;
  bool bad = false;
  for (int i = 0; i < na; ++i)
    for (int j = 0; j < nb; ++j) {
      const double v = D[(size_t)(fa + i) * N + fb + j];
      if (Df) Df[(size_t)(fa + i) * N + fb + j] = (float)v;
      if (!isfinite(v)) bad = true;
      mx = fmax(mx, fabs(v));
    }
  if (bad) atomicCAS(&g_status, 0, (int)FOCK_ERR_NONFINITE);
  Dsh[idx] = bad ? INFINITY : mx;
  if (Dshf) Dshf[idx] = bad ? INFINITY : (float)mx;
  // non-negative floats order like their bit patterns
  if (dmax) atomicMax(dmax, __float_as_uint(bad ? INFINITY : (float)mx));
}

__global__ void k_split_e(const double *__restrict__ E, long long n, float2 *__restrict__ E2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double x = E[i];
    const float h = (float)x;
    E2[i] = make_float2(h, (float)(x - (double)h));
  }
}

// --------------------------------------------------------------------------
// Decay bound of the density (Sec. 4.3.1, Eq. density_bound)
// --------------------------------------------------------------------------
// Centre distance of shells a and b, rounded the same way as a plain
// left-to-right evaluation (no fused multiply-adds), so that the 0.5-bohr bin
// of a pair is reproducible by any IEEE implementation.
__device__ __forceinline__ double centre_distance(const double *xyz, int a, int b) {
  const double dx = __dsub_rn(xyz[3 * a], xyz[3 * b]);
  const double dy = __dsub_rn(xyz[3 * a + 1], xyz[3 * b + 1]);
  const double dz = __dsub_rn(xyz[3 * a + 2], xyz[3 * b + 2]);
  return sqrt(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
}

constexpr double DECAY_BIN = 0.5;  // bohr

// Largest shell-block maximum of |D| per distance bin, over pairs of shells on
// different atoms (same-atom elements would skew the decay, Sec. 4.3.1).
// Non-negative doubles order like their bit patterns, so the maximum is an
// integer atomicMax.
__global__ void k_decay_bins(DevPairs dp, const double *__restrict__ Dsh, int nbins,
                             unsigned long long *__restrict__ bins) {
  const int ns = dp.nshell;
  const long long n = (long long)ns * ns;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * blockDim.x) {
    const int a = (int)(idx / ns), b = (int)(idx - (long long)a * ns);
    if (b <= a || dp.satom[a] == dp.satom[b]) continue;
    const double v = Dsh[idx];
    if (!(v > 0.0) || !isfinite(v)) continue;
    int k = (int)floor(centre_distance(dp.sxyz, a, b) / DECAY_BIN);
    if (k >= nbins) k = nbins - 1;
    atomicMax(bins + k, (unsigned long long)__double_as_longlong(v));
  }
}

// Least-squares line ln max|D| = ln H - Lambda r through the non-empty bins
// (r the bin centre), then ln H raised so that the line lies above each bin's
// maximum over the whole bin (its far edge when Lambda > 0).  Fewer than two
// bins: Lambda = 0, H the largest maximum.  One block.
__global__ void k_decay_fit(const unsigned long long *__restrict__ bins, int nbins, double *__restrict__ HL) {
  __shared__ double red[5][256];
  double n = 0, sx = 0, sy = 0, sxx = 0, sxy = 0;
  for (int i = threadIdx.x; i < nbins; i += blockDim.x) {
    const double v = __longlong_as_double((long long)bins[i]);
    if (!(v > 0.0)) continue;
    const double x = (i + 0.5) * DECAY_BIN, y = log(v);
    n += 1;
    sx += x;
    sy += y;
    sxx += x * x;
    sxy += x * y;
  }
  red[0][threadIdx.x] = n;
  red[1][threadIdx.x] = sx;
  red[2][threadIdx.x] = sy;
  red[3][threadIdx.x] = sxx;
  red[4][threadIdx.x] = sxy;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w)
      for (int k = 0; k < 5; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
    __syncthreads();
  }
  n = red[0][0];
  sx = red[1][0];
  sy = red[2][0];
  sxx = red[3][0];
  sxy = red[4][0];
  double lam = 0.0;
  if (n >= 2.0) {
    const double den = n * sxx - sx * sx;
    if (den > 0.0) lam = -(n * sxy - sx * sy) / den;
  }
  __syncthreads();
  // ln H = max over bins of y + Lambda * edge
  double m = -INFINITY;
  for (int i = threadIdx.x; i < nbins; i += blockDim.x) {
    const double v = __longlong_as_double((long long)bins[i]);
    if (!(v > 0.0)) continue;
    const double edge = (lam > 0.0 ? i + 1 : i) * DECAY_BIN;
    m = fmax(m, log(v) + lam * edge);
  }
  red[0][threadIdx.x] = m;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[0][threadIdx.x] = fmax(red[0][threadIdx.x], red[0][threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    HL[0] = red[0][0] == -INFINITY ? 0.0 : exp(red[0][0]);
    HL[1] = lam;
  }
}

// C = A B (transB = 0) or A B^T (transB = 1) for n x n row-major FP32
// matrices: 32 x 32 output tiles, 16 x 16 threads with 2 x 2 outputs each,
// K steps of 32 staged in shared memory; ragged edges read as zero.
__global__ void k_sgemm_nn(const float *__restrict__ A, const float *__restrict__ B, float *__restrict__ C, int n,
                           int transB) {
  __shared__ float As[32][33], Bs[32][33];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  for (int k0 = 0; k0 < n; k0 += 32) {
    for (int i = ty; i < 32; i += 16)
      for (int j = tx; j < 32; j += 16) {
        const int r = r0 + i, k = k0 + j;
        As[i][j] = (r < n && k < n) ? A[(size_t)r * n + k] : 0.f;
        const int kb = k0 + i, c = c0 + j;
        Bs[i][j] = (kb < n && c < n) ? (transB ? B[(size_t)c * n + kb] : B[(size_t)kb * n + c]) : 0.f;
      }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const float a0 = As[ty][k], a1 = As[ty + 16][k], b0 = Bs[k][tx], b1 = Bs[k][tx + 16];
      acc[0][0] = fmaf(a0, b0, acc[0][0]);
      acc[0][1] = fmaf(a0, b1, acc[0][1]);
      acc[1][0] = fmaf(a1, b0, acc[1][0]);
      acc[1][1] = fmaf(a1, b1, acc[1][1]);
    }
    __syncthreads();
  }
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      const int r = r0 + ty + 16 * i, c = c0 + tx + 16 * j;
      if (r < n && c < n) C[(size_t)r * n + c] = acc[i][j];
    }
}

// W_xy = H exp(-Lambda (|XY| - R_x - R_y)): for every kept pair (x z) and
// (y w), |ZW| >= |XY| - R_x - R_y, so W_xy bounds |D_zw|.  Where that distance
// bound is not positive the partners may share an atom (elements the fit
// excludes) and no bound is used (+inf).
// With GDG (the block bound (A Dsh A^T)_xy >= max |K_xy|, A_xz = n_z G_xz
// over kept pairs, Sec. 4.3.1's comparison with Luehr et al.) below tau*, the
// whole block K_xy is negligible and W_xy = 0 drops its contributions.
__global__ void k_decay_w(DevPairs dp, const double *__restrict__ HL, const float *__restrict__ GDG, float kthr,
                          float *__restrict__ W) {
  const int ns = dp.nshell;
  const long long n = (long long)ns * ns;
  const double H = HL[0], lam = HL[1];
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(idx / ns), y = (int)(idx - (long long)x * ns);
    const double r = centre_distance(dp.sxyz, x, y) - (double)dp.sRG[x].x - (double)dp.sRG[y].x;
    float w = r > 0.0 ? (float)(H * exp(-lam * r)) : INFINITY;
    // FP32 sums of non-negative terms: a relative margin of 1e-4 covers
    // their rounding, so the test only drops blocks the exact bound drops
    if (GDG && fmaxf(GDG[idx], GDG[(long long)y * ns + x]) * 1.0001f < kthr) w = 0.0f;
    W[idx] = w;
  }
}

static int grid_for(long long total) {
  long long b = (total + 255) / 256;
  if (b > 152 * 32) b = 152 * 32;
  return (int)(b > 0 ? b : 1);
}

cudaError_t launch_decay_bound(const DevPairs &dp, const double *Dsh, int nbins, double *bins, double *HL, float *W,
                               cudaStream_t st, const float *Gn, const float *Dshf, float *T, float *GDG,
                               double k_thresh) {
  if (nbins < 1 || !dp.satom || !dp.sRG) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(bins, 0, sizeof(double) * nbins, st);
  if (e != cudaSuccess) return e;
  const long long n = (long long)dp.nshell * dp.nshell;
  const int grid = (int)std::min<long long>((n + 255) / 256, 152 * 16);
  k_decay_bins<<<grid, 256, 0, st>>>(dp, Dsh, nbins, reinterpret_cast<unsigned long long *>(bins));
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_decay_fit<<<1, 256, 0, st>>>(reinterpret_cast<const unsigned long long *>(bins), nbins, HL);
  e = cudaGetLastError();
  if (e != cudaSuccess || !W) return e;
  const bool gdg = Gn && Dshf && T && GDG;
  if (gdg) {
    const int ns = dp.nshell;
    dim3 blk(16, 16), grd((ns + 31) / 32, (ns + 31) / 32);
    k_sgemm_nn<<<grd, blk, 0, st>>>(Gn, Dshf, T, ns, 0);    // T = A Dsh
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_sgemm_nn<<<grd, blk, 0, st>>>(T, Gn, GDG, ns, 1);     // GDG = T A^T
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  k_decay_w<<<grid, 256, 0, st>>>(dp, HL, gdg ? GDG : nullptr, (float)k_thresh, W);
  return cudaGetLastError();
}

// M <- M + M^T in place, for J (z = 0) and K (z = 1).
__global__ void k_symmetrize(double *J, double *K, int n) {
  double *M = (blockIdx.z == 0 && J) ? J : K;  // J or K may be absent (one z slice)
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= n || j >= n || i > j) return;
  if (i == j) {
    M[(size_t)i * n + i] *= 2.0;
  } else {
    const double s = M[(size_t)i * n + j] + M[(size_t)j * n + i];
    M[(size_t)i * n + j] = s;
    M[(size_t)j * n + i] = s;
  }
}

// --------------------------------------------------------------------------
// batched builds: one launch over every molecule (packed index spaces)
// --------------------------------------------------------------------------
__device__ __forceinline__ int find_mol(const long long *prefix, int nmol, long long idx) {
  int lo = 0, hi = nmol;  // prefix[lo] <= idx < prefix[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (prefix[mid] <= idx)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

__global__ void k_zero_batch(const MolEntry *__restrict__ mt, const long long *__restrict__ n2p, int nmol,
                             long long total) {
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const int m = find_mol(n2p, nmol, idx);
    const long long r = idx - n2p[m];
    mt[m].J[r] = 0.0;
    mt[m].K[r] = 0.0;
  }
}

__global__ void k_dprep_batch(const MolEntry *__restrict__ mt, const long long *__restrict__ dshp, int nmol,
                              long long total, const int *__restrict__ sbf, const int *__restrict__ sl,
                              double *__restrict__ Dsh, float *__restrict__ Dshf, unsigned *__restrict__ dmax) {
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const int m = find_mol(dshp, nmol, idx);
    const MolEntry &e = mt[m];
    const int r = (int)(idx - dshp[m]);
    const int a = e.s0 + r / e.ns, b = e.s0 + r % e.ns;
    const int fa = sbf[a], fb = sbf[b], na = ncart(sl[a]), nb = ncart(sl[b]);
    double mx = 0.0;
    bool bad = false;
    for (int i = 0; i < na; ++i)
      for (int j = 0; j < nb; ++j) {
        const size_t o = (size_t)(fa + i) * e.N + fb + j;
        const double v = e.D[o];
        if (e.Df) const_cast<float *>(e.Df)[o] = (float)v;
        if (!isfinite(v)) bad = true;
        mx = fmax(mx, fabs(v));
      }
    if (bad) atomicCAS(&g_status, 0, (int)FOCK_ERR_NONFINITE);
    Dsh[idx] = bad ? INFINITY : mx;
    Dshf[idx] = bad ? INFINITY : (float)mx;
    if (dmax) atomicMax(dmax + m, __float_as_uint(bad ? INFINITY : (float)mx));
  }
}

__global__ void k_symmetrize_batch(const MolEntry *__restrict__ mt, const long long *__restrict__ n2p, int nmol,
                                   long long total) {
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const int m = find_mol(n2p, nmol, idx);
    const MolEntry &e = mt[m];
    const int r = (int)(idx - n2p[m]);
    const int i = r / e.N, j = r % e.N;
    if (i > j) continue;
    for (int z = 0; z < 2; ++z) {
      double *M = z == 0 ? e.J : e.K;
      if (i == j) {
        M[(size_t)i * e.N + i] *= 2.0;
      } else {
        const double s = M[(size_t)i * e.N + j] + M[(size_t)j * e.N + i];
        M[(size_t)i * e.N + j] = s;
        M[(size_t)j * e.N + i] = s;
      }
    }
  }
}

cudaError_t launch_zero_batch(const MolEntry *mt, const long long *n2p, int nmol, long long total, cudaStream_t st) {
  k_zero_batch<<<grid_for(total), 256, 0, st>>>(mt, n2p, nmol, total);
  return cudaGetLastError();
}
cudaError_t launch_dprep_batch(const MolEntry *mt, const long long *dshp, int nmol, long long total, const int *sbf,
                               const int *sl, double *Dsh, float *Dshf, unsigned *dmax, cudaStream_t st) {
  k_dprep_batch<<<grid_for(total), 256, 0, st>>>(mt, dshp, nmol, total, sbf, sl, Dsh, Dshf, dmax);
  return cudaGetLastError();
}
cudaError_t launch_symmetrize_batch(const MolEntry *mt, const long long *n2p, int nmol, long long total,
                                    cudaStream_t st) {
  k_symmetrize_batch<<<grid_for(total), 256, 0, st>>>(mt, n2p, nmol, total);
  return cudaGetLastError();
}

// --------------------------------------------------------------------------
// host-side launch helpers
// --------------------------------------------------------------------------

cudaError_t upload_tables(cudaStream_t st) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (s_boys[dev] && s_tabs[dev] && s_boysf[dev] && s_boysff[dev]) return cudaSuccess;
  const std::vector<double> &bt = boys_table();
  const std::vector<float2> &bff = boys_table_ff();
  std::vector<float> btf(bt.begin(), bt.end());
  double *b = nullptr;
  float *bf = nullptr;
  float2 *b2 = nullptr;
  ClassTables *t = nullptr;
  e = cudaMalloc(&b, bt.size() * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&bf, btf.size() * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&b2, bff.size() * sizeof(float2));
  if (e == cudaSuccess) e = cudaMalloc(&t, sizeof(ClassTables));
  if (e == cudaSuccess) e = cudaMemcpyAsync(b, bt.data(), bt.size() * sizeof(double), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(bf, btf.data(), btf.size() * sizeof(float), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b2, bff.data(), bff.size() * sizeof(float2), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(t, &class_tables(), sizeof(ClassTables), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    cudaFree(b);
    cudaFree(bf);
    cudaFree(b2);
    cudaFree(t);
    return e;
  }
  s_boys[dev] = b;
  s_boysf[dev] = bf;
  s_boysff[dev] = b2;
  s_tabs[dev] = t;
  return cudaSuccess;
}

const double *dev_boys() {
  int dev = 0;
  cudaGetDevice(&dev);
  return s_boys[dev];
}
const float *dev_boys_f() {
  int dev = 0;
  cudaGetDevice(&dev);
  return s_boysf[dev];
}
const float2 *dev_boys_ff() {
  int dev = 0;
  cudaGetDevice(&dev);
  return s_boysff[dev];
}
const ClassTables *dev_class_tables() {
  int dev = 0;
  cudaGetDevice(&dev);
  return s_tabs[dev];
}

cudaError_t launch_dprep(const double *D, int nbf, const int *sbf, const int *sl, int nshell, double *Dsh,
                         cudaStream_t st, float *Df, float *Dshf, unsigned *dmax) {
  const int n = nshell * nshell;
  k_dprep<<<(n + 255) / 256, 256, 0, st>>>(D, nbf, sbf, sl, nshell, Dsh, Df, Dshf, dmax);
  return cudaGetLastError();
}

cudaError_t launch_split_e(const double *E, long long n, float2 *E2, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_split_e<<<grid_for(n), 256, 0, st>>>(E, n, E2);
  return cudaGetLastError();
}

cudaError_t launch_symmetrize(double *J, double *K, int n, cudaStream_t st) {
  const int nz = (J ? 1 : 0) + (K ? 1 : 0);
  if (nz == 0) return cudaSuccess;
  dim3 blk(32, 8), grd((n + 31) / 32, (n + 7) / 8, nz);
  k_symmetrize<<<grd, blk, 0, st>>>(J, K, n);
  return cudaGetLastError();
}

cudaError_t configure_tier(Tier &t, bool ff, bool mixed) {
  cudaError_t e = cudaSuccess;
  ff = ff && t.in_range;
  mixed = mixed && t.in_range;
  int dev = 0, nsm = 0, per_sm = 0, warps = 4;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  t.grp = t.g32 = GroupConfig{};
  auto blocks = [&](int lists) {  // every list has nunits units
    return std::min(nsm * std::max(per_sm, 1), std::max(1, (lists * t.nunits + warps - 1) / warps));
  };
  if (t.reg) {
    t.blocks_ff = 0;
    if (reg_merged(t.cb, t.ck)) {
      e = occupancy_reg(t.cb, t.ck, kRegAll, &warps, &per_sm);
      t.blocks = t.blocks_hi = blocks(2);
      return e;
    }
    e = occupancy_reg(t.cb, t.ck, kRegMain, &warps, &per_sm);
    t.blocks = blocks(1);
    // beside the two-float kernels an FP64 launch needs one warp per SM
    // sub-partition: an FP64 instruction occupies the pipe for 64 cycles, about
    // its latency
    t.blocks_hi = ff ? std::min(t.blocks, nsm) : t.blocks;
    if (e != cudaSuccess || !ff) return e;
    e = occupancy_reg(t.cb, t.ck, kRegFF, &warps, &per_sm);
    t.blocks_ff = blocks(1);
    return e;
  }
  e = configure_group(false, t.G, t.cb, t.ck, t.nunits, &t.grp);
  if (e != cudaSuccess || !mixed) return e;
  if (!t.r32) return configure_group(true, t.G, t.cb, t.ck, t.nunits, &t.g32);
  e = occupancy_reg32(t.cb, t.ck, &per_sm);
  t.blocks32 = blocks(1);
  return e;
}

static void set_screen_args(KArgs &a, double tau, const float *Dshf, double prim_eps,
                            const CallParts &cp = CallParts()) {
  a.parts = cp.parts;
  a.Wsh = cp.Wsh;
  a.k_thresh_f = (float)cp.k_thresh;
  a.Dshf = Dshf;
  a.tau_lo = (float)(tau * (1.0 - 1e-4));
  a.tau_hi = (float)(tau * (1.0 + 1e-4));
  a.tau_eps = prim_eps > 0.0 ? tau * prim_eps : 0.0;
  a.tau_eps_f = (float)a.tau_eps;
}

// Streams of the index-th tier: a separate FP64 launch that fills the chip (wide)
// or not, the other launches.
constexpr int kWide = 2;
static int hi_stream(int index, bool wide) { return wide ? index % kWide : kWide + index % (kHiStreams - kWide); }
static int lo_stream(int index, bool queued) { return kHiStreams + (queued ? 0 : index % kLoStreams); }
unsigned tier_streams(int index) {
  return 1u << hi_stream(index, true) | 1u << hi_stream(index, false) | 1u << lo_stream(index, false) | 1u << lo_stream(index, true);
}

// Launches of one tier: the kernel of all its lists, or one for FP64 (and FP32)
// and one for two floats; a group tier's FP32 list in mixed builds.  With a
// stream set they go to its streams.  A launch of FP64 alone then leaves room on
// every SM for the others, and those with work for every SM share two streams:
// two of them keep the FP64 pipe busy, more would only take registers from the
// two-float kernels.
static cudaError_t launch_tier(const Tier &t, KArgs &a, int *counters, cudaStream_t st, StreamSet *par, int index) {
  a.boys = dev_boys();
  a.boysf = dev_boys_f();
  a.boysff = dev_boys_ff();
  a.tabs = dev_class_tables();
  a.units = t.d_units;
  a.nunits = t.nunits;
  a.nsplit = t.nsplit;
  a.cb = t.cb;
  a.ck = t.ck;
  a.counters = counters;
  const bool mixed = a.fp32_cutoff > 0.0;
  const cudaStream_t lo = par ? par->s[lo_stream(index, t.queued)] : st;
  if (t.reg) {
    if (reg_merged(t.cb, t.ck)) return launch_reg(t.cb, t.ck, kRegAll, a, t.blocks, lo);
    const bool hi_only = par && a.dmax && !mixed;
    const cudaStream_t hi = hi_only ? par->s[hi_stream(index, t.blocks > t.blocks_hi)] : lo;
    cudaError_t e = launch_reg(t.cb, t.ck, kRegMain, a, hi_only ? t.blocks_hi : t.blocks, hi);
    if (e != cudaSuccess || !a.dmax) return e;
    return launch_reg(t.cb, t.ck, kRegFF, a, t.blocks_ff, lo);
  }
  cudaError_t e = launch_group(false, t.grp, a, lo);
  if (e != cudaSuccess || !mixed) return e;
  return t.r32 ? launch_reg32(t.cb, t.ck, a, t.blocks32, lo) : launch_group(true, t.g32, a, lo);
}

cudaError_t launch_jk_tier(const Tier &t, const DevPairs &dp, const double *D, const double *Dsh, double tau,
                           double prim_eps, double *J, double *K, int *counters, cudaStream_t st, StreamSet *par,
                           int index, const float *Df, double fp32_cutoff, const float *Dshf, const CallParts &cp) {
  if (t.nunits == 0) return cudaSuccess;
  KArgs a;
  memset(&a, 0, sizeof(a));
  a.dp = dp;
  a.nprimtot = dp.nprim_total;
  a.nEtot = dp.nE_total;
  a.D = D;
  a.Dsh = Dsh;
  a.tau = tau;
  a.J = J;
  a.K = K;
  a.fp32_cutoff = Df && t.in_range ? fp32_cutoff : 0.0;
  a.fp32_cutoff_f = (float)a.fp32_cutoff;
  a.Df = Df;
  a.dmax = dp.E2 && t.in_range ? cp.dmax : nullptr;
  a.gmax2 = cp.gmax2;
  set_screen_args(a, tau, Dshf, prim_eps, cp);
  return launch_tier(t, a, counters, st, par, index);
}

// One tier of a batched build: same kernels, per-molecule D/J/K from mt.
cudaError_t launch_jk_tier_batch(const Tier &t, const DevPairs &dp, const MolEntry *mt, const double *Dsh,
                                 const float *Dshf, const unsigned *dmax, double tau, double prim_eps,
                                 int *counters, cudaStream_t st, StreamSet *par, int index, double fp32_cutoff) {
  if (t.nunits == 0) return cudaSuccess;
  KArgs a;
  memset(&a, 0, sizeof(a));
  a.dp = dp;
  a.nprimtot = dp.nprim_total;
  a.nEtot = dp.nE_total;
  a.Dsh = Dsh;
  a.tau = tau;
  a.mt = mt;
  a.fp32_cutoff = t.in_range ? fp32_cutoff : 0.0;
  a.fp32_cutoff_f = (float)a.fp32_cutoff;
  a.dmax = dp.E2 && t.in_range ? dmax : nullptr;
  set_screen_args(a, tau, Dshf, prim_eps);
  return launch_tier(t, a, counters, st, par, index);
}

int read_and_clear_status(cudaStream_t st, int *status) {
  cudaError_t e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return (int)e;
  int v = 0, zero = 0;
  e = cudaMemcpyFromSymbol(&v, g_status, sizeof(int));
  if (e != cudaSuccess) return (int)e;
  e = cudaMemcpyToSymbol(g_status, &zero, sizeof(int));
  if (e != cudaSuccess) return (int)e;
  *status = v;
  return 0;
}

}  // namespace fk
