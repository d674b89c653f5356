// Schwarz factors from diagonal integrals (Eqs. cauchy-schwarz 1, 2):
// G_ab = sqrt(max_kc sum_ij [kc_i|kc_j]) over the Cartesian pairs kc of a shell
// pair, G_[ab] = sqrt(max_kc [kc_i|kc_i]) for each of its primitive pairs, with
// [kc_i|kc_j] = sum_p E^i_p sum_q (-1)^{|q|} E^j_q R_{p+q}.
//
// A row of a pair -- primitive pair i with the primitive pairs j >= i, the ones
// after it twice -- is one item of work: one thread with everything in
// registers for the classes up to la + lb = 2, one warp with the Hermite
// integrals in shared memory for the others.  The rows' sums are added up in
// order by a last kernel.  The rows make the parallel work: 0.65 ms for C12H26.
// One warp per pair that walks all n^2 primitive quartets of a contracted pair (up
// to 4096) takes the longest pair's latency instead: 3.1 ms, 7 ms for a
// triple-zeta ethane.
#include <algorithm>

#include "kernels_reg.cuh"

namespace fk {

namespace {

struct SchwarzArgs {
  DevPairs dp;
  const double *boys;
  const ClassTables *tabs;
  const int2 *rows;  // (pair, primitive pair of it) of this class
  int nrows;
  double *part;      // [Cartesian pair][row]
  double *Gprim;
};

template <int LA, int LB>
__global__ void __launch_bounds__(128) k_schwarz_thread(SchwarzArgs a) {
  constexpr int NB = ncart(LB), NAB = ncart(LA) * NB, L = 2 * (LA + LB), NHL = nherm(L);
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= a.nrows) return;
  const DevPairs &dp = a.dp;
  const int2 row = a.rows[r];
  const int2 pr = dp.prim[row.x];
  const int i = pr.x + row.y;
  const PZ P4 = dp.pz[i];
  const float4 Pf = dp.pf[i];
  double acc[NAB], diag = 0.0;
  sfor<NAB>([&](auto k) { acc[FK_CI(k)] = 0.0; });
  for (int j = i; j < pr.x + pr.y; ++j) {
    const PrimQuartet q = prim_quartet(P4, Pf, dp.pz[j], dp.pf[j]);
    double F[L + 1];
    boys_seeds<L>(a.boys, q, F);
    double R[NHL];
    hermite_r_reg<L, double>(F, q.X, q.Y, q.Z, R);
    sfor<NAB>([&](auto kk) {
      constexpr int kc = FK_CI(kk);
      constexpr TUV x = ct_cart(LA, kc / NB), y = ct_cart(LB, kc % NB);
      constexpr int TY = x.u + y.u + 1, TZ = x.v + y.v + 1, N = (x.t + y.t + 1) * TY * TZ;
      constexpr int e0 = ct_eoff(LA, LB, kc);
      double v = 0.0;
      sfor<N>([&](auto pp) {
        constexpr int p = FK_CI(pp);
        double inner = 0.0;
        sfor<N>([&](auto qq) {
          constexpr int s = FK_CI(qq);
          constexpr int t2 = s / (TY * TZ), u2 = (s / TZ) % TY, v2 = s % TZ;
          const double e = __ldg(dp.E + dp.eoff[j] + e0 + s);
          inner = fma(r_neg_if<((t2 + u2 + v2) & 1) != 0>(e),
                      R[ct_hidx(p / (TY * TZ) + t2, (p / TZ) % TY + u2, p % TZ + v2)], inner);
        });
        v = fma(__ldg(dp.E + dp.eoff[i] + e0 + p), inner, v);
      });
      if (j == i)
        diag = fmax(diag, fabs(v));
      else
        v *= 2.0;
      acc[kc] += v;
    });
  }
  sfor<NAB>([&](auto k) { a.part[(size_t)FK_CI(k) * a.nrows + r] = acc[FK_CI(k)]; });
  a.Gprim[i] = sqrt(diag);
}

static_assert(sizeof(ClassTables) % 16 == 0, "the scratch behind the tables is aligned");

// R^{(0)}_{tuv}, t+u+v <= L, into the returned buffer (one of R0/R1), by one warp.
// F must hold base values pref (-2alpha)^n F_n(T), n = 0..L; R0[0] = F[L].
__constant__ double c_small[16] = {0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15};
__device__ __forceinline__ double *hermite_r_warp(const ClassTables &ct, int L, double X, double Y, double Z,
                                                  const double *F, double *R0, double *R1, int lane) {
  double *cur = R0, *nxt = R1;
  for (int n = L - 1; n >= 0; --n) {
    const int cnt = nherm(L - n);
    for (int e = lane; e < cnt; e += 32) {
      double v;
      if (e == 0) {
        v = F[n];
      } else {
        const int t = ct.hvec[e][0], u = ct.hvec[e][1], w = ct.hvec[e][2];
        if (t > 0) {
          v = X * cur[hidx(t - 1, u, w)];
          if (t > 1) v = fma(c_small[t - 1], cur[hidx(t - 2, u, w)], v);
        } else if (u > 0) {
          v = Y * cur[hidx(t, u - 1, w)];
          if (u > 1) v = fma(c_small[u - 1], cur[hidx(t, u - 2, w)], v);
        } else {
          v = Z * cur[hidx(t, u, w - 1)];
          if (w > 1) v = fma(c_small[w - 1], cur[hidx(t, u, w - 2)], v);
        }
      }
      nxt[e] = v;
    }
    __syncwarp();
    double *tmp = cur;
    cur = nxt;
    nxt = tmp;
  }
  return cur;
}

// One warp per row, lanes over the Cartesian pairs.
__global__ void __launch_bounds__(128) k_schwarz_warp(SchwarzArgs a, int la, int lb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  {
    const int *src = reinterpret_cast<const int *>(a.tabs);
    int *dst = reinterpret_cast<int *>(smem_raw);
    for (int i = threadIdx.x; i < (int)(sizeof(ClassTables) / 4); i += blockDim.x) dst[i] = src[i];
  }
  __syncthreads();
  const ClassTables &ct = *reinterpret_cast<const ClassTables *>(smem_raw);
  const DevPairs &dp = a.dp;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double *scr = reinterpret_cast<double *>(smem_raw + sizeof(ClassTables)) + warp * (2 * NHMAX + LTOT + 2);
  double *R0 = scr, *R1 = scr + NHMAX, *F = scr + 2 * NHMAX;
  const int nb = ncart(lb), nab = ncart(la) * nb, L = 2 * (la + lb), c = pair_class(la, lb);
  const int r = blockIdx.x * (blockDim.x >> 5) + warp;
  if (r >= a.nrows) return;
  const int2 row = a.rows[r];
  const int2 pr = dp.prim[row.x];
  const int i = pr.x + row.y;
  const PZ P4 = dp.pz[i];
  const float4 Pf = dp.pf[i];
  double acc[4] = {0.0, 0.0, 0.0, 0.0}, pm = 0.0;
  for (int j = i; j < pr.x + pr.y; ++j) {
    const PrimQuartet q = prim_quartet(P4, Pf, dp.pz[j], dp.pf[j]);
    boys_seeds_warp(a.boys, q, L, F, R0, lane);
    __syncwarp();
    const double *R = hermite_r_warp(ct, L, q.X, q.Y, q.Z, F, R0, R1, lane);
    for (int k = 0; k < 4; ++k) {
      const int kc = lane + 32 * k;
      if (kc >= nab) break;
      const uint8_t *x = ct.comp[la][kc / nb], *y = ct.comp[lb][kc % nb];
      const int Tx = x[0] + y[0], Ty = x[1] + y[1], Tz = x[2] + y[2];
      const double *Ei = dp.E + dp.eoff[i] + ct.eoff[c][kc];
      const double *Ej = dp.E + dp.eoff[j] + ct.eoff[c][kc];
      double v = 0.0;
      int e1 = 0;
      for (int t1 = 0; t1 <= Tx; ++t1)
        for (int u1 = 0; u1 <= Ty; ++u1)
          for (int v1 = 0; v1 <= Tz; ++v1, ++e1) {
            double inner = 0.0;
            int e2 = 0;
            for (int t2 = 0; t2 <= Tx; ++t2)
              for (int u2 = 0; u2 <= Ty; ++u2)
                for (int v2 = 0; v2 <= Tz; ++v2, ++e2) {
                  const double rr = R[hidx(t1 + t2, u1 + u2, v1 + v2)];
                  inner = ((t2 + u2 + v2) & 1) ? fma(-Ej[e2], rr, inner) : fma(Ej[e2], rr, inner);
                }
            v = fma(Ei[e1], inner, v);
          }
      if (j == i)
        pm = fmax(pm, fabs(v));
      else
        v *= 2.0;
      acc[k] += v;
    }
    __syncwarp();
  }
  for (int k = 0; k < 4; ++k)
    if (lane + 32 * k < nab) a.part[(size_t)(lane + 32 * k) * a.nrows + r] = acc[k];
  for (int o = 16; o > 0; o >>= 1) pm = fmax(pm, __shfl_xor_sync(0xffffffffu, pm, o));
  if (lane == 0) a.Gprim[i] = sqrt(pm);
}

// Thread per first row of a pair: adds the pair's rows and takes the maximum.
__global__ void k_schwarz_sum(SchwarzArgs a, int nab, double *Gpair) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= a.nrows) return;
  const int2 row = a.rows[r];
  if (row.y != 0) return;
  const int n = a.dp.prim[row.x].y;
  double mx = 0.0;
  for (int k = 0; k < nab; ++k) {
    double s = 0.0;
    for (int i = 0; i < n; ++i) s += a.part[(size_t)k * a.nrows + r + i];
    mx = fmax(mx, s);
  }
  Gpair[row.x] = sqrt(mx);
}

template <int LA, int LB>
void launch_thread(const SchwarzArgs &a, cudaStream_t st) {
  k_schwarz_thread<LA, LB><<<(a.nrows + 127) / 128, 128, 0, st>>>(a);
}

}  // namespace

// rows: the rows of all pairs, class after class (nrows[class] of them, the
// rows of a pair consecutive); part: scratch of schwarz_part doubles.
cudaError_t launch_schwarz(const DevPairs &dp, const int2 *rows, const int *nrows, double *part, double *Gpair,
                           double *Gprim, cudaStream_t st) {
  const size_t smem = sizeof(ClassTables) + 4 * (2 * NHMAX + LTOT + 2) * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(k_schwarz_warp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  for (int la = 0; la <= LMAX; ++la)
    for (int lb = 0; lb <= la; ++lb) {
      const int c = pair_class(la, lb), n = nrows[c], nab = ncart(la) * ncart(lb);
      if (n == 0) continue;
      const SchwarzArgs a{dp, dev_boys(), dev_class_tables(), rows, n, part, Gprim};
      switch (c) {
        case 0: launch_thread<0, 0>(a, st); break;
        case 1: launch_thread<1, 0>(a, st); break;
        case 2: launch_thread<1, 1>(a, st); break;
        case 3: launch_thread<2, 0>(a, st); break;
        default: k_schwarz_warp<<<(n + 3) / 4, 128, smem, st>>>(a, la, lb);
      }
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      k_schwarz_sum<<<(n + 127) / 128, 128, 0, st>>>(a, nab, Gpair);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      rows += n;
      part += (size_t)n * nab;
    }
  return cudaSuccess;
}

}  // namespace fk
