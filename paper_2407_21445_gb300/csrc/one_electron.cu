// FP64 one-electron integrals over the same normalised Cartesian basis:
// overlap S, kinetic T and nuclear attraction V (the core Hamiltonian
// h = T + V of Sec. 2.2, Eq. fock_build), by the McMurchie-Davidson Hermite
// expansion (Sec. 4.1, Eqs. EabP def1-3):
//   S_ab = sum_prims U_P E^{ab}_{000}
//   T_ab = -1/2 sum_x [4 b^2 S_x(a, b+2) - 2b(2 b_x + 1) S_x(a, b) + b_x(b_x - 1) S_x(a, b-2)] S_y S_z
//   V_ab = -sum_C Z_C sum_prims U_P 2 sqrt(zeta/pi) sum_tuv E^{ab}_tuv R_tuv(zeta, P - C)
// with U_P = c_a c_b (pi/zeta)^{3/2} exp(-a b |AB|^2 / zeta) and R seeded by
// (-2 zeta)^n F_n(zeta |P - C|^2).
//
// Work decomposition: one thread per primitive pair of a shell pair (a, b) with
// la >= lb (a >= b when equal).  It sums Z_C R_tuv over the nuclei once in
// registers and contracts the sum with the Hermite coefficients of every
// Cartesian pair; a second kernel adds up the primitive pairs of each element in
// a fixed order and writes both triangles.  The nuclei are the inner loop and
// carry nearly all the work, about 16 (ss) to 250 (dd) FP64 operations each, so
// the kernel is bound by the FP64 pipe: 2.4 ms for (H2O)32 (608 functions, 96
// nuclei; call included), 1.2 ms of it the pipe's by the operation model.  A thread
// per Cartesian pair and order instead repeats the Boys function and the
// recursion up to 72 times (165 ms).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <array>
#include <vector>

#include "kernels_reg.cuh"

namespace fk {
fock_status validate_basis(const fock_basis_desc *d);
void normalised_coefs(const fock_basis_desc *d, int s, double *out);

namespace {

// Workspace of the per-primitive values: a class that needs more is done in
// pieces of whole shell pairs, a million threads each at least for s and p;
// where the device has not that much left, in smaller ones down to 64 KiB.
constexpr long long kPieceDoubles = 64ll << 20, kMinPieceDoubles = 8ll << 10;  // 512 MiB

// Shells of one kind, at perm[first ..].
struct ShellGroup {
  int first, count, l, np;
};
// Pairs of two kinds: shell pairs and primitive pairs before this entry, and
// whether the kinds are the same (then only a >= b).
struct GroupPair {
  int ga, gb, same, npp;
  long long pair0, prim0;
};

struct OneArgs {
  int nbf, natom, nsplit, ngp;
  long long pair_lo, npair, prim_lo, nprim;  // of this class, in this launch
  const ShellGroup *groups;
  const GroupPair *gp;    // pairs of kinds of this class
  const int *perm, *po, *bf;
  const double *xyz, *ex, *cc;
  const double *axyz, *Z;
  const double *boys;
  double *buf;            // [nsplit + 2][ncart pairs][nprim]: S, T, V of each split
  double *S, *T, *V;
};

// k-th pair of n shells with a >= b, or of na x nb
__device__ __forceinline__ void pair_of(const GroupPair &g, const ShellGroup &A, const ShellGroup &B, long long k, int &a,
                                        int &b) {
  if (g.same) {
    a = (int)((sqrtf(8.0f * (float)k + 1.0f) - 1.0f) * 0.5f);
    while ((long long)a * (a + 1) / 2 > k) --a;
    while ((long long)(a + 1) * (a + 2) / 2 <= k) ++a;
    b = (int)(k - (long long)a * (a + 1) / 2);
  } else {
    a = (int)(k / B.count);
    b = (int)(k - (long long)a * B.count);
  }
}

// last entry whose first index (pair or primitive) is <= i
template <class F>
__device__ __forceinline__ int find_gp(int n, long long i, F &&first) {
  int k = 0;
  while (k + 1 < n && first(k + 1) <= i) ++k;
  return k;
}

__host__ __device__ constexpr double ct_dfact(int n) { return n <= 1 ? 1.0 : n * ct_dfact(n - 2); }
// product of (2k-1)!! over the directions of a Cartesian component: the squared norm ratio
__host__ __device__ constexpr double ct_norm2(TUV c) {
  return ct_dfact(2 * c.t - 1) * ct_dfact(2 * c.u - 1) * ct_dfact(2 * c.v - 1);
}

// Hermite coefficients of one direction: E[i][j][t], i <= LA, j <= LB, and the
// overlaps S[i][j] = E^{ij}_0 up to j = LB + 2.
template <int LA, int LB>
struct Herm1 {
  double E[LA + 1][LB + 1][LA + LB + 1];
  double S[LA + 1][LB + 3];
};
template <int LA, int LB>
__device__ __forceinline__ void herm1(double h, double xpa, double xpb, Herm1<LA, LB> &o) {
  double e[LA + 1][LB + 3][LA + LB + 3];
  sfor<LA + 1>([&](auto ii) {
    constexpr int i = FK_CI(ii);
    sfor<LB + 3>([&](auto jj) {
      constexpr int j = FK_CI(jj);
      sfor<LA + LB + 3>([&](auto tt) {
        constexpr int t = FK_CI(tt);
        if constexpr (i == 0 && j == 0) {
          e[0][0][t] = t == 0 ? 1.0 : 0.0;
        } else if constexpr (t <= i + j) {
          constexpr int pi = j > 0 ? i : i - 1, pj = j > 0 ? j - 1 : 0;
          const double x = j > 0 ? xpb : xpa;
          double v = 0.0;
          if constexpr (t <= pi + pj) v = x * e[pi][pj][t];
          if constexpr (t > 0) v = fma(h, e[pi][pj][t - 1], v);
          if constexpr (t + 1 <= pi + pj) v = fma((double)(t + 1), e[pi][pj][t + 1], v);
          e[i][j][t] = v;
        } else {
          e[i][j][t] = 0.0;
        }
      });
      o.S[i][j] = e[i][j][0];
      if constexpr (j <= LB) sfor<LA + LB + 1>([&](auto tt) { o.E[i][j][FK_CI(tt)] = e[i][j][FK_CI(tt)]; });
    });
  });
}

template <int LA, int LB>
__global__ void __launch_bounds__(128) k_one_prims(OneArgs a) {
  constexpr int L = LA + LB, NH = nherm(L), NB = ncart(LB), NAB = ncart(LA) * NB;
  const long long item = blockIdx.x * (long long)blockDim.x + threadIdx.x, pp = a.prim_lo + item;
  if (item >= a.nprim) return;
  const GroupPair g = a.gp[find_gp(a.ngp, pp, [&](int k) { return a.gp[k].prim0; })];
  const ShellGroup ga = a.groups[g.ga], gb = a.groups[g.gb];
  const long long k = (pp - g.prim0) / g.npp;
  const int ij = (int)(pp - g.prim0 - k * g.npp), i = ij / gb.np, j = ij - i * gb.np;
  int ia, ib;
  pair_of(g, ga, gb, k, ia, ib);
  const int sa = a.perm[ga.first + ia], sb = a.perm[gb.first + ib];
  const double *A = a.xyz + 3 * sa, *B = a.xyz + 3 * sb;
  const double al = a.ex[a.po[sa] + i], be = a.ex[a.po[sb] + j], p = al + be;
  const double ABx = A[0] - B[0], ABy = A[1] - B[1], ABz = A[2] - B[2];
  const double U = a.cc[a.po[sa] + i] * a.cc[a.po[sb] + j] * pow(3.141592653589793 / p, 1.5) *
                   exp(-al * be / p * (ABx * ABx + ABy * ABy + ABz * ABz));
  const double Px = (al * A[0] + be * B[0]) / p, Py = (al * A[1] + be * B[1]) / p, Pz = (al * A[2] + be * B[2]) / p;
  Herm1<LA, LB> hx, hy, hz;
  const double h = 0.5 / p;
  herm1<LA, LB>(h, Px - A[0], Px - B[0], hx);
  herm1<LA, LB>(h, Py - A[1], Py - B[1], hy);
  herm1<LA, LB>(h, Pz - A[2], Pz - B[2], hz);
  auto put = [&](int m, int kc, double v) { a.buf[((long long)m * NAB + kc) * a.nprim + item] = v; };
  if (blockIdx.y == 0) {
    sfor<NAB>([&](auto kk) {
      constexpr int kc = FK_CI(kk);
      constexpr TUV x = ct_cart(LA, kc / NB), y = ct_cart(LB, kc % NB);
      constexpr double f2 = 1.0 / (ct_norm2(x) * ct_norm2(y));
      const double f = U * sqrt(f2);
      const double sx = hx.S[x.t][y.t], sy = hy.S[x.u][y.u], sz = hz.S[x.v][y.v];
      // per direction -1/2 <a| d^2/dx^2 |b>
      auto kin = [&](const Herm1<LA, LB> &H, auto bi, auto bj) -> double {
        constexpr int ii = FK_CI(bi), jj = FK_CI(bj);
        double d = 4.0 * be * be * H.S[ii][jj + 2] - 2.0 * be * (2 * jj + 1) * H.S[ii][jj];
        if constexpr (jj >= 2) d += jj * (jj - 1) * H.S[ii][jj - 2];
        return -0.5 * d;
      };
#define FK_N(v) std::integral_constant<int, (v)>{}
      const double t = kin(hx, FK_N(x.t), FK_N(y.t)) * (sy * sz) + kin(hy, FK_N(x.u), FK_N(y.u)) * (sx * sz) +
                       kin(hz, FK_N(x.v), FK_N(y.v)) * (sx * sy);
#undef FK_N
      put(0, kc, f * sx * sy * sz);
      put(1, kc, f * t);
    });
  }
  // sum over this share's nuclei of Z R_tuv(zeta, P - C)
  double W[NH];
  sfor<NH>([&](auto e) { W[FK_CI(e)] = 0.0; });
  const int c0 = (int)((long long)a.natom * blockIdx.y / a.nsplit), c1 = (int)((long long)a.natom * (blockIdx.y + 1) / a.nsplit);
  const double m2p = -2.0 * p;
  for (int c = c0; c < c1; ++c) {
    const double X = Px - a.axyz[3 * c], Y = Py - a.axyz[3 * c + 1], Z = Pz - a.axyz[3 * c + 2];
    const double T = p * fma(X, X, fma(Y, Y, Z * Z));
    double F[L + 1];
    // decisions on the integer units, by the high word of T: T < 64 reads the
    // table, T < 2^127 has an FP32 seed for the square root
    const unsigned th = (unsigned)__double2hiint(T) & 0x7fffffffu;
    if (th < 0x40500000u) {
      const int gi = __float2int_rn(d2f_small(T) * (float)BOYS_INVH);
      const double x = (gi == 0 ? 0.0 : f2d_pos((float)gi * (float)BOYS_H)) - T;
      sfor<L + 1>([&](auto m) { F[FK_CI(m)] = boys_taylor(a.boys, gi, FK_CI(m), x); });
    } else {
      const double rt = th < 0x47e00000u ? rsqrt_nh(T, d2f_small(T)) : rsqrt(T), it = rt * rt;
      F[0] = 0.88622692545275801365 * rt;
      sfor<L>([&](auto m) { F[FK_CI(m) + 1] = F[FK_CI(m)] * ((FK_CI(m) + 0.5) * it); });
    }
    double s = a.Z[c];
    sfor<L + 1>([&](auto m) {
      F[FK_CI(m)] *= s;
      s *= m2p;
    });
    double R[NH];
    hermite_r_reg<L, double>(F, X, Y, Z, R);
    sfor<NH>([&](auto e) { W[FK_CI(e)] += R[FK_CI(e)]; });
  }
  const double pref = -U * 2.0 * sqrt(p / 3.141592653589793);
  sfor<NAB>([&](auto kk) {
    constexpr int kc = FK_CI(kk);
    constexpr TUV x = ct_cart(LA, kc / NB), y = ct_cart(LB, kc % NB);
    constexpr double f2 = 1.0 / (ct_norm2(x) * ct_norm2(y));
    double acc = 0.0;
    sfor<x.t + y.t + 1>([&](auto tt) {
      double at = 0.0;
      sfor<x.u + y.u + 1>([&](auto uu) {
        double au = 0.0;
        sfor<x.v + y.v + 1>([&](auto vv) {
          au = fma(hz.E[x.v][y.v][FK_CI(vv)], W[ct_hidx(FK_CI(tt), FK_CI(uu), FK_CI(vv))], au);
        });
        at = fma(hy.E[x.u][y.u][FK_CI(uu)], au, at);
      });
      acc = fma(hx.E[x.t][y.t][FK_CI(tt)], at, acc);
    });
    put(2 + blockIdx.y, kc, pref * sqrt(f2) * acc);
  });
}

// Sums the primitive pairs (and the nuclei's shares) of every element.
template <int LA, int LB>
__global__ void __launch_bounds__(128) k_one_sum(OneArgs a) {
  constexpr int NB = ncart(LB), NAB = ncart(LA) * NB;
  const long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (id >= a.npair * NAB) return;
  const long long pair = a.pair_lo + id / NAB;
  const int kc = (int)(id % NAB);
  const GroupPair g = a.gp[find_gp(a.ngp, pair, [&](int k) { return a.gp[k].pair0; })];
  const ShellGroup ga = a.groups[g.ga], gb = a.groups[g.gb];
  int ia, ib;
  pair_of(g, ga, gb, pair - g.pair0, ia, ib);
  const int sa = a.perm[ga.first + ia], sb = a.perm[gb.first + ib];
  const long long p0 = g.prim0 + (pair - g.pair0) * g.npp - a.prim_lo;
  double s = 0.0, t = 0.0, v = 0.0;
  for (int i = 0; i < g.npp; ++i) {
    s += a.buf[(long long)kc * a.nprim + p0 + i];
    t += a.buf[((long long)NAB + kc) * a.nprim + p0 + i];
    for (int y = 0; y < a.nsplit; ++y) v += a.buf[((long long)(2 + y) * NAB + kc) * a.nprim + p0 + i];
  }
  const size_t r = a.bf[sa] + kc / NB, c = a.bf[sb] + kc % NB;
  a.S[r * a.nbf + c] = a.S[c * a.nbf + r] = s;
  a.T[r * a.nbf + c] = a.T[c * a.nbf + r] = t;
  a.V[r * a.nbf + c] = a.V[c * a.nbf + r] = v;
}

template <int LA, int LB>
cudaError_t launch_class(const OneArgs &a, cudaStream_t st) {
  k_one_prims<LA, LB><<<dim3((unsigned)((a.nprim + 127) / 128), a.nsplit), 128, 0, st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const long long n = a.npair * ncart(LA) * ncart(LB);
  k_one_sum<LA, LB><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_class(int la, int lb, const OneArgs &a, cudaStream_t st) {
  switch (pair_class(la, lb)) {
    case 0: return launch_class<0, 0>(a, st);
    case 1: return launch_class<1, 0>(a, st);
    case 2: return launch_class<1, 1>(a, st);
    case 3: return launch_class<2, 0>(a, st);
    case 4: return launch_class<2, 1>(a, st);
    case 5: return launch_class<2, 2>(a, st);
    case 6: return launch_class<3, 0>(a, st);
    case 7: return launch_class<3, 1>(a, st);
    case 8: return launch_class<3, 2>(a, st);
    case 9: return launch_class<3, 3>(a, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace
}  // namespace fk

using namespace fk;

extern "C" fock_status fock_one_electron(const fock_basis_desc *desc, int32_t natom, const double *Z,
                                         const double *xyz, double *S, double *T, double *V, cudaStream_t stream) {
  fock_status vs = validate_basis(desc);
  if (vs != FOCK_OK) return vs;
  if (natom < 0 || (natom > 0 && (!Z || !xyz)) || !S || !T || !V) return FOCK_ERR_INVALID_ARG;
  cudaError_t e = upload_tables(stream);
  if (e != cudaSuccess) return FOCK_ERR_CUDA;
  const int ns = desc->nshell;
  int np_tot = 0, nbf = 0;
  std::vector<int> bf(ns), po(ns), perm(ns);
  std::vector<std::vector<int>> kind((LMAX + 1) * (MAXPRIM + 1));
  for (int s = 0; s < ns; ++s) {
    bf[s] = nbf;
    nbf += ncart(desc->l[s]);
    po[s] = np_tot;
    np_tot += desc->nprim[s];
    kind[desc->l[s] * (MAXPRIM + 1) + desc->nprim[s]].push_back(s);
  }
  std::vector<ShellGroup> groups;
  int at = 0;
  for (int l = 0; l <= LMAX; ++l)
    for (int np = 1; np <= MAXPRIM; ++np) {
      const std::vector<int> &k = kind[l * (MAXPRIM + 1) + np];
      if (k.empty()) continue;
      groups.push_back(ShellGroup{at, (int)k.size(), l, np});
      for (int s : k) perm[at++] = s;
    }
  // pairs of kinds, by class
  struct ClassWork {
    int la, lb, gp0, ngp, nsplit;
    long long npair, nprim;
  };
  std::vector<GroupPair> gps;
  std::vector<ClassWork> work;
  long long piece = kPieceDoubles;
  // primitive pairs of a class whose values the workspace holds at a time
  auto piece_prims = [&piece](const ClassWork &w) {
    return std::max<long long>(MAXPRIM * MAXPRIM, piece / ((w.nsplit + 2) * ncart(w.la) * ncart(w.lb)));
  };
  for (int la = 0; la <= LMAX; ++la)
    for (int lb = 0; lb <= la; ++lb) {
      ClassWork w{la, lb, (int)gps.size(), 0, 1, 0, 0};
      for (int x = 0; x < (int)groups.size(); ++x)
        for (int y = 0; y < (int)groups.size(); ++y) {
          const ShellGroup &A = groups[x], &B = groups[y];
          if (A.l != la || B.l != lb || (la == lb && x < y)) continue;
          gps.push_back(GroupPair{x, y, x == y, A.np * B.np, w.npair, w.nprim});
          const long long n = x == y ? (long long)A.count * (A.count + 1) / 2 : (long long)A.count * B.count;
          w.npair += n;
          w.nprim += n * A.np * B.np;
          ++w.ngp;
        }
      if (w.npair == 0) continue;
      // few primitive pairs: share the nuclei, too, between up to 8 threads
      while (w.nsplit < 8 && 2 * w.nsplit <= natom && w.nprim * w.nsplit < kFillThreads) w.nsplit *= 2;
      work.push_back(w);
    }
  std::vector<double> ex(np_tot), cc(np_tot);
  for (int s = 0; s < ns; ++s) {
    normalised_coefs(desc, s, cc.data() + po[s]);
    for (int i = 0; i < desc->nprim[s]; ++i) ex[po[s] + i] = desc->exps[desc->prim_off[s] + i];
  }
  // one device block: the inputs, then the per-primitive values of one class
  std::vector<char> host;
  auto add = [&host](const void *p, size_t bytes) {
    const size_t o = (host.size() + 15) & ~(size_t)15;
    host.resize(o + bytes);
    if (bytes) memcpy(host.data() + o, p, bytes);
    return o;
  };
  const size_t o_g = add(groups.data(), groups.size() * sizeof(ShellGroup));
  const size_t o_gp = add(gps.data(), gps.size() * sizeof(GroupPair));
  const size_t o_perm = add(perm.data(), sizeof(int) * ns), o_po = add(po.data(), sizeof(int) * ns);
  const size_t o_bf = add(bf.data(), sizeof(int) * ns);
  const size_t o_xyz = add(desc->center, sizeof(double) * 3 * ns);
  const size_t o_ex = add(ex.data(), sizeof(double) * np_tot), o_cc = add(cc.data(), sizeof(double) * np_tot);
  const size_t o_a = add(xyz, natom > 0 ? sizeof(double) * 3 * natom : 0);
  const size_t o_z = add(Z, natom > 0 ? sizeof(double) * natom : 0);
  const size_t in_bytes = (host.size() + 255) & ~(size_t)255;
  char *d = nullptr;
  for (;; piece /= 8) {
    size_t buf_doubles = 0;
    for (const ClassWork &w : work)
      buf_doubles = std::max(buf_doubles, (size_t)((w.nsplit + 2) * ncart(w.la) * ncart(w.lb) *
                                                   std::min(w.nprim, piece_prims(w))));
    e = cudaMallocAsync((void **)&d, in_bytes + buf_doubles * sizeof(double), stream);
    if (e != cudaErrorMemoryAllocation || piece <= kMinPieceDoubles) break;
    cudaGetLastError();  // less may be left
  }
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? FOCK_ERR_OOM : FOCK_ERR_CUDA;
  e = cudaMemcpyAsync(d, host.data(), host.size(), cudaMemcpyHostToDevice, stream);
  OneArgs a{};
  a.nbf = nbf;
  a.natom = natom;
  a.groups = (const ShellGroup *)(d + o_g);
  a.perm = (const int *)(d + o_perm);
  a.po = (const int *)(d + o_po);
  a.bf = (const int *)(d + o_bf);
  a.xyz = (const double *)(d + o_xyz);
  a.ex = (const double *)(d + o_ex);
  a.cc = (const double *)(d + o_cc);
  a.axyz = (const double *)(d + o_a);
  a.Z = (const double *)(d + o_z);
  a.boys = dev_boys();
  a.buf = (double *)(d + in_bytes);
  a.S = S;
  a.T = T;
  a.V = V;
  for (const ClassWork &w : work) {
    if (e != cudaSuccess) break;
    a.gp = (const GroupPair *)(d + o_gp) + w.gp0;
    a.ngp = w.ngp;
    a.nsplit = w.nsplit;
    long long q = 0, prim = 0;
    int k = 0;
    while (q < w.npair && e == cudaSuccess) {  // the next piece: whole shell pairs
      a.pair_lo = q;
      a.prim_lo = prim;
      long long room = piece_prims(w);
      for (; k < w.ngp; ++k) {
        const GroupPair &g = gps[w.gp0 + k];
        const long long end = k + 1 < w.ngp ? gps[w.gp0 + k + 1].pair0 : w.npair;
        const long long take = std::min(end - q, room / g.npp);
        q += take;
        prim += take * g.npp;
        room -= take * g.npp;
        if (q < end) break;
      }
      a.npair = q - a.pair_lo;
      a.nprim = prim - a.prim_lo;
      e = launch_class(w.la, w.lb, a, stream);
    }
  }
  cudaError_t e2 = cudaFreeAsync(d, stream);
  if (e == cudaSuccess) e = e2;
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  return e == cudaSuccess ? FOCK_OK : FOCK_ERR_CUDA;
}
