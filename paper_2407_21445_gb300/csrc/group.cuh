// Group kernels: G lanes (1..32) own one contracted quartet (or one share of its
// primitive quartets); the intermediates live in a per-group shared-memory
// scratch, every loop is rolled and driven by small tables of the launch's class
// pair, built by each block at its start.  They serve the class pairs with total
// angular momentum >= 5 in FP64, FP32 and two floats.
//
// Why not one thread per quartet as in kernels_reg.cuh: the half-transformed
// integrals of these classes do not fit the registers of a thread, and the
// unrolled bodies would not fit the instruction caches.  A body here is a few KB.
// The tables replace index arithmetic (the untabulated version spent 30
// instructions per FP64 instruction) by one 8-bit and one 16-bit load per term
// of the transforms, and the digestion's six kinds of outputs by one record each.
//
// The transforms work on pairs: two bra Hermite indices per item in the ket
// transform, two ket components in the bra transform, which share the
// Hermite coefficient; in two floats a pair is a packed FP32 operand
// (fma.f32x2), so that a term costs ten packed instructions for two
// multiply-adds and the loads fit into the free issue slots.
#pragma once

#include "device_common.cuh"
#include "ff.cuh"
#include "kargs.cuh"
#include "prec.cuh"

// FK_CHECK(cond, site, value): diagnostic bounds check, set by the including file
#ifndef FK_CHECK
#define FK_CHECK(cond, site, val) \
  do {                            \
  } while (0)
#endif

namespace fk {

namespace {

// Sizes of a class pair, evaluated once per block from the class indices.
struct Dims {
  int la, lb, lc, ld, na, nb, nc, nd, nab, ncd, ncdp, nhab, nhcd, L, nhL;
};
__host__ __device__ constexpr Dims dims_of(int cb, int ck) {
  Dims d{};
  d.la = 0;
  while ((d.la + 1) * (d.la + 2) / 2 <= cb) ++d.la;
  d.lb = cb - d.la * (d.la + 1) / 2;
  d.lc = 0;
  while ((d.lc + 1) * (d.lc + 2) / 2 <= ck) ++d.lc;
  d.ld = ck - d.lc * (d.lc + 1) / 2;
  d.na = ncart(d.la);
  d.nb = ncart(d.lb);
  d.nc = ncart(d.lc);
  d.nd = ncart(d.ld);
  d.nab = d.na * d.nb;
  d.ncd = d.nc * d.nd;
  d.ncdp = (d.ncd + 1) & ~1;
  d.nhab = nherm(d.la + d.lb);
  d.nhcd = nherm(d.lc + d.ld);
  d.L = d.la + d.lb + d.lc + d.ld;
  d.nhL = nherm(d.L);
  return d;
}

// One entry of the Hermite recursion: R[e] = XYZ[axis] R'[i1] + k R'[i2]
// (k = 0: i2 = i1).
struct RecEntry {
  uint16_t i1, i2, axis, pad;
};

// One element of the density blocks / of the outputs, in the order D_ab, D_cd,
// D_ac, D_ad, D_bc, D_bd and J_ab, J_cd, K_ac, K_ad, K_bc, K_bd: its block and
// place, and for the output the ERI start x and strides so, si, the loop lengths
// no, ni and the start y of the density block it is contracted with.
struct __align__(16) OutEntry {
  uint16_t x, so, si, y;
  uint8_t no, ni, blk, r, c, pad[3];
};

// Shared-memory layout of a block: tables, then the groups' scratch.
struct TabLayout {
  int out, rec, reck, rtab, klist, blist, koff, boff, total;
};
__host__ __device__ constexpr int nstage_of(const Dims &d) { return d.nab + d.ncd + (d.na + d.nb) * (d.nc + d.nd); }
__host__ __device__ constexpr TabLayout tab_layout(const Dims &d, int nEb, int nEk) {
  TabLayout t{};
  int o = 0;
  t.out = o;
  o += nstage_of(d) * (int)sizeof(OutEntry);
  t.rec = o;
  o += d.nhL * (int)sizeof(RecEntry);
  t.reck = o;
  o += d.nhL * 4;
  t.rtab = o;
  o += (d.nhab * d.nhcd * 2 + 3) & ~3;
  t.koff = o;
  o += ((d.ncd + 1) * 2 + 3) & ~3;
  t.boff = o;
  o += ((d.nab + 1) * 2 + 3) & ~3;
  t.klist = o;
  o += (nEk + 3) & ~3;
  t.blist = o;
  o += (nEb + 3) & ~3;
  t.total = (o + 15) & ~15;
  return t;
}

// Scratch of one group in 32-bit words: ERIs, Y, two Hermite buffers, seeds,
// P - Q; the density blocks of the digestion reuse everything behind the ERIs.
// Every array holds an even number of values, so that pairs are aligned.
struct ScrLayout {
  int y, r0, r1, f, xyz, total;
};
template <int G, int PREC>
__host__ __device__ constexpr ScrLayout scr_layout(const Dims &d) {
  constexpr int W = PREC == kF32 ? 1 : 2;
  ScrLayout s{};
  s.y = W * d.nab * d.ncdp;
  s.r0 = s.y + W * d.nhab * d.ncdp;
  s.r1 = s.r0 + W * ((d.nhL + 1) & ~1);
  s.f = s.r1 + W * ((d.nhL + 1) & ~1);
  s.xyz = s.f + W * ((d.L + 2) & ~1);
  int t = s.xyz + W * 4;
  const int st = s.y + W * ((nstage_of(d) + 1) & ~1);
  if (t < st) t = st;
  // the groups of a warp start as many banks apart as their lanes read at once
  constexpr int want = PREC == kF64 ? (2 * G < 4 ? 4 : 2 * G) & 31 : (G < 2 ? 2 : G) & 31;
  while ((t & 31) != want) ++t;
  s.total = t;
  return s;
}

// Arrays of values in the scratch: two floats keep high and low parts apart.
template <int PREC>
struct Arr;
template <>
struct Arr<kF64> {
  double *p;
  __device__ Arr(float *b, int) : p(reinterpret_cast<double *>(b)) {}
  __device__ double ld(int i) const { return p[i]; }
  __device__ void st(int i, double v) const { p[i] = v; }
};
template <>
struct Arr<kF32> {
  float *p;
  __device__ Arr(float *b, int) : p(b) {}
  __device__ float ld(int i) const { return p[i]; }
  __device__ void st(int i, float v) const { p[i] = v; }
};
template <>
struct Arr<kFF> {
  float *p;
  int n;
  __device__ Arr(float *b, int n_) : p(b), n(n_) {}
  __device__ ff ld(int i) const { return {p[i], p[n + i]}; }
  __device__ void st(int i, ff v) const {
    p[i] = v.h;
    p[n + i] = v.l;
  }
};

// Pairs of values: gathered, contiguous (even index), and c + e x.
struct D2 {
  double a, b;
};
template <int PREC>
struct PairOf;
template <>
struct PairOf<kF64> {
  using T = D2;
};
template <>
struct PairOf<kF32> {
  using T = f2;
};
template <>
struct PairOf<kFF> {
  using T = ff2;
};
__device__ __forceinline__ D2 p_zero(D2 *) { return {0.0, 0.0}; }
__device__ __forceinline__ f2 p_zero(f2 *) { return 0ull; }
__device__ __forceinline__ ff2 p_zero(ff2 *) { return {0ull, 0ull}; }
__device__ __forceinline__ D2 p_gather(const Arr<kF64> &x, int i, int j) { return {x.p[i], x.p[j]}; }
__device__ __forceinline__ f2 p_gather(const Arr<kF32> &x, int i, int j) { return f2_pack(x.p[i], x.p[j]); }
__device__ __forceinline__ ff2 p_gather(const Arr<kFF> &x, int i, int j) {
  return {f2_pack(x.p[i], x.p[j]), f2_pack(x.p[x.n + i], x.p[x.n + j])};
}
__device__ __forceinline__ D2 p_load(const Arr<kF64> &x, int i) {
  const double2 v = *reinterpret_cast<const double2 *>(x.p + i);
  return {v.x, v.y};
}
__device__ __forceinline__ f2 p_load(const Arr<kF32> &x, int i) { return *reinterpret_cast<const f2 *>(x.p + i); }
__device__ __forceinline__ ff2 p_load(const Arr<kFF> &x, int i) {
  return {*reinterpret_cast<const f2 *>(x.p + i), *reinterpret_cast<const f2 *>(x.p + x.n + i)};
}
__device__ __forceinline__ void p_store(const Arr<kF64> &x, int i, D2 v) {
  *reinterpret_cast<double2 *>(x.p + i) = make_double2(v.a, v.b);
}
__device__ __forceinline__ void p_store(const Arr<kF32> &x, int i, f2 v) { *reinterpret_cast<f2 *>(x.p + i) = v; }
__device__ __forceinline__ void p_store(const Arr<kFF> &x, int i, ff2 v) {
  *reinterpret_cast<f2 *>(x.p + i) = v.h;
  *reinterpret_cast<f2 *>(x.p + x.n + i) = v.l;
}
__device__ __forceinline__ void p_split(D2 v, double &a, double &b) {
  a = v.a;
  b = v.b;
}
__device__ __forceinline__ void p_split(f2 v, float &a, float &b) { f2_unpack(v, a, b); }
__device__ __forceinline__ void p_split(ff2 v, ff &a, ff &b) {
  f2_unpack(v.h, a.h, b.h);
  f2_unpack(v.l, a.l, b.l);
}
__device__ __forceinline__ D2 p_fma(double e, D2 x, D2 c) { return {fma(e, x.a, c.a), fma(e, x.b, c.b)}; }
__device__ __forceinline__ f2 p_fma(float e, f2 x, f2 c) { return f2_fma(f2_pack(e, e), x, c); }
__device__ __forceinline__ ff2 p_fma(ff e, ff2 x, ff2 c) {
  return ff2_fma({f2_pack(e.h, e.h), f2_pack(e.l, e.l)}, x, c);
}
// e with its sign flipped when bit 31 of s is set
__device__ __forceinline__ double r_flip(double e, unsigned s) {
  return __hiloint2double(__double2hiint(e) ^ (int)s, __double2loint(e));
}
__device__ __forceinline__ float r_flip(float e, unsigned s) { return __uint_as_float(__float_as_uint(e) ^ s); }
__device__ __forceinline__ ff r_flip(ff e, unsigned s) { return {r_flip(e.h, s), r_flip(e.l, s)}; }
// c + k x, k a small integer (0 allowed)
__device__ __forceinline__ double r_addk(float k, double x, double c) { return fma((double)k, x, c); }
__device__ __forceinline__ float r_addk(float k, float x, float c) { return fmaf(k, x, c); }
__device__ __forceinline__ ff r_addk(float k, ff x, ff c) { return ff_fmak(k, x, c); }

// F_m(T) for one order (see boys_seeds_ff)
__device__ __forceinline__ ff boys_one_ff(const float2 *__restrict__ tab, ff T, int m) {
  if (T.h < (float)BOYS_TMAX) {
    const int gi = __float2int_rn(T.h * BOYSFF_INVH);
    const float2 *row = tab + (size_t)gi * BOYSFF_NORD + m;
    const float2 g0 = __ldg(row), g1 = __ldg(row + 1), g2 = __ldg(row + 2);
    return boys_taylor_ff(boys_arg_ff(T, gi), {g0.x, g0.y}, {g1.x, g1.y}, {g2.x, g2.y}, __ldg(row + 3).x,
                          __ldg(row + 4).x, __ldg(row + 5).x);
  }
  const ff rt = ff_norm(ff_rsqrt(T)), it = ff_norm(ff_sqr(rt));
  ff f = boys_far0_ff(rt);
  for (int k = 1; k <= m; ++k) f = boys_far_ff(f, it, k);
  return f;
}

// F_m(T) pref (-2 alpha)^m of one order, FP64 and FP32 (see boys_seeds,
// boys_seeds_f32).
__device__ __forceinline__ double seed_f64(const KArgs &a, const PrimQuartet &q, int m) {
  double f;
  if (q.gi >= 0) {
    const double x = q.Ti - q.T;
    f = boys_taylor_split(a.boys, a.boysf, q.gi, m, x, d2f_small(x));
  } else {
    const double rt = rsqrt_nh(q.T, q.Tf), it = rt * rt;
    f = 0.88622692545275801365 * rt;
    for (int k = 1; k <= m; ++k) f *= (k - 0.5) * it;
  }
  double c = q.pref;
  for (int k = 0; k < m; ++k) c *= q.m2a;
  return f * c;
}
__device__ __forceinline__ float seed_f32(const KArgs &a, float T, float pref, float m2a, int m) {
  float f;
  if (T < (float)BOYS_TMAX) {
    const int gi = __float2int_rn(T * (float)BOYS_INVH);
    const float x = (float)gi * (float)BOYS_H - T;
    const float4 *c = reinterpret_cast<const float4 *>(a.boysf + ((size_t)gi * (LTOT + 1) + m) * BOYS_TAYLOR);
    const float4 c03 = __ldg(c);
    const float2 c45 = __ldg(reinterpret_cast<const float2 *>(c + 1));
    f = fmaf(c45.y, x, c45.x);
    f = fmaf(f, x, c03.w);
    f = fmaf(f, x, c03.z);
    f = fmaf(f, x, c03.y);
    f = fmaf(f, x, c03.x);
  } else {
    const float rt = rsqrtf(T), it = rt * rt;
    f = 0.886226925452758f * rt;
    for (int k = 1; k <= m; ++k) f *= ((float)k - 0.5f) * it;
  }
  float c = pref;
  for (int k = 0; k < m; ++k) c *= m2a;
  return f * c;
}

struct Tabs {
  const OutEntry *out;
  const RecEntry *rec;
  const float *reck;
  const uint16_t *rtab;
  const uint16_t *koff, *boff;
  const uint8_t *klist, *blist;  // blist: bit 7 = odd Hermite degree
};

// The tables of the launch's class pair, at the start of a block's shared memory.
__device__ __forceinline__ Tabs tabs_at(const KArgs &a, const Dims &d, const unsigned char *smem) {
  const TabLayout tl = tab_layout(d, a.tabs->nE[a.cb], a.tabs->nE[a.ck]);
  Tabs tb;
  tb.out = reinterpret_cast<const OutEntry *>(smem + tl.out);
  tb.rec = reinterpret_cast<const RecEntry *>(smem + tl.rec);
  tb.reck = reinterpret_cast<const float *>(smem + tl.reck);
  tb.rtab = reinterpret_cast<const uint16_t *>(smem + tl.rtab);
  tb.koff = reinterpret_cast<const uint16_t *>(smem + tl.koff);
  tb.boff = reinterpret_cast<const uint16_t *>(smem + tl.boff);
  tb.klist = smem + tl.klist;
  tb.blist = smem + tl.blist;
  return tb;
}

// Fills them (every thread of the block takes part) and returns their size.
__device__ __noinline__ int build_tabs(const KArgs &a, unsigned char *smem) {
  const Dims d = dims_of(a.cb, a.ck);
  const ClassTables &ct = *a.tabs;
  const TabLayout tl = tab_layout(d, ct.nE[a.cb], ct.nE[a.ck]);
  {
    OutEntry *out = reinterpret_cast<OutEntry *>(smem + tl.out);
    RecEntry *rec = reinterpret_cast<RecEntry *>(smem + tl.rec);
    float *reck = reinterpret_cast<float *>(smem + tl.reck);
    uint16_t *rtab = reinterpret_cast<uint16_t *>(smem + tl.rtab);
    uint16_t *koff = reinterpret_cast<uint16_t *>(smem + tl.koff), *boff = reinterpret_cast<uint16_t *>(smem + tl.boff);
    uint8_t *klist = smem + tl.klist, *blist = smem + tl.blist;
    const int nb[6] = {d.nab, d.ncd, d.na * d.nc, d.na * d.nd, d.nb * d.nc, d.nb * d.nd};  // block sizes
    const int nc[6] = {d.nb, d.nd, d.nc, d.nd, d.nc, d.nd};                                // their columns
    const int sb = d.ncdp, sa = d.nb * d.ncdp;  // ERI strides of the b and a indices
    for (int i = threadIdx.x; i < nstage_of(d); i += blockDim.x) {
      int blk = 0, first = 0;
      while (i >= first + nb[blk]) first += nb[blk++];
      const int r = (i - first) / nc[blk], c = (i - first) - r * nc[blk];
      // (ERI start; outer stride and length; inner stride and length; density block)
      int x, so, no, si, ni, db;
      if (blk == 0) {  // J_ab += (ab|cd) D_cd
        x = r * sa + c * sb, so = d.nd, no = d.nc, si = 1, ni = d.nd, db = 1;
      } else if (blk == 1) {  // J_cd += (ab|cd) D_ab
        x = r * d.nd + c, so = sa, no = d.na, si = sb, ni = d.nb, db = 0;
      } else if (blk == 2) {  // K_ac += (ab|cd) D_bd
        x = r * sa + c * d.nd, so = sb, no = d.nb, si = 1, ni = d.nd, db = 5;
      } else if (blk == 3) {  // K_ad += (ab|cd) D_bc
        x = r * sa + c, so = sb, no = d.nb, si = d.nd, ni = d.nc, db = 4;
      } else if (blk == 4) {  // K_bc += (ab|cd) D_ad
        x = r * sb + c * d.nd, so = sa, no = d.na, si = 1, ni = d.nd, db = 3;
      } else {  // K_bd += (ab|cd) D_ac
        x = r * sb + c, so = sa, no = d.na, si = d.nd, ni = d.nc, db = 2;
      }
      int y = 0;
      for (int k = 0; k < db; ++k) y += nb[k];
      OutEntry o{};
      o.x = (uint16_t)x;
      o.so = (uint16_t)so;
      o.si = (uint16_t)si;
      o.y = (uint16_t)y;
      o.no = (uint8_t)no;
      o.ni = (uint8_t)ni;
      o.blk = (uint8_t)blk;
      o.r = (uint8_t)r;
      o.c = (uint8_t)c;
      out[i] = o;
    }
    for (int e = threadIdx.x; e < d.nhL; e += blockDim.x) {
      int v[3] = {ct.hvec[e][0], ct.hvec[e][1], ct.hvec[e][2]};
      const int ax = v[0] > 0 ? 0 : (v[1] > 0 ? 1 : 2);
      int k = 0, i1 = 0, i2 = 0;
      if (e > 0) {
        v[ax] -= 1;
        k = v[ax];
        i1 = i2 = hidx(v[0], v[1], v[2]);
        if (k > 0) {
          v[ax] -= 1;
          i2 = hidx(v[0], v[1], v[2]);
        }
      }
      rec[e] = RecEntry{(uint16_t)i1, (uint16_t)i2, (uint16_t)ax, 0};
      reck[e] = (float)k;
    }
    for (int i = threadIdx.x; i < d.nhab * d.nhcd; i += blockDim.x) {
      const int p = i / d.nhcd, q = i - p * d.nhcd;
      rtab[i] = (uint16_t)hidx(ct.hvec[p][0] + ct.hvec[q][0], ct.hvec[p][1] + ct.hvec[q][1],
                               ct.hvec[p][2] + ct.hvec[q][2]);
    }
    // Hermite index of every entry of a pair class' E block
    auto fill = [&](int c, int l1, int l2, int n1, int n2, uint16_t *off, uint8_t *list, bool sign) {
      for (int k = threadIdx.x; k <= n1 * n2; k += blockDim.x) {
        const int e0 = ct.eoff[c][k];
        off[k] = (uint16_t)e0;
        if (k == n1 * n2) continue;
        const uint8_t *x = ct.comp[l1][k / n2], *y = ct.comp[l2][k % n2];
        int e = e0;
        for (int t = 0; t <= x[0] + y[0]; ++t)
          for (int u = 0; u <= x[1] + y[1]; ++u)
            for (int v = 0; v <= x[2] + y[2]; ++v)
              list[e++] = (uint8_t)(hidx(t, u, v) | (sign && ((t + u + v) & 1) ? 0x80 : 0));
      }
    };
    fill(a.ck, d.lc, d.ld, d.nc, d.nd, koff, klist, false);
    fill(a.cb, d.la, d.lb, d.na, d.nb, boff, blist, true);
  }
  __syncthreads();
  return tl.total;
}

template <int G>
__device__ __forceinline__ void gsync(unsigned mask) {
  if constexpr (G > 1) __syncwarp(mask);
}

template <int G, int PREC>
__device__ __forceinline__ void quartet_group(const KArgs &a, const Dims &d, const Tabs &tb, const ScrLayout &sl,
                                              float *scr, int P, int Q, int part, int gl, unsigned gmask,
                                              const MolView &mv) {
  using R = typename RealOf<PREC>::T;
  using P2 = typename PairOf<PREC>::T;
  const DevPairs &dp = a.dp;
  const int2 ab = dp.ab[P], cd = dp.ab[Q];
  const int sA = ab.x, sB = ab.y, sC = cd.x, sD = cd.y;
  FK_CHECK(P >= 0 && P < dp.npair && Q >= 0 && Q < dp.npair, 2, Q);
  FK_CHECK(dp.cls[P] == a.cb && dp.cls[Q] == a.ck, 1, dp.cls[Q]);
  FK_CHECK(dp.prim[P].x >= 0 && dp.prim[P].x + dp.prim[P].y <= a.nprimtot, 3, dp.prim[P].x);
  FK_CHECK(dp.prim[Q].x >= 0 && dp.prim[Q].x + dp.prim[Q].y <= a.nprimtot, 4, dp.prim[Q].x);
  FK_CHECK(dp.eoff[dp.prim[P].x + dp.prim[P].y - 1] + a.tabs->nE[a.cb] <= a.nEtot, 5, a.cb);
  FK_CHECK(dp.eoff[dp.prim[Q].x + dp.prim[Q].y - 1] + a.tabs->nE[a.ck] <= a.nEtot, 6, a.ck);
  FK_CHECK(dp.sbf[sA] + d.na <= mv.N && dp.sbf[sB] + d.nb <= mv.N && dp.sbf[sC] + d.nc <= mv.N &&
               dp.sbf[sD] + d.nd <= mv.N, 7, sA);
  const int neri = d.nab * d.ncdp, nh = (d.nhL + 1) & ~1, nf = (d.L + 2) & ~1;
  const Arr<PREC> eri(scr, neri), Yh(scr + sl.y, d.nhab * d.ncdp), F(scr + sl.f, nf), xyz(scr + sl.xyz, 4);
  for (int i = gl; i < sl.y; i += G) scr[i] = 0.0f;  // zero ERIs
  const int2 pb = dp.prim[P], pk = dp.prim[Q];
  const int sip = bra_split(a.nsplit, pb.y), sjq = a.nsplit / sip;  // this group's share
  const PrimScreen ps = prim_screen(a, mv, sA, sB, sC, sD);
  const CentreDiff<PREC> ac = centre_diff<PREC>(dp, sA, sC);
  bool any = false;
  for (int ip = pb.x + (part & (sip - 1)); ip < pb.x + pb.y; ip += sip) {
    const float gi = dp.Gpf[ip];
    if (prim_skip(a, mv, ps, ip, pk.x, gi * dp.Gpf[pk.x])) break;
    if (PREC == kF64 && !prim_hi(ps, gi * dp.Gpf[pk.x])) break;
    const BraPrim<PREC> bp = bra_prim<PREC>(dp, ip, ac);
    bool anyk = false;
    for (int jq = pk.x + part / sip; jq < pk.x + pk.y; jq += sjq) {
      const float x = gi * dp.Gpf[jq];
      if (prim_skip(a, mv, ps, ip, jq, x)) break;
      if constexpr (PREC == kF64) {
        if (!prim_hi(ps, x)) break;  // the rest is the two-float window
      } else if constexpr (PREC == kFF) {
        if (prim_hi(ps, x)) continue;
      }
      // ---- seeds: lanes over the orders ------------------------------------
      // Q - P instead of P - Q: R(-X) = (-1)^{|h|} R(X), which leaves the sign
      // (-1)^{|q|} of the ket to the bra transform as (-1)^{|p|}
      {
        R X, Y, Z;
        auto seeds = [&](auto &&seed) {
          for (int m = gl; m <= d.L; m += G) {
            const R f = seed(m);
            F.st(m, f);
            if (m == d.L) Arr<PREC>(scr + sl.r0, nh).st(0, f);
          }
        };
        if constexpr (PREC == kF64) {
          const PrimQuartet q = prim_quartet(bp.P4, bp.Pf, dp.pz[jq], dp.pf[jq]);
          X = -q.X;
          Y = -q.Y;
          Z = -q.Z;
          seeds([&](int m) { return seed_f64(a, q, m); });
        } else if constexpr (PREC == kF32) {
          const float4 QC = dp.paf[jq];
          X = -(bp.PA.x - QC.x + ac.x);
          Y = -(bp.PA.y - QC.y + ac.y);
          Z = -(bp.PA.z - QC.z + ac.z);
          const float rs = rsqrtf(bp.PA.w + QC.w);
          const float alpha = (bp.PA.w * QC.w) * (rs * rs);
          const float T = alpha * fmaf(X, X, fmaf(Y, Y, Z * Z));
          seeds([&](int m) { return seed_f32(a, T, rs, -2.0f * alpha, m); });
        } else {
          const float4 h = dp.paf[jq], l = dp.pal[jq];
          X = ff_norm(ff_sub({h.x, l.x}, bp.X));
          Y = ff_norm(ff_sub({h.y, l.y}, bp.Y));
          Z = ff_norm(ff_sub({h.z, l.z}, bp.Z));
          const ff eta = {h.w, l.w};
          const ff rs = ff_norm(ff_rsqrt(ff_norm(ff_add(bp.w, eta))));
          const ff alpha = ff_norm(ff_mul(ff_norm(ff_mul(bp.w, rs)), ff_norm(ff_mul(eta, rs))));
          const ff T = ff_norm(ff_mul(alpha, ff_norm(ff_fma(X, X, ff_fma(Y, Y, ff_sqr(Z))))));
          const ff m2a = {-2.0f * alpha.h, -2.0f * alpha.l};
          seeds([&](int m) {
            ff f = ff_norm(ff_mul(boys_one_ff(a.boysff, T, m), rs));
            for (int k = 0; k < m; ++k) f = ff_norm(ff_mul(f, m2a));
            return f;
          });
        }
        for (int c = gl; c < 3; c += G) xyz.st(c, c == 0 ? X : (c == 1 ? Y : Z));
      }
      gsync<G>(gmask);
      // ---- Hermite recursion -------------------------------------------------
      int cur = sl.r0, nxt = sl.r1;
      for (int n = d.L - 1; n >= 0; --n) {
        const int cnt = nherm(d.L - n);
        const Arr<PREC> c(scr + cur, nh), o(scr + nxt, nh);
        for (int e = gl; e < cnt; e += G) {
          R v;
          if (e == 0) {
            v = F.ld(n);
          } else {
            const RecEntry r = tb.rec[e];
            v = r_addk(tb.reck[e], c.ld(r.i2), r_mul(xyz.ld(r.axis), c.ld(r.i1)));
          }
          o.st(e, v);
        }
        gsync<G>(gmask);
        const int t = cur;
        cur = nxt;
        nxt = t;
      }
      // ---- ket transform: two bra Hermite indices per item ------------------
      const Arr<PREC> Rh(scr + cur, nh);
      const int eq = dp.eoff[jq];
      const int npp = (d.nhab + 1) >> 1;
      for (int kc = 0, pp = gl;; pp += G) {
        while (pp >= npp) {
          pp -= npp;
          ++kc;
        }
        if (kc >= d.ncd) break;
        const int p0 = 2 * pp, p1 = p0 + 1 < d.nhab ? p0 + 1 : p0;
        const uint16_t *t0 = tb.rtab + p0 * d.nhcd, *t1 = tb.rtab + p1 * d.nhcd;
        const int y0 = p0 * d.ncdp + kc, y1 = p1 * d.ncdp + kc;
        P2 acc = anyk ? p_gather(Yh, y0, y1) : p_zero((P2 *)nullptr);
        const int e1 = tb.koff[kc + 1];
#pragma unroll 2
        for (int e = tb.koff[kc]; e < e1; ++e) {
          const int q = tb.klist[e];
          acc = p_fma(load_e<PREC>(dp, eq, e), p_gather(Rh, t0[q], t1[q]), acc);
        }
        R v0, v1;
        p_split(acc, v0, v1);
        Yh.st(y0, v0);
        if (p1 != p0) Yh.st(y1, v1);
      }
      anyk = true;
      gsync<G>(gmask);
    }
    if (!anyk) continue;
    any = true;
    // ---- bra transform: two ket components per item ---------------------------
    const int ep = dp.eoff[ip];
    const int ncp = d.ncdp >> 1;
    for (int ka = 0, jp = gl;; jp += G) {
      while (jp >= ncp) {
        jp -= ncp;
        ++ka;
      }
      if (ka >= d.nab) break;
      const int o = ka * d.ncdp + 2 * jp;
      P2 acc = p_load(eri, o);
      const int e1 = tb.boff[ka + 1];
#pragma unroll 2
      for (int e = tb.boff[ka]; e < e1; ++e) {
        const int q = tb.blist[e];
        acc = p_fma(r_flip(load_e<PREC>(dp, ep, e), (unsigned)(q & 0x80) << 24),
                    p_load(Yh, (q & 0x7f) * d.ncdp + 2 * jp), acc);
      }
      p_store(eri, o, acc);
    }
    gsync<G>(gmask);
  }
  if (!any) return;
  // ---- digestion: density blocks staged, then one output per lane and pass
  // (8-fold symmetry, Sec. 2.3 / 3.2) ---------------------------------------------
  float fac = 1.0f;
  if (sA == sB) fac *= 0.5f;
  if (sC == sD) fac *= 0.5f;
  if (P == Q) fac *= 0.5f;
  const int N = mv.N;
  const int fa = dp.sbf[sA], fb = dp.sbf[sB], fc = dp.sbf[sC], fd = dp.sbf[sD];
  // place of an element of block blk (ab, cd, ac, ad, bc, bd) in an N x N matrix
  auto place = [&](const OutEntry &o) -> size_t {
    const int r0 = o.blk == 1 ? fc : (o.blk >= 4 ? fb : fa);
    const int c0 = o.blk == 0 ? fb : ((o.blk & 1) ? fd : fc);
    return (size_t)(r0 + o.r) * N + c0 + o.c;
  };
  const int nst = nstage_of(d);
  const Arr<PREC> Ds(scr + sl.y, (nst + 1) & ~1);
  for (int i = gl; i < nst; i += G) {
    const size_t at = place(tb.out[i]);
    if constexpr (PREC == kF64)
      Ds.st(i, __ldg(mv.D + at));
    else if constexpr (PREC == kF32)
      Ds.st(i, __ldg(mv.Df + at));
    else
      Ds.st(i, ff_from_double(__ldg(mv.D + at)));
  }
  gsync<G>(gmask);
  const int o0 = (a.parts & 1) ? 0 : d.nab + d.ncd, o1 = (a.parts & 2) ? nst : d.nab + d.ncd;
  for (int o = o0 + gl; o < o1; o += G) {
    const OutEntry t = tb.out[o];
    int x = t.x, y = t.y;
    R s0 = r_zero<R>(), s1 = r_zero<R>();  // two chains
    for (int i = 0; i < t.no; ++i, x += t.so) {
      int xi = x, j = 0;
      for (; j + 1 < t.ni; j += 2, xi += 2 * t.si, y += 2) {
        s0 = r_fma(eri.ld(xi), Ds.ld(y), s0);
        s1 = r_fma(eri.ld(xi + t.si), Ds.ld(y + 1), s1);
      }
      if (j < t.ni) s0 = r_fma(eri.ld(xi), Ds.ld(y++), s0);
    }
    const float f = t.blk < 2 ? 2.0f * fac : fac;
    double v;
    if constexpr (PREC == kF64) {
      v = (double)f * (s0 + s1);
    } else if constexpr (PREC == kF32) {
      v = f2d_any(f * (s0 + s1));
    } else {
      const ff s = ff_add(s0, s1);
      v = f2d_any(f * s.h) + f2d_fin(f * s.l);  // l is finite where h is
    }
    atomicAdd((t.blk < 2 ? mv.J : mv.K) + place(t), v);
  }
  gsync<G>(gmask);
}

// One pass of a warp over the work units for one arithmetic.  Warp-level work
// queue, as in the register kernels: the unit's kets are screened 32 at a time
// and the survivors of this arithmetic appended to a queue that is drained NG
// quartets at a time (one per group), so no group holds a screened quartet
// while the others compute; the rest carries over to the next unit.
template <int G, int PREC>
__device__ __forceinline__ void run_group_list(const KArgs &a, int *counter, const Dims &d, const Tabs &tb, float *warp_scr,
                                         QEntry *q, int lane) {
  constexpr int NG = 32 / G;
  const ScrLayout sl = scr_layout<G, PREC>(d);
  const int grp = lane / G, gl = lane - grp * G;
  float *scr = warp_scr + (size_t)grp * sl.total;
  const unsigned gmask = G == 32 ? 0xffffffffu : (((1u << (G & 31)) - 1u) << (grp * G));
  const unsigned lt = (1u << lane) - 1u;
  int n = 0, P = 0, k0 = 0, c = 0, end = 0;
  bool more = true;
  for (;;) {
    if (more && c >= end) {
      const int u = next_unit(counter, lane);
      if (u < a.nunits) {
        const Unit un = a.units[u];
        P = un.bra;
        k0 = un.k0;
        c = 0;
        end = (un.k1 - un.k0) * a.nsplit;
      } else {
        more = false;
      }
    }
    if (more) {
      const int2 ab = a.dp.ab[P];
      const int i = c + lane;
      const int Q = k0 + i / a.nsplit, part = i % a.nsplit;
      bool in = false;
      if (i < end) {
        const MolView mv = mol_view(a, ab.x);
        const int2 cd = a.dp.ab[Q];
        const float b = quartet_bound(a, mv, ab.x, ab.y, cd.x, cd.y, P, Q);
        if (b >= 0.0f && share_used(a, P, Q, part)) {
          const QuartetWindows w = quartet_windows(a, mv, ab.x, ab.y, cd.x, cd.y, P, Q, b);
          in = PREC == kF64 ? w.f64 : (PREC == kFF ? w.ff : w.f32);
        }
      }
      c += 32;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (in) q[n + __popc(m & lt)] = QEntry{P, Q, part};
      n += __popc(m);
      __syncwarp();
    }
    const int k = more ? (n / NG) * NG : n;  // after the last unit the rest too
    for (int i = 0; i < k; i += NG)
      if (i + grp < k) {
        const QEntry e = q[i + grp];
        const MolView mv = mol_view(a, a.dp.ab[e.P].x);
        quartet_group<G, PREC>(a, d, tb, sl, scr, e.P, e.Q, e.part, gl, gmask, mv);
      }
    __syncwarp();
    const int rest = n - k;  // < NG <= 32 entries move to the front
    QEntry v{0, 0, 0};
    if (lane < rest) v = q[k + lane];
    __syncwarp();
    if (k > 0 && lane < rest) q[lane] = v;
    n = rest;
    __syncwarp();
    if (!more && n == 0) break;
  }
}

}  // namespace

}  // namespace fk
