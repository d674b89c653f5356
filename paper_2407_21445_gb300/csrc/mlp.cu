// Atom-pair MLP for the learned initial density: three dense layers
// (nin -> H -> H -> nout) with SiLU activations, BF16 weights, FP32
// activations and FP32 accumulation; forward, masked mean-squared-error loss
// with backward pass, and an Adam step on FP32 master weights.  Written for
// the SCF extension (no counterpart in the paper).
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <new>
#include <type_traits>
#include <vector>

#include "fock_impl.h"

struct fock_mlp {
  int nin, H, nout, max_batch;
  size_t nparam;
  // parameters (FP32 master), BF16 copies of the three weight matrices
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
  __nv_bfloat16 *w16 = nullptr;
  // activations for max_batch rows
  float *z1 = nullptr, *a1 = nullptr, *z2 = nullptr, *a2 = nullptr, *dy = nullptr;
  float *d1 = nullptr, *d2 = nullptr, *loss = nullptr;
  long long step = 0;
  size_t off_w1, off_b1, off_w2, off_b2, off_w3, off_b3;
  size_t o16_w1, o16_w2, o16_w3;
};

namespace {

// Round an FP32 value to TF32 (10-bit mantissa, round to nearest away) and
// return it as its 32-bit pattern, the operand format of mma .tf32.
__device__ __forceinline__ uint32_t to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}

// D = A B + C for one m16n8k8 tile on the tensor cores (TF32 inputs, FP32
// accumulation; fragment layouts of the PTX ISA for mma.m16n8k8 .tf32).
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// What a GEMM does with its accumulators.
enum Epi {
  kStore,     // C = acc (+ bias)
  kSilu,      // C = acc + bias, act = silu(C)
  kSiluBwd,   // C = acc * silu'(aux), aux the layer's pre-activation
  kLoss       // C = 2 mask (y - t) / norm with y = acc + bias, loss += mask (y - t)^2 / norm
};

// C[m][n] = sum_k A[m*lda+k] B(k,n), B(k,n) = TB ? B[n*ldb+k] : B[k*ldb+n]
// (BF16 weights), on the tensor cores: a block of eight warps owns a 32 x 64 tile
// of C (each warp 16 x 16), K in steps of 32, the operands of the next four
// steps under way in registers while one is multiplied (K = 128: all of them from
// the start).  A is split into a TF32 high part and a TF32 remainder whose
// products are both accumulated in FP32, which keeps the product accurate to
// about FP32 rounding (BF16 weights are exact in TF32).
//
// At the training sizes (4096 rows, 128 hidden units) the work is a few
// microseconds of any unit's rate; what counts is blocks in flight, hidden load
// latency and launches.  32-row tiles give 256 blocks for 152 SMs, 64-row tiles
// 128; loss and activation derivative ride along in the epilogues; the three weight
// gradients with their bias sums are one launch (k_grads).  A training step at
// 4096 rows takes 0.20 ms, with four warps and one step ahead 15 us more.
constexpr int BM = 32, BN = 64, GK = 32, GTHREADS = 256, GDEPTH = 4;
struct GemmArgs {
  int M, N, K, lda, ldb, ldc;
  const float *A;
  const __nv_bfloat16 *B;
  float *C, *act;
  const float *bias, *aux;
  const float *target, *mask;
  float inv_norm;
  float *loss;
};

// element (row, k) of a staged tile of ROWS rows: k-contiguous in memory is kept
// [row][k], row-contiguous [k][row], both free of bank conflicts for the fragments
template <int ROWS, bool KMAJOR>
__device__ __forceinline__ int tile_at(int row, int k) {
  return KMAJOR ? k * (ROWS + 8) + row : row * (GK + 4) + k;
}

template <bool TB, int EPI>
__global__ void __launch_bounds__(GTHREADS) k_gemm(GemmArgs g) {
  __shared__ float As2[2][BM * (GK + 4)];
  __shared__ float Bs2[2][TB ? BN * (GK + 4) : GK * (BN + 8)];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gq = lane >> 2, t = lane & 3;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int wm = (warp >> 2) * 16, wn = (warp & 3) * 16;
  constexpr int NA_ = BM * GK / GTHREADS, NB_ = BN * GK / GTHREADS;
  float ras[GDEPTH][NA_], rbs[GDEPTH][NB_];
  // thread i takes elements i, i + GTHREADS, ...: the contiguous index runs fastest
  auto read = [&](float (&ra)[NA_], float (&rb)[NB_], int k0) {
#pragma unroll
    for (int q = 0; q < NA_; ++q) {
      const int i = tid + GTHREADS * q, k = k0 + i % GK, m = m0 + i / GK;
      ra[q] = (m < g.M && k < g.K) ? g.A[(size_t)m * g.lda + k] : 0.0f;
    }
#pragma unroll
    for (int q = 0; q < NB_; ++q) {
      const int i = tid + GTHREADS * q, r = TB ? i / GK : i % BN, k = k0 + (TB ? i % GK : i / BN), n = n0 + r;
      rb[q] = (n < g.N && k < g.K) ? __bfloat162float(g.B[TB ? (size_t)n * g.ldb + k : (size_t)k * g.ldb + n]) : 0.0f;
    }
  };
  float acc[2][4];
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[j][r] = 0.0f;
#pragma unroll
  for (int u = 0; u < GDEPTH; ++u) read(ras[u], rbs[u], u * GK);
  for (int kc = 0; kc < g.K; kc += GDEPTH * GK) {
#pragma unroll
    for (int u = 0; u < GDEPTH; ++u) {
      const int k0 = kc + u * GK;
      if (k0 >= g.K) break;
      float (&ra)[NA_] = ras[u], (&rb)[NB_] = rbs[u];
      // two buffers: whoever writes one again has passed the barrier after its last use
      float *As = As2[u & 1], *Bs = Bs2[u & 1];
#pragma unroll
      for (int q = 0; q < NA_; ++q) {
        const int i = tid + GTHREADS * q;
        As[tile_at<BM, false>(i / GK, i % GK)] = ra[q];
      }
#pragma unroll
      for (int q = 0; q < NB_; ++q) {
        const int i = tid + GTHREADS * q;
        Bs[tile_at<BN, !TB>(TB ? i / GK : i % BN, TB ? i % GK : i / BN)] = rb[q];
      }
      __syncthreads();
      if (k0 + GDEPTH * GK < g.K) read(ra, rb, k0 + GDEPTH * GK);
#pragma unroll
      for (int ks = 0; ks < GK; ks += 8) {
        uint32_t ah[4], al[4];
        const int r = wm + gq;
        const float va[4] = {As[tile_at<BM, false>(r, ks + t)], As[tile_at<BM, false>(r + 8, ks + t)],
                             As[tile_at<BM, false>(r, ks + t + 4)], As[tile_at<BM, false>(r + 8, ks + t + 4)]};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          ah[q] = to_tf32(va[q]);
          al[q] = to_tf32(va[q] - __uint_as_float(ah[q]));
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          uint32_t bh[2];
          const int c = wn + 8 * j + gq;
          const float vb[2] = {Bs[tile_at<BN, !TB>(c, ks + t)], Bs[tile_at<BN, !TB>(c, ks + t + 4)]};
          bh[0] = __float_as_uint(vb[0]);
          bh[1] = __float_as_uint(vb[1]);
          mma_tf32(acc[j], al, bh);
          mma_tf32(acc[j], ah, bh);
        }
      }
    }
  }
  float lsum = 0.0f;
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int row = m0 + wm + gq + (r >= 2 ? 8 : 0), col = n0 + wn + 8 * j + 2 * t + (r & 1);
      if (row >= g.M || col >= g.N) continue;
      float v = acc[j][r];
      if (EPI != kSiluBwd && g.bias) v += g.bias[col];
      const size_t at = (size_t)row * g.ldc + col;
      if constexpr (EPI == kSilu) {
        g.act[at] = v * (1.0f / (1.0f + __expf(-v)));
      } else if constexpr (EPI == kSiluBwd) {
        const float z = g.aux[at], s = 1.0f / (1.0f + __expf(-z));
        v = v * s * (1.0f + z * (1.0f - s));
      } else if constexpr (EPI == kLoss) {
        const float w = g.mask ? g.mask[at] : 1.0f, e = v - g.target[at], d = e * w;
        lsum += d * e * g.inv_norm;
        v = 2.0f * d * g.inv_norm;
      }
      g.C[at] = v;
    }
  if constexpr (EPI == kLoss) {
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if (lane == 0) atomicAdd(g.loss, lsum);
  }
}

// Weight and bias gradients of all three layers, dW += d^T x and db += column
// sums of d over the batch's rows, in one launch.  A warp owns a 16 x 8 tile of
// one dW and walks all rows, eight per step; a block is four tiles side by side,
// which read the same columns of d.  The rows are not split over warps: the
// tensor core rounds its FP32 sums toward zero, so splitting changes the
// gradients by more than 1e-5.  One warp's latency per eight rows (3 dependent
// mma, 12 conversions, loads) bounds the kernel, so nothing else stands in the
// chain and every scheduler has a warp of its own: the operands come from L2
// straight into registers, GAHEAD steps ahead, without shared memory or barriers,
// and the tile is the smallest that the instruction has.  Against it, in a training
// step at 4096 rows and 128 hidden units: 32 x 32 tiles behind a four-stage cp.async
// pipeline 32 us more, GAHEAD = 8 12 us more, all loads of eight steps in one go
// into two buffers 5 us more than one by one.
constexpr int GTM = 16, GTN = 32, GAHEAD = 16;
struct GradLayer {
  const float *d, *x;  // [rows][M], [rows][N]
  float *gw, *gb;
  int M, N, tiles_n, block0;
};
struct GradArgs {
  GradLayer l[3];
  int rows;
};
__global__ void __launch_bounds__(128) k_grads(GradArgs g) {
  int li = 0;
  while (li < 2 && (int)blockIdx.x >= g.l[li + 1].block0) ++li;
  const GradLayer &l = g.l[li];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gq = lane >> 2, t = lane & 3;
  const int tile = blockIdx.x - l.block0, m0 = tile / l.tiles_n * GTM, n0 = tile % l.tiles_n * GTN + 8 * warp;
  const int ma = m0 + gq, nb = n0 + gq, rows = g.rows;
  // Rows t and t + 4 of the next step to load, columns ma and ma + 8 of d and nb
  // of x.  Columns past the edge read the last one: a tile's rows and columns do
  // not mix, and theirs are not written.
  const int c0 = min(ma, l.M - 1), c1 = min(ma + 8, l.M - 1), cx = min(nb, l.N - 1);
  const size_t sd = 4 * (size_t)l.M, sx = 4 * (size_t)l.N;
  const float *pd[4], *px[2];
#pragma unroll
  for (int q = 0; q < 4; ++q) pd[q] = l.d + (size_t)t * l.M + (q >> 1) * sd + (q & 1 ? c1 : c0);
#pragma unroll
  for (int q = 0; q < 2; ++q) px[q] = l.x + (size_t)t * l.N + q * sx + cx;
  int row = t;
  float fa[GAHEAD][4], fb[GAHEAD][2];
  // WHOLE: all eight rows of the step are there; else a missing row is zero
  auto load = [&](float (&va)[4], float (&vb)[2], auto whole) {
    constexpr bool WHOLE = decltype(whole)::value;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      va[q] = WHOLE || row + 4 * (q >> 1) < rows ? __ldg(pd[q]) : 0.0f;
      pd[q] += 2 * sd;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      vb[q] = WHOLE || row + 4 * q < rows ? __ldg(px[q]) : 0.0f;
      px[q] += 2 * sx;
    }
    if constexpr (!WHOLE) row += 8;
  };
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f}, s0 = 0.0f, s1 = 0.0f;
  auto steps = [&](auto whole) {  // GAHEAD steps, each followed by the load GAHEAD steps later
#pragma unroll
    for (int u = 0; u < GAHEAD; ++u) {
      uint32_t ah[4], al[4], bh[2], bl[2];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        ah[q] = to_tf32(fa[u][q]);
        al[q] = to_tf32(fa[u][q] - __uint_as_float(ah[q]));
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        bh[q] = to_tf32(fb[u][q]);
        bl[q] = to_tf32(fb[u][q] - __uint_as_float(bh[q]));
      }
      s0 += fa[u][0] + fa[u][2];
      s1 += fa[u][1] + fa[u][3];
      load(fa[u], fb[u], whole);
      mma_tf32(acc, al, bh);
      mma_tf32(acc, ah, bl);
      mma_tf32(acc, ah, bh);
    }
  };
#pragma unroll
  for (int u = 0; u < GAHEAD; ++u) load(fa[u], fb[u], std::false_type{});
  int r0 = 0;
  for (; r0 + 16 * GAHEAD <= rows; r0 += 8 * GAHEAD) steps(std::true_type{});
  row = r0 + 8 * GAHEAD + t;
  for (; r0 < rows; r0 += 8 * GAHEAD) steps(std::false_type{});  // steps past the last row add zeros
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int m = ma + (r >= 2 ? 8 : 0), n = n0 + 2 * t + (r & 1);
    if (m < l.M && n < l.N) l.gw[(size_t)m * l.N + n] += acc[r];
  }
  if (n0 == 0) {  // one warp per 16 rows of dW: column sums of d
    s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
    s0 += __shfl_xor_sync(0xffffffffu, s0, 2);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 2);
    if (t == 0 && ma < l.M) l.gb[ma] += s0;
    if (t == 0 && ma + 8 < l.M) l.gb[ma + 8] += s1;
  }
}

// Where the BF16 copies of the three weight matrices lie in the parameter vector.
struct Bf16Map {
  long long begin[3], end[3], dst[3];
};
__device__ __forceinline__ void store_bf16(const Bf16Map &m, long long i, float v, __nv_bfloat16 *w) {
#pragma unroll
  for (int k = 0; k < 3; ++k)
    if (i >= m.begin[k] && i < m.end[k]) w[m.dst[k] + i - m.begin[k]] = __float2bfloat16_rn(v);
}

// Adam step; the BF16 copies follow in the same pass.
__global__ void k_adam(long long n, float *__restrict__ p, float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, __nv_bfloat16 *__restrict__ w16, Bf16Map map, float lr, float b1, float b2,
                       float eps, float wd, float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i] + wd * p[i];
    m[i] = b1 * m[i] + (1.0f - b1) * gi;
    v[i] = b2 * v[i] + (1.0f - b2) * gi * gi;
    const float x = p[i] - lr * (m[i] * c1) / (sqrtf(v[i] * c2) + eps);
    p[i] = x;
    g[i] = 0.0f;
    store_bf16(map, i, x, w16);
  }
}

__global__ void k_to_bf16(long long n, const float *__restrict__ p, __nv_bfloat16 *__restrict__ w16, Bf16Map map) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    store_bf16(map, i, p[i], w16);
}

int blocks_for(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b > 4096 ? 4096 : (b < 1 ? 1 : b));
}

// A grid has at most 65535 blocks of columns: wider layers take several launches.
constexpr int kMaxCols = 65535 * BN;
template <bool TB, int EPI>
cudaError_t gemm(GemmArgs g, cudaStream_t st) {
  for (int left = g.N;; left -= kMaxCols) {
    g.N = left < kMaxCols ? left : kMaxCols;
    k_gemm<TB, EPI><<<dim3((g.M + BM - 1) / BM, (g.N + BN - 1) / BN), GTHREADS, 0, st>>>(g);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || left <= kMaxCols) return e;
    // the next columns; rows keep their stride
    g.B += TB ? (size_t)kMaxCols * g.ldb : (size_t)kMaxCols;
    g.C += kMaxCols;
    if (g.act) g.act += kMaxCols;
    if (g.bias) g.bias += kMaxCols;
    if (g.aux) g.aux += kMaxCols;
    if (g.target) g.target += kMaxCols;
    if (g.mask) g.mask += kMaxCols;
  }
}

Bf16Map bf16_map(const fock_mlp *n) {
  const long long H = n->H;
  return Bf16Map{{(long long)n->off_w1, (long long)n->off_w2, (long long)n->off_w3},
                 {(long long)n->off_w1 + H * n->nin, (long long)n->off_w2 + H * H, (long long)n->off_w3 + n->nout * H},
                 {(long long)n->o16_w1, (long long)n->o16_w2, (long long)n->o16_w3}};
}

cudaError_t refresh_bf16(fock_mlp *n, cudaStream_t st) {
  k_to_bf16<<<blocks_for((long long)n->nparam), 256, 0, st>>>((long long)n->nparam, n->p, n->w16, bf16_map(n));
  return cudaGetLastError();
}

// dense layer Y = X W^T + b (weights in BF16)
GemmArgs layer(int B, int nout, int nin, const float *X, const __nv_bfloat16 *W, const float *bias, float *C) {
  GemmArgs g{};
  g.M = B;
  g.N = nout;
  g.K = nin;
  g.A = X;
  g.lda = nin;
  g.B = W;
  g.ldb = nin;
  g.C = C;
  g.ldc = nout;
  g.bias = bias;
  return g;
}

cudaError_t hidden_layers(fock_mlp *n, const float *X, int B, cudaStream_t st) {
  GemmArgs g = layer(B, n->H, n->nin, X, n->w16 + n->o16_w1, n->p + n->off_b1, n->z1);
  g.act = n->a1;
  cudaError_t e = gemm<true, kSilu>(g, st);
  if (e != cudaSuccess) return e;
  g = layer(B, n->H, n->H, n->a1, n->w16 + n->o16_w2, n->p + n->off_b2, n->z2);
  g.act = n->a2;
  return gemm<true, kSilu>(g, st);
}

cudaError_t weight_grads(fock_mlp *n, int B, const float *X, cudaStream_t st) {
  GradArgs g{};
  g.rows = B;
  int blocks = 0;
  auto add = [&](int i, const float *d, const float *x, size_t off_w, size_t off_b, int M, int N) {
    const int tn = (N + GTN - 1) / GTN;
    g.l[i] = GradLayer{d, x, n->g + off_w, n->g + off_b, M, N, tn, blocks};
    blocks += (M + GTM - 1) / GTM * tn;
  };
  add(0, n->dy, n->a2, n->off_w3, n->off_b3, n->nout, n->H);
  add(1, n->d2, n->a1, n->off_w2, n->off_b2, n->H, n->H);
  add(2, n->d1, X, n->off_w1, n->off_b1, n->H, n->nin);
  k_grads<<<blocks, 128, 0, st>>>(g);
  return cudaGetLastError();
}

// da = d W, times silu'(z): the gradient at the layer below
cudaError_t input_grad(int B, int nout, int nin, const float *d, const __nv_bfloat16 *W, const float *z, float *out,
                       cudaStream_t st) {
  GemmArgs g{};
  g.M = B;
  g.N = nin;
  g.K = nout;
  g.A = d;
  g.lda = nout;
  g.B = W;
  g.ldb = nin;
  g.C = out;
  g.ldc = nin;
  g.aux = z;
  return gemm<false, kSiluBwd>(g, st);
}

fock_status st_of(cudaError_t e) {
  if (e == cudaSuccess) return FOCK_OK;
  return e == cudaErrorMemoryAllocation ? FOCK_ERR_OOM : FOCK_ERR_CUDA;
}

}  // namespace

extern "C" {

fock_status fock_mlp_create(int32_t nin, int32_t nhidden, int32_t nout, int32_t max_batch, uint64_t seed,
                            fock_mlp **out) {
  if (!out || nin < 1 || nhidden < 1 || nout < 1 || max_batch < 1) return FOCK_ERR_INVALID_ARG;
  *out = nullptr;
  fock_mlp *n = new (std::nothrow) fock_mlp();
  if (!n) return FOCK_ERR_OOM;
  n->nin = nin;
  n->H = nhidden;
  n->nout = nout;
  n->max_batch = max_batch;
  const size_t H = nhidden;
  n->off_w1 = 0;
  n->off_b1 = n->off_w1 + H * nin;
  n->off_w2 = n->off_b1 + H;
  n->off_b2 = n->off_w2 + H * H;
  n->off_w3 = n->off_b2 + H;
  n->off_b3 = n->off_w3 + (size_t)nout * H;
  n->nparam = n->off_b3 + nout;
  n->o16_w1 = 0;
  n->o16_w2 = H * nin;
  n->o16_w3 = n->o16_w2 + H * H;
  const size_t n16 = n->o16_w3 + (size_t)nout * H;
  const size_t act = (size_t)max_batch * (4 * H + (size_t)nout + 2 * H);
  float *buf = nullptr;
  cudaError_t e = cudaMalloc(&buf, sizeof(float) * (4 * n->nparam + act + 1) + sizeof(__nv_bfloat16) * n16);
  if (e != cudaSuccess) {
    delete n;
    return st_of(e);
  }
  n->p = buf;
  n->g = n->p + n->nparam;
  n->m = n->g + n->nparam;
  n->v = n->m + n->nparam;
  float *a = n->v + n->nparam;
  const size_t B = max_batch;
  n->z1 = a;
  n->a1 = n->z1 + B * H;
  n->z2 = n->a1 + B * H;
  n->a2 = n->z2 + B * H;
  n->dy = n->a2 + B * H;
  n->d1 = n->dy + B * nout;
  n->d2 = n->d1 + B * H;
  n->loss = n->d2 + B * H;
  n->w16 = (__nv_bfloat16 *)(n->loss + 1);
  // He-style initialisation from a 64-bit LCG (host), biases zero
  std::vector<float> p(n->nparam, 0.0f);
  uint64_t s = seed * 6364136223846793005ull + 1442695040888963407ull;
  auto uni = [&]() {
    s = s * 6364136223846793005ull + 1442695040888963407ull;
    return (double)(s >> 11) * (1.0 / 9007199254740992.0);
  };
  auto fill = [&](size_t off, size_t cnt, int fan_in) {
    const double r = sqrt(3.0 / fan_in);
    for (size_t i = 0; i < cnt; ++i) p[off + i] = (float)((2.0 * uni() - 1.0) * r);
  };
  fill(n->off_w1, H * nin, nin);
  fill(n->off_w2, H * H, (int)H);
  fill(n->off_w3, (size_t)nout * H, (int)H);
  e = cudaMemcpy(n->p, p.data(), sizeof(float) * n->nparam, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(n->g, 0, sizeof(float) * 3 * n->nparam);
  if (e == cudaSuccess) e = refresh_bf16(n, 0);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    cudaFree(buf);
    delete n;
    return st_of(e);
  }
  *out = n;
  return FOCK_OK;
}

fock_status fock_mlp_free(fock_mlp *n) {
  if (!n) return FOCK_OK;
  cudaFree(n->p);
  delete n;
  return FOCK_OK;
}

int64_t fock_mlp_num_params(const fock_mlp *n) { return n ? (int64_t)n->nparam : -1; }

fock_status fock_mlp_get_params(const fock_mlp *n, float *host_params, float *host_grads) {
  if (!n) return FOCK_ERR_INVALID_ARG;
  cudaError_t e = cudaSuccess;
  if (host_params) e = cudaMemcpy(host_params, n->p, sizeof(float) * n->nparam, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && host_grads) e = cudaMemcpy(host_grads, n->g, sizeof(float) * n->nparam, cudaMemcpyDeviceToHost);
  return st_of(e);
}

fock_status fock_mlp_set_params(fock_mlp *n, const float *host_params) {
  if (!n || !host_params) return FOCK_ERR_INVALID_ARG;
  cudaError_t e = cudaMemcpy(n->p, host_params, sizeof(float) * n->nparam, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = refresh_bf16(n, 0);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return st_of(e);
}

fock_status fock_mlp_forward(fock_mlp *n, const float *X, int32_t B, float *Y, cudaStream_t st) {
  if (!n || !X || !Y || B < 0 || B > n->max_batch) return FOCK_ERR_INVALID_ARG;
  if (B == 0) return FOCK_OK;
  cudaError_t e = hidden_layers(n, X, B, st);
  if (e == cudaSuccess)
    e = gemm<true, kStore>(layer(B, n->nout, n->H, n->a2, n->w16 + n->o16_w3, n->p + n->off_b3, Y), st);
  return st_of(e);
}

fock_status fock_mlp_loss_backward(fock_mlp *n, const float *X, const float *T, const float *mask, int32_t B,
                                   double norm, float *loss_host, cudaStream_t st) {
  if (!n || !X || !T || B < 1 || B > n->max_batch || !(norm > 0.0)) return FOCK_ERR_INVALID_ARG;
  const int H = n->H, O = n->nout;
  cudaError_t e = cudaMemsetAsync(n->loss, 0, sizeof(float), st);
  if (e == cudaSuccess) e = hidden_layers(n, X, B, st);
  if (e == cudaSuccess) {
    GemmArgs g = layer(B, O, H, n->a2, n->w16 + n->o16_w3, n->p + n->off_b3, n->dy);
    g.target = T;
    g.mask = mask;
    g.inv_norm = (float)(1.0 / norm);
    g.loss = n->loss;
    e = gemm<true, kLoss>(g, st);
  }
  if (e == cudaSuccess) e = input_grad(B, O, H, n->dy, n->w16 + n->o16_w3, n->z2, n->d2, st);
  if (e == cudaSuccess) e = input_grad(B, H, H, n->d2, n->w16 + n->o16_w2, n->z1, n->d1, st);
  if (e == cudaSuccess) e = weight_grads(n, B, X, st);
  if (e == cudaSuccess && loss_host) {
    e = cudaMemcpyAsync(loss_host, n->loss, sizeof(float), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  return st_of(e);
}

fock_status fock_mlp_step(fock_mlp *n, float lr, float beta1, float beta2, float eps, float weight_decay,
                          cudaStream_t st) {
  if (!n || !(lr >= 0.0f)) return FOCK_ERR_INVALID_ARG;
  n->step += 1;
  const float c1 = (float)(1.0 / (1.0 - pow((double)beta1, (double)n->step)));
  const float c2 = (float)(1.0 / (1.0 - pow((double)beta2, (double)n->step)));
  k_adam<<<blocks_for((long long)n->nparam), 256, 0, st>>>((long long)n->nparam, n->p, n->g, n->m, n->v, n->w16,
                                                           bf16_map(n), lr, beta1, beta2, eps, weight_decay, c1, c2);
  return st_of(cudaGetLastError());
}

fock_status fock_mlp_zero_grad(fock_mlp *n, cudaStream_t st) {
  if (!n) return FOCK_ERR_INVALID_ARG;
  return st_of(cudaMemsetAsync(n->g, 0, sizeof(float) * n->nparam, st));
}

}  // extern "C"
