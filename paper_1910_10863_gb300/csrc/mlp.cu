// Learned warm start for GMRES: a small MLP predicts, from (kH, theta, fiber
// centres and radii), the low Fourier modes of both densities on every fiber;
// decoding them at the element angles gives an initial guess Psi_0.  The
// network is trained on solutions the solver itself produces.  Forward,
// backward and Adam run in the kernels below (FP32).
//
// Layers: in -> hidden (GELU) x layers -> out (linear).  Parameters are one
// flat FP32 array: for every layer W [out][in] row-major, then b [out].
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "internal.h"

struct pfmbem_mlp {
  int in = 0, hidden = 0, layers = 0, out = 0;
  cudaStream_t stream = nullptr;
  int dev = 0;                     // device current at create
  std::vector<int> dims;           // layer widths: in, hidden..., out
  std::vector<size_t> woff, boff;  // offsets of W and b of each layer in params
  size_t nparams = 0;
  float* params = nullptr;
  float* grad = nullptr;
  float* m1 = nullptr;             // Adam first moment
  float* m2 = nullptr;             // Adam second moment
  int64_t step = 0;
  int cap = 0;                     // batch capacity of the work buffers
  std::vector<float*> act;         // activations per layer boundary [cap][dims[l]] (0: a host batch; the last:
                                   // the output, or a host batch's targets in training)
  std::vector<float*> pre;         // pre-activations per hidden layer
  float* dA = nullptr;             // work: gradient w.r.t. pre-activations, two in turn
  float* dB = nullptr;
  float* loss = nullptr;           // device scalar
};

namespace {

// ------------------------------------------------------------ FP32 products
// Every pass of the network is a product C[M][N] = sum_k A(m, k) B(k, n) whose
// operands lie along k ([m][k], [n][k]: AK, BK) or across it ([k][m], [k][n]):
//   forward  Z = X W^T       AK, BK    bias and GELU (or the loss) in the epilogue
//   dX       dZ W            AK, !BK   GELU' in the epilogue: the next layer's dZ
//   dW       dZ^T X          !AK, !BK  the bias gradient from the staged dZ tile
// The layers are small (256 x 256 at K = 256 and a batch of 256): what bounds them
// is latency, so each pass is one launch with everything elementwise in it, and a
// small tile (32 x 32, eight groups of 64 threads sharing each K stage of 128) keeps
// the chain short on the 64 blocks such a layer has; a tile of 64 x 64 with the
// block's threads over the outputs alone takes over where it fills the chip by
// itself (BIG_TILES).  4 x 4 outputs per thread: a 16 x 32 tile with 1 x 4 was bound
// by its shared-memory reads (20 against 15 us for 256 x 1088 at K = 256).  All loads
// of a stage are issued before the previous stage's arithmetic.  FP32 FMA
// throughout; the groups' sums are added in a fixed order.
// Measured at 50 -> 3 x 256 -> 1088: a training step of 256 rows 354 -> 128 us (16 x 16
// tiles, one output per thread, bias, GELU, loss and column sums as launches of their
// own: 26 launches, now 9), then 102 with 4 x 4 outputs a thread; a forward pass of 1024
// rows 215 -> 57 us.
struct Mat {
  const float* A;
  const float* B;
  int M, N, K, lda, ldb;
};

// Element e of a [TK][T] tile staged from an operand along k (KM) or across it: a
// warp covers 8 k x 4 rows (32-byte sectors; with a row stride of 4 mod 32 words, 36 or
// 68 here, its stores meet 32 different banks), or rows one after another.
template <bool KM, int T>
__device__ __forceinline__ void tile_at(int e, int& k, int& m) {
  if (KM) {
    const int r = e >> 5;
    m = ((e >> 3) & 3) + 4 * (r % (T / 4));
    k = (e & 7) + 8 * (r / (T / 4));
  } else {
    m = e % T;
    k = e / T;
  }
}

template <bool KM, int T, int TK, int NT>
struct Stage {
  static constexpr int NV = T * TK / NT;
  float v[NV];
  __device__ __forceinline__ void load(const float* __restrict__ P, int ld, int m0, int k0, int M, int K) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      int k, m;
      tile_at<KM, T>((int)threadIdx.x + i * NT, k, m);
      k += k0;
      m += m0;
      v[i] = k < K && m < M ? __ldg(P + (KM ? (size_t)m * ld + k : (size_t)k * ld + m)) : 0.f;
    }
  }
  __device__ __forceinline__ void store(float* s) const {       // [TK][T + 4]
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      int k, m;
      tile_at<KM, T>((int)threadIdx.x + i * NT, k, m);
      s[k * (T + 4) + m] = v[i];
    }
  }
};

constexpr int SM_T = 32, SN_T = 32, SK_T = 128, SNT = 512;       // small tile
constexpr int SGRP = SNT / 64;                                   // shares of its K stage
constexpr int S_SMEM = SK_T * (SM_T + 4 + SN_T + 4);             // floats
constexpr int L_T = 64, LK_T = 32, LNT = 256;                    // large tile
// Large tiles from which it is taken: at 64, 128, 256 and never a forward pass to 1088 outputs takes
// 66, 57, 58, 68 us at 1024 rows and 86, 86, 98, 115 at 2048, a training step 270, 205, 206, 218 and
// 354, 354, 334, 354 us.
constexpr int BIG_TILES = 128;

// Small tile: out(m, n, value) for every entry of the tile at (m0, n0), n along the
// lanes.  64 threads of 4 x 4 outputs hold the tile; SGRP such groups share every K
// stage.  rowsum (if not null): sum_k A(m, k), m = m0 ..
template <bool AK, bool BK, class Out>
__device__ __forceinline__ void small_tile(const Mat& g, int m0, int n0, float* sm, float* rowsum, Out out) {
  float* sA = sm;
  float* sB = sm + SK_T * (SM_T + 4);
  Stage<AK, SM_T, SK_T, SNT> a;
  Stage<BK, SN_T, SK_T, SNT> b;
  const int t = threadIdx.x, grp = t >> 6, r = 4 * ((t & 63) >> 3), c = 4 * (t & 7);
  float acc[4][4], rs = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  a.load(g.A, g.lda, m0, 0, g.M, g.K);
  b.load(g.B, g.ldb, n0, 0, g.N, g.K);
  for (int k0 = 0; k0 < g.K; k0 += SK_T) {
    __syncthreads();
    a.store(sA);
    b.store(sB);
    __syncthreads();
    if (k0 + SK_T < g.K) {
      a.load(g.A, g.lda, m0, k0 + SK_T, g.M, g.K);
      b.load(g.B, g.ldb, n0, k0 + SK_T, g.N, g.K);
    }
    const float* pa = sA + (grp * (SK_T / SGRP)) * (SM_T + 4) + r;
    const float* pb = sB + (grp * (SK_T / SGRP)) * (SN_T + 4) + c;
#pragma unroll 8
    for (int k = 0; k < SK_T / SGRP; ++k) {
      const float4 av = *reinterpret_cast<const float4*>(pa + k * (SM_T + 4));
      const float4 bv = *reinterpret_cast<const float4*>(pb + k * (SN_T + 4));
      const float ax[4] = {av.x, av.y, av.z, av.w}, bx[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ax[i], bx[j], acc[i][j]);
    }
    if (rowsum)
#pragma unroll
      for (int k = 0; k < SK_T / 16; ++k) rs += sA[((t >> 5) * (SK_T / 16) + k) * (SM_T + 4) + (t & 31)];
  }
  __syncthreads();
  float* red = sm;                                     // [SGRP][32][32], then [16][32]
#pragma unroll
  for (int i = 0; i < 4; ++i)
    *reinterpret_cast<float4*>(red + (grp * SM_T + r + i) * SN_T + c) =
        make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  float* red2 = sm + SGRP * SM_T * SN_T;
  if (rowsum) red2[t] = rs;                            // [t >> 5][t & 31]
  __syncthreads();
#pragma unroll
  for (int h = 0; h < SM_T * SN_T / SNT; ++h) {
    const int i = t + h * SNT, m = i >> 5, n = i & 31;
    if (m0 + m < g.M && n0 + n < g.N) {
      float v = 0.f;
#pragma unroll
      for (int q = 0; q < SGRP; ++q) v += red[q * SM_T * SN_T + i];
      out(m0 + m, n0 + n, v);
    }
  }
  if (rowsum && t < SM_T && m0 + t < g.M) {
    float v = 0.f;
    for (int i = 0; i < 16; ++i) v += red2[i * SM_T + t];
    rowsum[m0 + t] = v;
  }
}

template <bool AK, bool BK, class Out>
__device__ __forceinline__ void large_tile(const Mat& g, int m0, int n0, float* sm, Out out) {
  float* sA = sm;
  float* sB = sm + LK_T * (L_T + 4);
  Stage<AK, L_T, LK_T, LNT> a;
  Stage<BK, L_T, LK_T, LNT> b;
  const int t = threadIdx.x, r = 4 * (t >> 4), c = 4 * (t & 15);
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  a.load(g.A, g.lda, m0, 0, g.M, g.K);
  b.load(g.B, g.ldb, n0, 0, g.N, g.K);
  for (int k0 = 0; k0 < g.K; k0 += LK_T) {
    __syncthreads();
    a.store(sA);
    b.store(sB);
    __syncthreads();
    if (k0 + LK_T < g.K) {
      a.load(g.A, g.lda, m0, k0 + LK_T, g.M, g.K);
      b.load(g.B, g.ldb, n0, k0 + LK_T, g.N, g.K);
    }
#pragma unroll 8
    for (int k = 0; k < LK_T; ++k) {
      const float4 av = *reinterpret_cast<const float4*>(sA + k * (L_T + 4) + r);
      const float4 bv = *reinterpret_cast<const float4*>(sB + k * (L_T + 4) + c);
      const float ax[4] = {av.x, av.y, av.z, av.w}, bx[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ax[i], bx[j], acc[i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (m0 + r + i < g.M && n0 + c + j < g.N) out(m0 + r + i, n0 + c + j, acc[i][j]);
}

// The block's tile of a product of tm x tn tiles, m fastest.
template <bool BIG, bool AK, bool BK, class Out>
__device__ __forceinline__ void tile(const Mat& g, int b, float* sm, float* rowsum, Out out) {
  constexpr int TM = BIG ? L_T : SM_T, TN = BIG ? L_T : SN_T;
  const int tm = (g.M + TM - 1) / TM, mi = b % tm, ni = b / tm;
  if constexpr (BIG)
    large_tile<AK, BK>(g, mi * TM, ni * TN, sm, out);
  else
    small_tile<AK, BK>(g, mi * TM, ni * TN, sm, ni == 0 ? rowsum : nullptr, out);
}

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x) {
  return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// One forward layer: z = X W^T + bias; hidden layers write gelu(z) to Y and, for a
// training pass, z to Z; the output layer writes z to Y or, with targets, the
// gradient of the mean-squared error 2 (z - T) scale to Y and adds (z - T)^2 scale
// to the loss.  clear: the loss, cleared by the first layer's first block.
template <bool BIG>
__global__ void __launch_bounds__(BIG ? LNT : SNT, 2) layer_kernel(const Mat g, const float* __restrict__ bias,
                                                                int hidden, float* __restrict__ Z,
                                                                float* __restrict__ Y, const float* __restrict__ T,
                                                                float scale, float* loss, float* clear) {
  __shared__ __align__(16) float sm[S_SMEM];
  __shared__ float red[SNT / 32];
  if (clear && blockIdx.x == 0 && threadIdx.x == 0) *clear = 0.f;
  float l = 0.f;
  tile<BIG, true, true>(g, blockIdx.x, sm, nullptr, [&](int m, int n, float v) {
    const float z = v + bias[n];
    const size_t i = (size_t)m * g.N + n;
    if (hidden) {
      if (Z) Z[i] = z;
      Y[i] = gelu(z);
    } else if (T) {
      const float d = z - T[i];
      Y[i] = 2.f * d * scale;
      l += d * d * scale;
    } else {
      Y[i] = z;
    }
  });
  if (!T || hidden) return;
  for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = l;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < (int)(blockDim.x >> 5); ++i) l += red[i];
    atomicAdd(loss, l);
  }
}

// One backward layer in one launch: the first ndx blocks form dX = dZ W times
// GELU'(Z) of the layer below (its dZ), the others dW = dZ^T X and the bias
// gradient, the column sums of dZ.
__global__ void __launch_bounds__(SNT, 2) back_kernel(const Mat dx, int ndx, const float* __restrict__ Zb,
                                                   float* __restrict__ dZb, const Mat dw, float* __restrict__ gw,
                                                   float* __restrict__ gb) {
  __shared__ __align__(16) float sm[S_SMEM];
  if ((int)blockIdx.x < ndx) {
    tile<false, true, false>(dx, blockIdx.x, sm, nullptr, [&](int m, int n, float v) {
      const size_t i = (size_t)m * dx.N + n;
      dZb[i] = v * gelu_grad(Zb[i]);
    });
  } else {
    tile<false, false, false>(dw, blockIdx.x - ndx, sm, gb,
                              [&](int m, int n, float v) { gw[(size_t)m * dw.N + n] = v; });
  }
}

__global__ void __launch_bounds__(LNT) back_dx_kernel(const Mat dx, const float* __restrict__ Zb,
                                                      float* __restrict__ dZb) {
  __shared__ __align__(16) float sm[2 * LK_T * (L_T + 4)];
  tile<true, true, false>(dx, blockIdx.x, sm, nullptr, [&](int m, int n, float v) {
    const size_t i = (size_t)m * dx.N + n;
    dZb[i] = v * gelu_grad(Zb[i]);
  });
}

__global__ void adam_kernel(size_t n, float lr, float b1, float b2, float eps, float c1, float c2,
                            float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
}

// counter-based uniform in (-1, 1) from (seed, index): SplitMix64
__global__ void init_kernel(size_t n, uint64_t seed, const int64_t* __restrict__ fan_in_of, float* __restrict__ p) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint64_t z = seed + 0x9E3779B97F4A7C15ull * (i + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  const float u = (float)((z >> 11) * (1.0 / 9007199254740992.0)) * 2.f - 1.f;
  const int64_t fi = fan_in_of[i];
  p[i] = fi > 0 ? u * sqrtf(3.f / (float)fi) : 0.f;   // Var = 1/fan_in, biases zero
}

int tiles(int M, int N, int TM, int TN) { return ((M + TM - 1) / TM) * ((N + TN - 1) / TN); }

cudaError_t ensure_cap(pfmbem_mlp* m, int B) {
  if (B <= m->cap) return cudaSuccess;
  for (float* p : m->act) cudaFree(p);
  for (float* p : m->pre) cudaFree(p);
  cudaFree(m->dA);
  cudaFree(m->dB);
  m->dA = m->dB = nullptr;
  m->cap = 0;
  m->act.assign(m->dims.size(), nullptr);
  m->pre.assign(m->dims.size(), nullptr);
  int wmax = 0;
  for (int d : m->dims) wmax = d > wmax ? d : wmax;
  for (size_t l = 0; l < m->dims.size(); ++l) {
    if (cudaMalloc(&m->act[l], sizeof(float) * (size_t)B * m->dims[l]) != cudaSuccess) return cudaErrorMemoryAllocation;
    if (cudaMalloc(&m->pre[l], sizeof(float) * (size_t)B * m->dims[l]) != cudaSuccess) return cudaErrorMemoryAllocation;
  }
  if (cudaMalloc(&m->dA, sizeof(float) * (size_t)B * wmax) != cudaSuccess) return cudaErrorMemoryAllocation;
  if (cudaMalloc(&m->dB, sizeof(float) * (size_t)B * wmax) != cudaSuccess) return cudaErrorMemoryAllocation;
  m->cap = B;
  return cudaSuccess;
}

// Forward pass from X to Y ([B][out]).  With targets T, Y receives the gradient of
// the loss instead, m->loss the loss, and the pre-activations are kept.
void forward(pfmbem_mlp* m, int B, const float* X, float* Y, const float* T) {
  const int L = (int)m->dims.size() - 1;
  const float scale = 1.f / (float)((size_t)B * m->out);
  for (int l = 0; l < L; ++l) {
    const int I = m->dims[l], O = m->dims[l + 1], hidden = l < L - 1;
    const Mat g{l == 0 ? X : m->act[l], m->params + m->woff[l], B, O, I, I, I};
    float* y = hidden ? m->act[l + 1] : Y;
    float* z = hidden && T ? m->pre[l + 1] : nullptr;
    float* clear = T && l == 0 ? m->loss : nullptr;
    const int nb = tiles(B, O, L_T, L_T);
    if (nb >= BIG_TILES)
      layer_kernel<true><<<nb, LNT, 0, m->stream>>>(g, m->params + m->boff[l], hidden, z, y, T, scale, m->loss, clear);
    else
      layer_kernel<false><<<tiles(B, O, SM_T, SN_T), SNT, 0, m->stream>>>(g, m->params + m->boff[l], hidden, z, y, T,
                                                                          scale, m->loss, clear);
  }
}

// Backward pass from the loss gradient in m->dA ([B][out]); writes grad.
void backward(pfmbem_mlp* m, int B, const float* X, float* grad) {
  const int L = (int)m->dims.size() - 1;
  float* dcur = m->dA;   // gradient w.r.t. pre-activation of layer l+1
  float* dnext = m->dB;
  for (int l = L - 1; l >= 0; --l) {
    const int I = m->dims[l], O = m->dims[l + 1];
    const Mat dx{dcur, m->params + m->woff[l], B, I, O, O, I};
    const Mat dw{dcur, l == 0 ? X : m->act[l], O, I, B, O, I};
    const int nbig = l > 0 ? tiles(B, I, L_T, L_T) : 0;
    const bool big = nbig >= BIG_TILES;
    if (big) back_dx_kernel<<<nbig, LNT, 0, m->stream>>>(dx, m->pre[l], dnext);
    const int ndx = l > 0 && !big ? tiles(B, I, SM_T, SN_T) : 0;
    back_kernel<<<ndx + tiles(O, I, SM_T, SN_T), SNT, 0, m->stream>>>(dx, ndx, l > 0 ? m->pre[l] : nullptr, dnext, dw,
                                                                      grad + m->woff[l], grad + m->boff[l]);
    float* t = dcur;
    dcur = dnext;
    dnext = t;
  }
}

bool is_dev(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Memory that the network's kernels may read and write in place: its own device's, aligned
// to its floats (another device's, or at an odd byte, is copied, as host memory is).
bool is_local(const pfmbem_mlp* m, const void* p) {
  if (reinterpret_cast<uintptr_t>(p) % alignof(float) != 0) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice && a.device == m->dev;
}

cudaError_t copy_in(pfmbem_mlp* m, float* dst, const float* src, size_t n) {
  return cudaMemcpyAsync(dst, src, n * sizeof(float), is_dev(src) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                         m->stream);
}

// ---------------------------------------------------------------- features
// x = [kH / 8, theta / (pi/2), then per fiber ((cx - x0)/H, (cy - y0)/H, 4 r / H)]
__global__ void features_kernel(int M, float kH, float th, const double* __restrict__ fc, double x0, double y0,
                                double H, float* __restrict__ x) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    x[0] = kH / 8.f;
    x[1] = th / 1.5707963267948966f;
  }
  if (i < M) {
    x[2 + 3 * i] = (float)((fc[3 * i] - x0) / H);
    x[3 + 3 * i] = (float)((fc[3 * i + 1] - y0) / H);
    x[4 + 3 * i] = (float)(4.0 * fc[3 * i + 2] / H);
  }
}

// Per-fiber network input (one row per fiber, 5 + 3K floats): kH/8,
// theta/(pi/2), 4 r_i/H, the distances (x_i - x_min)/H and (x_max - x_i)/H to
// the block's left and right edges, then the K nearest other fibers in order of
// distance, each as (4 dx/H, 4 dy/H, 4 r_j/H) with dy taken to the nearest
// periodic image; missing neighbours are zeros.  The row depends on positions
// only through differences along y, so a model on these rows is equivariant
// under shifts of the block along the period.  One thread per fiber.
#define PF_WARM_KMAX 32
__global__ void features_local_kernel(int M, int K, float kH, float th, const double* __restrict__ fc, double H,
                                      float* __restrict__ x) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M) return;
  const double cx = fc[3 * i], cy = fc[3 * i + 1], ri = fc[3 * i + 2];
  double xmin = 1e300, xmax = -1e300;
  for (int j = 0; j < M; ++j) {
    xmin = fmin(xmin, fc[3 * j] - fc[3 * j + 2]);
    xmax = fmax(xmax, fc[3 * j] + fc[3 * j + 2]);
  }
  double bd[PF_WARM_KMAX];
  int bj[PF_WARM_KMAX];
  double bdy[PF_WARM_KMAX];
  int nb = 0;
  for (int j = 0; j < M; ++j) {
    if (j == i) continue;
    const double dx = fc[3 * j] - cx;
    double dy = fc[3 * j + 1] - cy;
    dy -= H * rint(dy / H);
    const double d2 = dx * dx + dy * dy;
    // insertion into the K nearest so far
    int pos = nb < K ? nb : K;
    while (pos > 0 && bd[pos - 1] > d2) {
      if (pos < K) { bd[pos] = bd[pos - 1]; bj[pos] = bj[pos - 1]; bdy[pos] = bdy[pos - 1]; }
      --pos;
    }
    if (pos < K) {
      bd[pos] = d2;
      bj[pos] = j;
      bdy[pos] = dy;
      if (nb < K) ++nb;
    }
  }
  float* o = x + (size_t)i * (5 + 3 * K);
  o[0] = kH / 8.f;
  o[1] = th / 1.5707963267948966f;
  o[2] = (float)(4.0 * ri / H);
  o[3] = (float)((cx - xmin) / H);
  o[4] = (float)((xmax - cx) / H);
  for (int q = 0; q < K; ++q) {
    float* v = o + 5 + 3 * q;
    if (q < nb) {
      const int j = bj[q];
      v[0] = (float)(4.0 * (fc[3 * j] - cx) / H);
      v[1] = (float)(4.0 * bdy[q] / H);
      v[2] = (float)(4.0 * fc[3 * j + 2] / H);
    } else {
      v[0] = v[1] = v[2] = 0.f;
    }
  }
}

// Fourier coefficients of a solution: for fiber i, density d, mode n = -8..8,
//   c = (1/N_i) sum_e psi_{e,d} e^{-i n t_e} e^{-i k c_i.dir},
// t_e = angle of c_e about c_i measured from the incidence direction, so that an
// isolated circle's response has the same coefficients at every incidence angle.
// One block per (fiber, density); threads over modes.
__global__ void targets_kernel(int M, int nm, const int* __restrict__ foff, const double* __restrict__ fc,
                               const double2* __restrict__ oc, double k, double dx, double dy,
                               const cplx* __restrict__ psi, float* __restrict__ t) {
  const int i = blockIdx.x >> 1, d = blockIdx.x & 1;
  const int n = (int)threadIdx.x - nm;
  if (threadIdx.x >= 2 * nm + 1) return;
  const int f0 = foff[i], N = foff[i + 1] - f0;
  const double cx = fc[3 * i], cy = fc[3 * i + 1];
  cplx acc{0, 0};
  for (int e = f0; e < f0 + N; ++e) {
    // angle of (c_e - c_i) relative to dir = (dx, dy)
    const double ux = oc[e].x - cx, uy = oc[e].y - cy;
    const double te = atan2(uy * dx - ux * dy, ux * dx + uy * dy);
    double s, c;
    sincos(-n * te, &s, &c);
    acc += psi[2 * e + d] * cplx{c, s};
  }
  double s, c;
  sincos(-k * (cx * dx + cy * dy), &s, &c);
  acc = (1.0 / N) * (acc * cplx{c, s});
  const size_t o = (((size_t)i * 2 + d) * (2 * nm + 1) + (n + nm)) * 2;
  t[o] = (float)acc.re;
  t[o + 1] = (float)acc.im;
}

// psi0_{e,d} = e^{i k c_i.dir} sum_n c_{i,d,n} e^{i n t_e} (t_e as above); one thread per element.
__global__ void decode_kernel(int E, int nm, const int* __restrict__ fib, const double* __restrict__ fc,
                              const double2* __restrict__ oc, double k, double dx, double dy,
                              const float* __restrict__ y, cplx* __restrict__ psi) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  const int i = fib[e];
  const double cx = fc[3 * i], cy = fc[3 * i + 1];
  const double ux = oc[e].x - cx, uy = oc[e].y - cy;
  const double te = atan2(uy * dx - ux * dy, ux * dx + uy * dy);
  double s, c;
  sincos(k * (cx * dx + cy * dy), &s, &c);
  const cplx ph{c, s};
  for (int d = 0; d < 2; ++d) {
    cplx acc{0, 0};
    for (int n = -nm; n <= nm; ++n) {
      const size_t o = (((size_t)i * 2 + d) * (2 * nm + 1) + (n + nm)) * 2;
      double sn, cn;
      sincos(n * te, &sn, &cn);
      acc += cplx{(double)y[o], (double)y[o + 1]} * cplx{cn, sn};
    }
    psi[2 * e + d] = ph * acc;
  }
}

}  // namespace

// ====================================================================== C ABI
extern "C" {

pfmbem_status pfmbem_mlp_create(int in, int hidden, int layers, int out, uint64_t seed, void* stream,
                                pfmbem_mlp_t* res) {
  if (!res || in < 1 || hidden < 1 || layers < 1 || out < 1 || layers > 16) return PFMBEM_EINVAL;
  *res = nullptr;
  pfmbem_mlp* m = new pfmbem_mlp();
  m->in = in;
  m->hidden = hidden;
  m->layers = layers;
  m->out = out;
  m->stream = static_cast<cudaStream_t>(stream);
  cudaGetDevice(&m->dev);
  m->dims.push_back(in);
  for (int l = 0; l < layers; ++l) m->dims.push_back(hidden);
  m->dims.push_back(out);
  size_t off = 0;
  std::vector<int64_t> fan;
  for (size_t l = 0; l + 1 < m->dims.size(); ++l) {
    const size_t nw = (size_t)m->dims[l] * m->dims[l + 1];
    m->woff.push_back(off);
    off += nw;
    m->boff.push_back(off);
    off += m->dims[l + 1];
    fan.insert(fan.end(), nw, m->dims[l]);
    fan.insert(fan.end(), m->dims[l + 1], 0);
  }
  m->nparams = off;
  int64_t* fan_d = nullptr;
  if (cudaMalloc(&m->params, off * sizeof(float)) != cudaSuccess || cudaMalloc(&m->grad, off * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&m->m1, off * sizeof(float)) != cudaSuccess || cudaMalloc(&m->m2, off * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&fan_d, off * sizeof(int64_t)) != cudaSuccess) {
    pfmbem_mlp_destroy(m);
    return PFMBEM_ENOMEM;
  }
  cudaMemcpyAsync(fan_d, fan.data(), off * sizeof(int64_t), cudaMemcpyHostToDevice, m->stream);
  init_kernel<<<(unsigned)((off + 255) / 256), 256, 0, m->stream>>>(off, seed, fan_d, m->params);
  cudaMemsetAsync(m->m1, 0, off * sizeof(float), m->stream);
  cudaMemsetAsync(m->m2, 0, off * sizeof(float), m->stream);
  cudaStreamSynchronize(m->stream);
  cudaFree(fan_d);
  if (cudaMalloc(&m->loss, sizeof(float)) != cudaSuccess) {
    pfmbem_mlp_destroy(m);
    return PFMBEM_ENOMEM;
  }
  if (cudaGetLastError() != cudaSuccess) {
    pfmbem_mlp_destroy(m);
    return PFMBEM_ECUDA;
  }
  *res = m;
  return PFMBEM_OK;
}

void pfmbem_mlp_destroy(pfmbem_mlp_t m) {
  if (!m) return;
  cudaStreamSynchronize(m->stream);
  cudaFree(m->params);
  cudaFree(m->grad);
  cudaFree(m->m1);
  cudaFree(m->m2);
  cudaFree(m->loss);
  for (float* p : m->act) cudaFree(p);
  for (float* p : m->pre) cudaFree(p);
  cudaFree(m->dA);
  cudaFree(m->dB);
  delete m;
}

pfmbem_status pfmbem_mlp_params(pfmbem_mlp_t m, int64_t* nparams, float* get, const float* set) {
  if (!m || !nparams) return PFMBEM_EINVAL;
  *nparams = (int64_t)m->nparams;
  if (set && copy_in(m, m->params, set, m->nparams) != cudaSuccess) return PFMBEM_ECUDA;
  if (get) {
    if (cudaMemcpyAsync(get, m->params, m->nparams * sizeof(float),
                        is_dev(get) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, m->stream) != cudaSuccess)
      return PFMBEM_ECUDA;
  }
  return cudaStreamSynchronize(m->stream) == cudaSuccess ? PFMBEM_OK : PFMBEM_ECUDA;
}

pfmbem_status pfmbem_mlp_forward(pfmbem_mlp_t m, int B, const float* X, float* Y) {
  if (!m || B < 1 || !X || !Y) return PFMBEM_EINVAL;
  if (ensure_cap(m, B) != cudaSuccess) return PFMBEM_ENOMEM;
  // batches on the device are read and written in place, in the stream's order
  // (an input that overlaps the output is copied first)
  const bool ydev = is_dev(Y), yin = is_local(m, Y);
  if (!is_local(m, X) || (yin && X < Y + (size_t)B * m->out && Y < X + (size_t)B * m->in)) {
    if (copy_in(m, m->act[0], X, (size_t)B * m->in) != cudaSuccess) return PFMBEM_ECUDA;
    X = m->act[0];
  }
  forward(m, B, X, yin ? Y : m->act.back(), nullptr);
  if (!yin && cudaMemcpyAsync(Y, m->act.back(), sizeof(float) * (size_t)B * m->out,
                              ydev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, m->stream) != cudaSuccess)
    return PFMBEM_ECUDA;
  if (!ydev && cudaStreamSynchronize(m->stream) != cudaSuccess) return PFMBEM_ECUDA;
  return cudaGetLastError() == cudaSuccess ? PFMBEM_OK : PFMBEM_ECUDA;
}

// Mean-squared error over the batch and, if grad != NULL, its gradient with
// respect to every parameter (flat layout); lr > 0 additionally takes one Adam
// step (beta1 0.9, beta2 0.999, eps 1e-8).
pfmbem_status pfmbem_mlp_train(pfmbem_mlp_t m, int B, const float* X, const float* T, float lr, float* loss,
                               float* grad) {
  if (!m || B < 1 || !X || !T) return PFMBEM_EINVAL;
  if (ensure_cap(m, B) != cudaSuccess) return PFMBEM_ENOMEM;
  // a batch on the device is read, and a gradient there written, in place (the
  // call waits for the stream at its end)
  if (!is_local(m, X)) {
    if (copy_in(m, m->act[0], X, (size_t)B * m->in) != cudaSuccess) return PFMBEM_ECUDA;
    X = m->act[0];
  }
  if (!is_local(m, T)) {
    // (a training pass leaves the output's place free: it writes the loss gradient to dA)
    if (copy_in(m, m->act.back(), T, (size_t)B * m->out) != cudaSuccess) return PFMBEM_ECUDA;
    T = m->act.back();
  }
  float* g = m->grad;
  if (grad && is_local(m, grad)) {
    // (a gradient that shares memory with the batch is copied out at the end)
    auto apart = [&](const float* p, size_t n) { return p + n <= grad || grad + m->nparams <= p; };
    if (apart(X, (size_t)B * m->in) && apart(T, (size_t)B * m->out)) g = grad;
  }
  forward(m, B, X, m->dA, T);
  backward(m, B, X, g);
  if (lr > 0) {
    m->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f / (1.f - (float)std::pow(b1, (double)m->step));
    const float c2 = 1.f / (1.f - (float)std::pow(b2, (double)m->step));
    adam_kernel<<<(unsigned)((m->nparams + 255) / 256), 256, 0, m->stream>>>(m->nparams, lr, b1, b2, 1e-8f, c1, c2,
                                                                            m->params, g, m->m1, m->m2);
  }
  if (grad && g != grad &&
      cudaMemcpyAsync(grad, g, m->nparams * sizeof(float),
                      is_dev(grad) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, m->stream) != cudaSuccess)
    return PFMBEM_ECUDA;
  if (loss && cudaMemcpyAsync(loss, m->loss, sizeof(float), cudaMemcpyDeviceToHost, m->stream) != cudaSuccess)
    return PFMBEM_ECUDA;
  if (cudaStreamSynchronize(m->stream) != cudaSuccess) return PFMBEM_ECUDA;
  return cudaGetLastError() == cudaSuccess ? PFMBEM_OK : PFMBEM_ECUDA;
}

}  // extern "C"

// ---------------------------------------------------------------- handle side
cudaError_t k_warm_features(pfmbem* h, float* x_dev) {
  features_kernel<<<(h->M + 127) / 128, 128, 0, h->stream>>>(h->M, (float)(h->k * h->H), (float)h->theta, h->fib_geo,
                                                             h->x0, h->y0, h->H, x_dev);
  return cudaGetLastError();
}

cudaError_t k_warm_features_local(pfmbem* h, int K, float* x_dev) {
  features_local_kernel<<<(h->M + 127) / 128, 128, 0, h->stream>>>(h->M, K, (float)(h->k * h->H), (float)h->theta,
                                                                   h->fib_geo, h->H, x_dev);
  return cudaGetLastError();
}

cudaError_t k_warm_targets(pfmbem* h, int nm, const cplx* psi, float* t_dev) {
  targets_kernel<<<2 * h->M, 32 * ((2 * nm + 1 + 31) / 32), 0, h->stream>>>(h->M, nm, h->fib_off, h->fib_geo, h->o_c, h->k,
                                                                              cos(h->theta), sin(h->theta), psi, t_dev);
  return cudaGetLastError();
}

cudaError_t k_warm_decode(pfmbem* h, int nm, const float* y_dev, cplx* psi) {
  decode_kernel<<<(h->E + 127) / 128, 128, 0, h->stream>>>(h->E, nm, h->o_fiber, h->fib_geo, h->o_c, h->k,
                                                          cos(h->theta), sin(h->theta), y_dev, psi);
  return cudaGetLastError();
}
