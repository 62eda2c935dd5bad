// The learned slice-count predictor: block features, a 16 -> 64 -> 64 -> 8
// MLP (FP32, ReLU, softmax over slice counts 1..8) with hand-written forward,
// backward and Adam kernels, and the label generator (per-block K error of
// the emulated build at every slice count against the native FP64 build).
//
// Parameter layout (one float buffer, row-major weights, y = W x + b):
//   W1 [64][16], b1 [64], W2 [64][64], b2 [64], W3 [8][64], b3 [8].
#include "df_ctx.h"

#include <cooperative_groups.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

namespace {

namespace cg = cooperative_groups;

constexpr int kIn = 16, kH = 64, kOut = 8;
constexpr int oW1 = 0, oB1 = oW1 + kH * kIn, oW2 = oB1 + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH,
              oB3 = oW3 + kOut * kH, kNParams = oB3 + kOut;
static_assert(kNParams == 5768, "parameter count");

// One warp per row: forward pass; optionally keeps activations for backward.
__device__ __forceinline__ void mlp_row_forward(const float *__restrict__ P, const float *x, float *h1, float *h2,
                                                float *z, int lane) {
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int j = lane + 32 * r;
    float a = P[oB1 + j];
#pragma unroll
    for (int k = 0; k < kIn; ++k) a = fmaf(P[oW1 + j * kIn + k], x[k], a);
    h1[j] = a > 0.f ? a : 0.f;
  }
  __syncwarp();
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int j = lane + 32 * r;
    float a = P[oB2 + j];
    for (int k = 0; k < kH; ++k) a = fmaf(P[oW2 + j * kH + k], h1[k], a);
    h2[j] = a > 0.f ? a : 0.f;
  }
  __syncwarp();
  if (lane < kOut) {
    float a = P[oB3 + lane];
    for (int k = 0; k < kH; ++k) a = fmaf(P[oW3 + lane * kH + k], h2[k], a);
    z[lane] = a;
  }
  __syncwarp();
}

__device__ __forceinline__ void softmax8(const float *z, float *p) {
  float m = z[0];
  for (int c = 1; c < kOut; ++c) m = fmaxf(m, z[c]);
  float s = 0.f;
  for (int c = 0; c < kOut; ++c) {
    p[c] = __expf(z[c] - m);
    s += p[c];
  }
  for (int c = 0; c < kOut; ++c) p[c] /= s;
}

constexpr int kRowsPerBlock = 8;

__global__ void __launch_bounds__(256) mlp_forward_kernel(const float *__restrict__ P, const float *__restrict__ X,
                                                          int n, float *__restrict__ probs) {
  __shared__ float sx[kRowsPerBlock][kIn], sh1[kRowsPerBlock][kH], sh2[kRowsPerBlock][kH], sz[kRowsPerBlock][kOut];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * kRowsPerBlock + w;
  if (row >= n) return;
  if (lane < kIn) sx[w][lane] = X[(long long)row * kIn + lane];
  __syncwarp();
  mlp_row_forward(P, sx[w], sh1[w], sh2[w], sz[w], lane);
  if (lane == 0) {
    float p[kOut];
    softmax8(sz[w], p);
    for (int c = 0; c < kOut; ++c) probs[(long long)row * kOut + c] = p[c];
  }
}

// Gradients of the summed cross-entropy (labels y in 0..7; the sum kernel divides by n).  A CTA takes tiles of
// 32 rows with the weights and the tile's activations in shared memory; every
// thread owns a fixed part of the gradient (16 entries of W2, 4 of W1, 2 of W3)
// and keeps it in registers over all its tiles, so a CTA writes one partial
// gradient and a second kernel adds the partials in order.  (A warp per row
// with an atomicAdd per entry and row, 40 million of them for 6992 rows, took
// 0.98 ms; the result is the same on every run.)
// A warp takes four rows of a tile through all the layers on its own; a lane holds two
// columns of the four rows, so an 8-byte load of weights (two wavefronts a warp) and four
// broadcast activations serve eight FMAs, and the warps meet only where the gradient sums
// over the tile's rows.  Weights are transposed on their way in by lanes along the other
// index, rows that eight lanes read side by side are a pitch of 68 apart.  (With a row and
// eight columns a thread, scalar accesses of stride 8 and block barriers between the layers
// a tile took 21.5 us, which made a step on one row slower, 32 us, than the kernel with
// the atomics, 20; now 8.7 and 18.5.)
constexpr int kTileRows = 32;
constexpr int kPart = kNParams + 1;  // a partial gradient and its part of the loss
// Partial gradients a network holds: with its parameters below 1 MB, up to which cudaMalloc
// takes 1.5 us and past which 55 (with 256 of them a network took 110 us to create, 40 before
// it held any).  More tiles than that run in clusters of 8 CTAs, each of which adds its
// CTAs' gradients through distributed shared memory and writes one partial.
constexpr int kOwnParts = 40;
constexpr int kCluster = 8;
// Clusters that get an SM to each CTA (the GPCs hold 15 of eight), and at most: a tile takes 14.4
// us in a cluster, another one of the same CTA 6.6 more, two CTAs on an SM 22.5 together and
// 3 a further one.  So two tiles to a CTA of 15 clusters (4600 rows: 20.9 us, in 18
// clusters 22.1), from 241 tiles on 32 clusters (8192 rows: 22.7 us, 27.6 in 15).
constexpr int kClustersAlone = 15;
constexpr int kMaxClusters = 32;
static_assert(kMaxClusters <= kOwnParts, "a partial gradient per cluster");
constexpr int kHP = kH + 4;       // activation pitch: rows of a tile on different banks, 16-byte aligned

struct alignas(16) MlpTile {
  float w1t[kIn][kH], w2t[kH][kH], w2[kH][kH], w3[kOut][kHP], b1[kH], b2[kH], b3[kOut];
  float x[kTileRows][kIn], h1[kTileRows][kHP], h2[kTileRows][kHP], d1[kTileRows][kHP], d2[kTileRows][kHP];
  float z[kTileRows][kOut], dz[kTileRows][kOut], loss[kTileRows];
};
static_assert(kPart <= kTileRows * (kIn + 4 * kHP), "a CTA's gradient takes the place of its activations");

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// a[i][.] += sum_k in[i][k] W[k][c .. c + 1] for four rows (k ascending).
template <int kK, int kPitchW, int kPitchIn>
__device__ __forceinline__ void layer4(float (&a)[4][2], const float *W, const float *in, int c) {
#pragma unroll 2
  for (int k = 0; k < kK; k += 4) {
    float v[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 u = ld4(in + i * kPitchIn + k);
      v[i][0] = u.x, v[i][1] = u.y, v[i][2] = u.z, v[i][3] = u.w;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float2 w = *reinterpret_cast<const float2 *>(W + (k + q) * kPitchW + c);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i][0] = fmaf(w.x, v[i][q], a[i][0]);
        a[i][1] = fmaf(w.y, v[i][q], a[i][1]);
      }
    }
  }
}

// out[i][c .. c + 1] = a[i][.] where the activation of the same place is positive, else 0.
__device__ __forceinline__ void put4(float *out, const float (&a)[4][2], const float *act, int c) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 t = act ? *reinterpret_cast<const float2 *>(act + i * kHP + c) : make_float2(a[i][0], a[i][1]);
    *reinterpret_cast<float2 *>(out + i * kHP + c) = make_float2(t.x > 0.f ? a[i][0] : 0.f, t.y > 0.f ? a[i][1] : 0.f);
  }
}

// kGroups: clusters of kCluster CTAs, one partial gradient each; else one a CTA.
template <bool kGroups>
__global__ void __launch_bounds__(256) mlp_backward_kernel(const float *__restrict__ P, const float *__restrict__ X,
                                                           const int *__restrict__ y, int n,
                                                           float *__restrict__ part) {
  extern __shared__ __align__(16) unsigned char mlp_smem[];
  MlpTile &s = *reinterpret_cast<MlpTile *>(mlp_smem);
  const int tid = threadIdx.x;
  {
    // lanes along the output index: the transposed stores are contiguous
    const int j = tid & 63, kq = (tid >> 6) * 4;
    const float4 u1 = ld4(P + oW1 + j * kIn + kq);
    float4 u2[4], u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      u2[i] = ld4(P + oW2 + j * kH + 16 * i + kq);
      u[i] = ld4(P + oW2 + 4 * (tid + 256 * i));
    }
    const float4 u3 = tid < kOut * kH / 4 ? ld4(P + oW3 + 4 * tid) : make_float4(0.f, 0.f, 0.f, 0.f);
    s.w1t[kq][j] = u1.x, s.w1t[kq + 1][j] = u1.y, s.w1t[kq + 2][j] = u1.z, s.w1t[kq + 3][j] = u1.w;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = 16 * i + kq;
      s.w2t[k][j] = u2[i].x, s.w2t[k + 1][j] = u2[i].y, s.w2t[k + 2][j] = u2[i].z, s.w2t[k + 3][j] = u2[i].w;
      *reinterpret_cast<float4 *>(&s.w2[0][0] + 4 * (tid + 256 * i)) = u[i];
    }
    if (tid < kOut * kH / 4) *reinterpret_cast<float4 *>(&s.w3[tid >> 4][4 * (tid & 15)]) = u3;
  }
  if (tid < kH) {
    s.b1[tid] = P[oB1 + tid];
    s.b2[tid] = P[oB2 + tid];
    if (tid < kOut) s.b3[tid] = P[oB3 + tid];
  }
  // activations: warp (rows r0 .. r0 + 3), lane (columns c0, c0 + 1); gradients: W2 block
  // (gj, gk) 4 x 4, W1 row w1j and 4 columns, W3 row w3c and 2 columns
  const int lane = tid & 31, r0 = (tid >> 5) * 4, c0 = 2 * lane;
  const int gj = (tid >> 4) * 4, gk = (tid & 15) * 4;
  const int w1j = tid >> 2, w1k = (tid & 3) * 4;
  const int w3c = tid >> 5, w3k = (tid & 31) * 2;
  float g2[4][4] = {}, g1[4] = {}, g3[2] = {}, gb = 0.f, loss = 0.f;
  const int ntiles = (n + kTileRows - 1) / kTileRows;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int row0 = tile * kTileRows, rows = min(kTileRows, n - row0);
    // the warp's rows of X (two values a lane) and, in lanes 0 to 3, a row's label
    const int xi = r0 * kIn + 2 * lane;
    const float x0 = xi < rows * kIn ? X[(long long)row0 * kIn + xi] : 0.f;
    const float x1 = xi < rows * kIn ? X[(long long)row0 * kIn + xi + 1] : 0.f;
    const bool valid = lane < 4 && r0 + lane < rows;
    const int yc = valid ? y[row0 + r0 + lane] : 0;
    __syncthreads();  // the weights are there; the tile before is used up
    (&s.x[0][0])[xi] = x0;
    (&s.x[0][0])[xi + 1] = x1;
    __syncwarp();
    float a[4][2];
    auto start = [&](const float *bias) {
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i][0] = bias ? bias[c0] : 0.f, a[i][1] = bias ? bias[c0 + 1] : 0.f;
    };
    start(s.b1);
    layer4<kIn, kH, kIn>(a, &s.w1t[0][0], s.x[r0], c0);
    put4(s.h1[r0], a, nullptr, c0);
    __syncwarp();
    start(s.b2);
    layer4<kH, kH, kHP>(a, &s.w2t[0][0], s.h1[r0], c0);
    put4(s.h2[r0], a, nullptr, c0);
    __syncwarp();
    {
      const int r = r0 + (lane >> 3), c = lane & 7;
      float v = s.b3[c];
#pragma unroll 4
      for (int k = 0; k < kH; k += 4) {
        const float4 w = ld4(&s.w3[c][k]), h = ld4(&s.h2[r][k]);
        v = fmaf(w.x, h.x, v);
        v = fmaf(w.y, h.y, v);
        v = fmaf(w.z, h.z, v);
        v = fmaf(w.w, h.w, v);
      }
      s.z[r][c] = v;
    }
    __syncwarp();
    if (lane < 4) {
      float p[kOut];
      softmax8(s.z[r0 + lane], p);
      float py = 0.f;
#pragma unroll
      for (int c = 0; c < kOut; ++c) {
        if (c == yc) py = p[c];
        s.dz[r0 + lane][c] = valid ? p[c] - (c == yc ? 1.f : 0.f) : 0.f;
      }
      if (valid) loss -= logf(fmaxf(py, 1e-30f));
    }
    __syncwarp();
    start(nullptr);
    layer4<kOut, kHP, kOut>(a, &s.w3[0][0], s.dz[r0], c0);
    put4(s.d2[r0], a, s.h2[r0], c0);
    __syncwarp();
    start(nullptr);
    layer4<kH, kH, kHP>(a, &s.w2[0][0], s.d2[r0], c0);
    put4(s.d1[r0], a, s.h1[r0], c0);
    __syncthreads();
    // rows past the end have dz = 0, so their d2 and d1 are zero
#pragma unroll 4
    for (int r = 0; r < kTileRows; ++r) {
      const float4 d = *reinterpret_cast<const float4 *>(&s.d2[r][gj]);
      const float4 h = *reinterpret_cast<const float4 *>(&s.h1[r][gk]);
      const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) g2[i][k] = fmaf(dv[i], hv[k], g2[i][k]);
      const float e = s.d1[r][w1j];
      const float4 xv = *reinterpret_cast<const float4 *>(&s.x[r][w1k]);
      g1[0] = fmaf(e, xv.x, g1[0]);
      g1[1] = fmaf(e, xv.y, g1[1]);
      g1[2] = fmaf(e, xv.z, g1[2]);
      g1[3] = fmaf(e, xv.w, g1[3]);
      const float dzv = s.dz[r][w3c];
      const float2 hh = *reinterpret_cast<const float2 *>(&s.h2[r][w3k]);
      g3[0] = fmaf(dzv, hh.x, g3[0]);
      g3[1] = fmaf(dzv, hh.y, g3[1]);
    }
    if (tid < 2 * kH + kOut) {
      const float *col = tid < kH ? &s.d1[0][tid] : tid < 2 * kH ? &s.d2[0][tid - kH] : &s.dz[0][tid - 2 * kH];
      const int pitch = tid < 2 * kH ? kHP : kOut;
#pragma unroll 8
      for (int r = 0; r < kTileRows; ++r) gb += col[r * pitch];
    }
  }
  float *G = part + (long long)blockIdx.x * kPart;
  if constexpr (kGroups) {
    __syncthreads();  // the last tile is used up
    G = &s.x[0][0];
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int k = 0; k < 4; ++k) G[oW2 + (gj + i) * kH + gk + k] = g2[i][k];
    G[oW1 + w1j * kIn + w1k + i] = g1[i];
  }
  G[oW3 + w3c * kH + w3k] = g3[0];
  G[oW3 + w3c * kH + w3k + 1] = g3[1];
  if (tid < kH)
    G[oB1 + tid] = gb;
  else if (tid < 2 * kH)
    G[oB2 + tid - kH] = gb;
  else if (tid < 2 * kH + kOut)
    G[oB3 + tid - 2 * kH] = gb;
  if (lane < 4) s.loss[r0 + lane] = loss;
  __syncthreads();
  if (tid < kTileRows) {
    loss = s.loss[tid];
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (tid == 0) G[kNParams] = loss;
  }
  if constexpr (kGroups) {
    const cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    float *out = part + (long long)(blockIdx.x / kCluster) * kPart;
    for (int i = (int)cluster.block_rank() * 256 + tid; i < kPart; i += 256 * kCluster) {
      double v = 0.0;
#pragma unroll
      for (int c = 0; c < kCluster; ++c) v += (double)*cluster.map_shared_rank(G + i, c);
      out[i] = (float)v;
    }
    cluster.sync();  // no CTA leaves while its gradient is being read
  }
}

// G and the loss from the partials: 8 threads per entry add strided
// partials, then each other's sums (a fixed order), in FP64, and divide by the rows:
// neither up to 40 additions nor a rounded 1 / n are in the result.
__global__ void __launch_bounds__(256) mlp_sum_kernel(const float *__restrict__ part, int nparts, int n,
                                                      float *__restrict__ G, float *__restrict__ loss) {
  __shared__ double red[8][33];
  const int e = threadIdx.x & 31, q = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + e;
  double v = 0.0;
  if (i < kPart) {
#pragma unroll 4
    for (int b = q; b < nparts; b += 8) v += (double)part[(long long)b * kPart + i];
  }
  red[q][e] = v;
  __syncthreads();
  if (q == 0 && i < kPart) {
    for (int k = 1; k < 8; ++k) v += red[k][e];
    v /= (double)n;
    if (i < kNParams)
      G[i] = (float)v;
    else
      *loss = (float)v;
  }
}

__global__ void adam_kernel(float *__restrict__ P, const float *__restrict__ G, float *__restrict__ m1,
                            float *__restrict__ m2, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float g = G[i];
  const float a = b1 * m1[i] + (1.f - b1) * g;
  const float v = b2 * m2[i] + (1.f - b2) * g * g;
  m1[i] = a;
  m2[i] = v;
  P[i] -= lr * (a / c1) / (sqrtf(v / c2) + eps);
}

// ---- block features and labels ------------------------------------------------

// Static per-block statistics of B: [0] max|B|, [1] sum B^2, [2] sum of row
// exponents over nonzero rows, [3] nonzero rows, [4] min exponent, [5] max
// exponent, [6] rows with exponent < max_e - 20 (filled in a second pass).
// packed: B holds per P the upper triangle row by row (off-diagonal entries
// then count twice in the sum of squares).
__global__ void __launch_bounds__(256) block_stats_kernel(const double *__restrict__ B, const int *__restrict__ eB,
                                                          const int *__restrict__ perm, int naux, int nao,
                                                          double *__restrict__ stats, bool packed) {
  const int b = blockIdx.x;
  const int p0 = b * df::kBlock;
  const int nP = min(df::kBlock, naux - p0);
  const long long n2 = (long long)nao * nao;
  const long long npk = (long long)nao * (nao + 1) / 2;
  double mx = 0.0, ss = 0.0;
  for (int pl = 0; pl < nP; ++pl) {
    const int P = perm ? perm[p0 + pl] : p0 + pl;
    if (packed) {
      const double *src = B + (long long)P * npk;
      const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
      for (int mu = warp; mu < nao; mu += (int)(blockDim.x >> 5)) {
        const double *row = src + (long long)mu * nao - (long long)mu * (mu - 1) / 2 - mu;
        for (int nu = mu + lane; nu < nao; nu += 32) {
          const double v = row[nu];
          mx = fmax(mx, fabs(v));
          ss = fma(nu == mu ? v : 2.0 * v, v, ss);
        }
      }
    } else {
      const double *src = B + (long long)P * n2;
      for (long long i = threadIdx.x; i < n2; i += blockDim.x) {
        const double v = src[i];
        mx = fmax(mx, fabs(v));
        ss = fma(v, v, ss);
      }
    }
  }
  double esum = 0.0, cnt = 0.0, emin = 1e9, emax = -1e9;
  const int rows = nP * nao;
  for (int r = threadIdx.x; r < rows; r += blockDim.x) {
    const int e = eB[(long long)p0 * nao + r];
    // every row of the block counts (a zero row has exponent 0)
    esum += e;
    cnt += 1.0;
    emin = fmin(emin, (double)e);
    emax = fmax(emax, (double)e);
  }
  __shared__ double red[6][8];
  double vals[6] = {mx, ss, esum, cnt, emin, emax};
  for (int q = 0; q < 6; ++q) {
    double v = vals[q];
    for (int o = 16; o > 0; o >>= 1) {
      const double w = __shfl_xor_sync(0xffffffffu, v, o);
      v = (q == 0 || q == 5) ? fmax(v, w) : (q == 4 ? fmin(v, w) : v + w);
    }
    if ((threadIdx.x & 31) == 0) red[q][threadIdx.x >> 5] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 0; q < 6; ++q) {
      double v = red[q][0];
      for (int k = 1; k < 8; ++k)
        v = (q == 0 || q == 5) ? fmax(v, red[q][k]) : (q == 4 ? fmin(v, red[q][k]) : v + red[q][k]);
      stats[b * 8 + q] = v;
    }
  }
  __syncthreads();
  // second pass: rows far below the block's largest row
  const int emx = (int)stats[b * 8 + 5];
  double small = 0.0;
  for (int r = threadIdx.x; r < rows; r += blockDim.x) small += (eB[(long long)p0 * nao + r] < emx - 20) ? 1.0 : 0.0;
  for (int o = 16; o > 0; o >>= 1) small += __shfl_xor_sync(0xffffffffu, small, o);
  __shared__ double rs[8];
  if ((threadIdx.x & 31) == 0) rs[threadIdx.x >> 5] = small;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int k = 0; k < 8; ++k) v += rs[k];
    stats[b * 8 + 6] = v;
  }
}

// 16 features per block from the static statistics and the iteration's scalars.
// dD_dev, when given, replaces dD (the density change measured on the device).
__global__ void block_features_kernel(const double *__restrict__ stats, int nblk, int naux, int nao, int nocc,
                                      double tau, double dD, const double *__restrict__ dD_dev, double dE,
                                      int s_rule, float *__restrict__ F) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nblk) return;
  if (dD_dev) dD = *dD_dev;
  if (!(dD >= 0.0 && dD <= 1e300)) dD = 1.0;  // a non-finite change reads as "large", never as NaN
  double gmax = 0.0, gss = 0.0;
  for (int k = 0; k < nblk; ++k) {
    gmax = fmax(gmax, stats[k * 8 + 0]);
    gss += stats[k * 8 + 1];
  }
  const double *st = stats + b * 8;
  const double tiny = 1e-300;
  const int nP = min(df::kBlock, naux - b * df::kBlock);
  float f[16];
  f[0] = (float)(log2(st[0] + tiny) / 32.0);
  f[1] = (float)(0.5 * log2(st[1] + tiny) / 32.0);
  f[2] = (float)(st[2] / fmax(st[3], 1.0) / 32.0);
  f[3] = (float)((st[5] - st[4]) / 32.0);
  f[4] = (float)(log10(tau) / 16.0);
  f[5] = (float)(log10(dD + 1e-30) / 16.0);
  f[6] = (float)((double)b / (double)nblk);
  f[7] = (float)(log2((double)nP) / 8.0);
  f[8] = (float)(log2((double)nao) / 12.0);
  f[9] = (float)(log2((double)nocc) / 10.0);
  f[10] = (float)(log2(st[1] / fmax(gss, tiny) + tiny) / 32.0);
  f[11] = (float)(st[6] / fmax(st[3], 1.0));
  f[12] = (float)(s_rule / 8.0);
  f[13] = (float)((log2(st[0] + tiny) - log2(gmax + tiny)) / 32.0);
  f[14] = (float)(log10(dE + 1e-30) / 16.0);
  f[15] = 1.0f;
  for (int k = 0; k < 16; ++k) F[b * 16 + k] = f[k];
}

// max over (mu <= nu) of |K_b(s) - K_b^FP64| per block b, from the second
// GEMM's int64 partials of the last emulated build (blocks of slice count s).
__global__ void block_error_kernel(const long long *__restrict__ Rp, const int *__restrict__ eX,
                                   const int *__restrict__ s_blk, df::ShiftTable T, const double *__restrict__ K64,
                                   int nao, int nblk, int nsplit, unsigned long long *__restrict__ err) {
  const int nu = blockIdx.x * blockDim.x + threadIdx.x;
  const int mu = blockIdx.y;
  const int b = blockIdx.z;
  if (nu >= nao || nu < mu) return;
  const long long bs = (long long)nao * nao;
  long long R = 0;
  for (int sp = 0; sp < nsplit; ++sp) R += Rp[((long long)b * nsplit + sp) * bs + (long long)nu * nao + mu];
  const int s = s_blk[b];
  const int k = eX[b * nao + mu] + eX[b * nao + nu] - 14 - 8 * (s - 1) + T.v[s];
  const double d = fabs(df::ldexp_i64(R, k) - K64[(long long)b * bs + (long long)mu * nao + nu]);
  atomicMax(&err[b], (unsigned long long)__double_as_longlong(d));
}

// Learned counts: per block the most probable class + 1, or s_rule when that
// probability is below min_conf (flag set); counts capped at s_max.
__global__ void pick_slices_kernel(const float *__restrict__ probs, int nblk, float min_conf, int s_rule, int s_max,
                                   int *__restrict__ out) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nblk) return;
  int best = 0;
  float pb = probs[b * kOut];
  for (int c = 1; c < kOut; ++c)
    if (probs[b * kOut + c] > pb) {
      pb = probs[b * kOut + c];
      best = c;
    }
  const bool low = pb < min_conf;
  const int s = low ? s_rule : best + 1;
  out[b] = s < s_max ? s : s_max;
  out[nblk + b] = low ? 1 : 0;
}

// Exponents of the error-bound check: out[b] = max_mu eX[b, mu], out[nblk + b]
// = max eB over the block's (P, mu) rows, out[2 nblk] = max eC.  One CTA per
// block (plus one for eC).
__global__ void __launch_bounds__(256) check_exponents_kernel(const int *__restrict__ eX, const int *__restrict__ eB,
                                                              const int *__restrict__ eC, int nblk, int nao, int naux,
                                                              int nocc, int *__restrict__ out) {
  const int b = blockIdx.x;
  int ex = INT_MIN, eb = INT_MIN;
  if (b < nblk) {
    for (int mu = threadIdx.x; mu < nao; mu += blockDim.x) ex = max(ex, eX[b * nao + mu]);
    const long long r0 = (long long)b * df::kBlock * nao;
    const long long r1 = (long long)min(naux, (b + 1) * df::kBlock) * nao;
    for (long long r = r0 + threadIdx.x; r < r1; r += blockDim.x) eb = max(eb, eB[r]);
  } else {
    for (int i = threadIdx.x; i < nocc; i += blockDim.x) ex = max(ex, eC[i]);
  }
  for (int o = 16; o > 0; o >>= 1) {
    ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
    eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, o));
  }
  __shared__ int rx[8], rb[8];
  if ((threadIdx.x & 31) == 0) {
    rx[threadIdx.x >> 5] = ex;
    rb[threadIdx.x >> 5] = eb;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) {
      ex = max(ex, rx[w]);
      eb = max(eb, rb[w]);
    }
    if (b < nblk) {
      out[b] = ex;
      out[nblk + b] = eb;
    } else {
      out[2 * nblk] = ex;
    }
  }
}

}  // namespace

struct df_mlp {
  float *P = nullptr, *G = nullptr, *m1 = nullptr, *m2 = nullptr, *loss = nullptr;
  float *part = nullptr;  // [kOwnParts][kPart] partial gradients
  int t = 0;
};

extern "C" {

df_status df_mlp_create(df_mlp **out) {
  if (!out) return DF_ERR_ARG;
  df_mlp *m = new (std::nothrow) df_mlp();
  if (!m) return DF_ERR_OOM;
  // one allocation: P, the two moments, G, the loss, the partial gradients
  const size_t np = (kNParams + 63) / 64 * 64;
  static_assert(sizeof(float) * (4 * (kNParams + 63) / 64 * 64 + 64 + kOwnParts * kPart) <= 1 << 20, "a cheap allocation");
  cudaError_t e = cudaMalloc(&m->P, sizeof(float) * (4 * np + 64 + (size_t)kOwnParts * kPart));
  if (e == cudaSuccess) {
    m->m1 = m->P + np;
    m->m2 = m->P + 2 * np;
    m->G = m->P + 3 * np;
    m->loss = m->P + 4 * np;
    m->part = m->loss + 64;
  }
  if (e == cudaSuccess) e = cudaMemset(m->P, 0, sizeof(float) * 3 * np);
  if (e != cudaSuccess) {
    df_mlp_destroy(m);
    return DF_ERR_CUDA;
  }
  *out = m;
  return DF_OK;
}

void df_mlp_destroy(df_mlp *m) {
  if (!m) return;
  cudaFree(m->P);
  delete m;
}

int df_mlp_num_params(void) { return kNParams; }

df_status df_mlp_set_params(df_mlp *m, const float *host, int n) {
  if (!m || !host || n != kNParams) return DF_ERR_ARG;
  m->t = 0;
  cudaError_t e = cudaMemcpy(m->P, host, sizeof(float) * n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(m->m1, 0, sizeof(float) * kNParams);
  if (e == cudaSuccess) e = cudaMemset(m->m2, 0, sizeof(float) * kNParams);
  return e == cudaSuccess ? DF_OK : DF_ERR_CUDA;
}

df_status df_mlp_get_params(const df_mlp *m, float *host, int n) {
  if (!m || !host || n != kNParams) return DF_ERR_ARG;
  return cudaMemcpy(host, m->P, sizeof(float) * n, cudaMemcpyDeviceToHost) == cudaSuccess ? DF_OK : DF_ERR_CUDA;
}

df_status df_mlp_forward(df_mlp *m, const float *X, int n, float *probs, void *stream) {
  if (!m || !X || !probs || n < 0) return DF_ERR_ARG;
  if (n == 0) return DF_OK;
  mlp_forward_kernel<<<(n + kRowsPerBlock - 1) / kRowsPerBlock, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      m->P, X, n, probs);
  return cudaGetLastError() == cudaSuccess ? DF_OK : DF_ERR_CUDA;
}

df_status df_mlp_gradients(df_mlp *m, const float *X, const int *y, int n, float *grad_host, float *loss_host,
                           void *stream) {
  if (!m || !X || !y || n <= 0) return DF_ERR_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int ntiles = (n + kTileRows - 1) / kTileRows;
  const bool groups = ntiles > kOwnParts;
  const int most = ntiles <= 2 * kCluster * kClustersAlone ? kClustersAlone : kMaxClusters;
  const int parts = groups ? std::min((ntiles + kCluster - 1) / kCluster, most) : ntiles;
  auto kern = groups ? mlp_backward_kernel<true> : mlp_backward_kernel<false>;
  // the attribute is per device and cheap to set; no process-wide flag to keep
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlpTile));
  if (e != cudaSuccess) return DF_ERR_CUDA;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(groups ? parts * kCluster : parts));
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = sizeof(MlpTile);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kCluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = groups ? 1 : 0;
  e = cudaLaunchKernelEx(&cfg, kern, (const float *)m->P, X, y, n, m->part);
  if (e != cudaSuccess) return DF_ERR_CUDA;
  mlp_sum_kernel<<<(kPart + 31) / 32, 256, 0, st>>>(m->part, parts, n, m->G, m->loss);
  e = cudaGetLastError();
  if (e != cudaSuccess) return DF_ERR_CUDA;
  if (grad_host) e = cudaMemcpyAsync(grad_host, m->G, sizeof(float) * kNParams, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && loss_host) e = cudaMemcpyAsync(loss_host, m->loss, sizeof(float), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && (grad_host || loss_host)) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? DF_OK : DF_ERR_CUDA;
}

df_status df_mlp_train_step(df_mlp *m, const float *X, const int *y, int n, float lr, float *loss_host,
                            void *stream) {
  df_status r = df_mlp_gradients(m, X, y, n, nullptr, nullptr, stream);
  if (r != DF_OK) return r;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  m->t += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)m->t), c2 = 1.f - powf(b2, (float)m->t);
  adam_kernel<<<(kNParams + 255) / 256, 256, 0, st>>>(m->P, m->G, m->m1, m->m2, kNParams, lr, b1, b2, 1e-8f, c1, c2);
  if (cudaGetLastError() != cudaSuccess) return DF_ERR_CUDA;
  if (loss_host) {
    if (cudaMemcpyAsync(loss_host, m->loss, sizeof(float), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return DF_ERR_CUDA;
  }
  return DF_OK;
}

df_status df_block_features(df_ctx *c, int nocc, double tau, double dD, double dE, int s_rule, float *F,
                            void *stream) {
  if (!c || !F || nocc <= 0 || !(tau > 0.0)) return DF_ERR_ARG;
  if (!c->ready) return DF_ERR_STATE;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (!c->bstats) {
    if (cudaMalloc(&c->bstats, sizeof(double) * 8 * c->nblk) != cudaSuccess) return DF_ERR_OOM;
    block_stats_kernel<<<c->nblk, 256, 0, st>>>(c->B, c->eB, c->perm, c->naux, c->nao, c->bstats, c->packed);
    if (cudaGetLastError() != cudaSuccess) return DF_ERR_CUDA;
  }
  block_features_kernel<<<(c->nblk + 127) / 128, 128, 0, st>>>(c->bstats, c->nblk, c->naux, c->nao, nocc, tau, dD,
                                                               nullptr, dE, s_rule, F);
  return cudaGetLastError() == cudaSuccess ? DF_OK : DF_ERR_CUDA;
}

df_status df_block_errors(df_ctx *c, const double *C, int nocc, double *err_host, double *kmax_host, void *stream) {
  if (!c || !C || !err_host || nocc <= 0 || nocc > c->nocc_max) return DF_ERR_ARG;
  if (!c->ready) return DF_ERR_STATE;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int nao = c->nao, nblk = c->nblk;
  const long long bs = (long long)nao * nao;
  double *K64 = nullptr, *Kfull = nullptr;
  unsigned long long *err = nullptr;
  df_status r = DF_OK;
  cudaError_t e = cudaMalloc(&K64, sizeof(double) * bs * nblk);
  if (e == cudaSuccess) e = cudaMalloc(&Kfull, sizeof(double) * bs);
  if (e == cudaSuccess) e = cudaMalloc(&err, sizeof(unsigned long long) * nblk);
  if (e != cudaSuccess) r = DF_ERR_OOM;
  // FP64 reference: X^T by cuBLAS (as in the native build), then K_b = Xt_b^T Xt_b per block
  if (r == DF_OK) r = df_build_K(c, C, nocc, 0, Kfull, nullptr, stream);
  if (r == DF_OK) {
    // the FP64 build leaves X^T [mu][(P, i)] in the natural P order; a block of
    // the exchange order (df_setup_ordered) gathers its functions' columns first
    const double one = 1.0, zero = 0.0;
    const long long ldx = (long long)c->naux * nocc;
    const long long kbw = (long long)df::kBlock * nocc;
    double *Xg = nullptr;
    if (!c->perm_h.empty() && cudaMalloc(&Xg, sizeof(double) * nao * kbw) != cudaSuccess) r = DF_ERR_OOM;
    for (int b = 0; b < nblk && r == DF_OK; ++b) {
      const int nP = (b + 1) * df::kBlock <= c->naux ? df::kBlock : c->naux - b * df::kBlock;
      const double *Xb = c->X + (long long)b * df::kBlock * nocc;
      long long ld = ldx;
      if (Xg) {
        for (int j = 0; j < nP && r == DF_OK; ++j)
          if (cudaMemcpy2DAsync(Xg + (long long)j * nocc, sizeof(double) * kbw,
                                c->X + (long long)c->perm_h[b * df::kBlock + j] * nocc, sizeof(double) * ldx,
                                sizeof(double) * nocc, nao, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
            r = DF_ERR_CUDA;
        Xb = Xg;
        ld = kbw;
      }
      if (r == DF_OK && cublasDgemm(c->cublas, CUBLAS_OP_T, CUBLAS_OP_N, nao, nao, nP * nocc, &one, Xb, (int)ld, Xb,
                                    (int)ld, &zero, K64 + (long long)b * bs, nao) != CUBLAS_STATUS_SUCCESS)
        r = DF_ERR_CUDA;
    }
    if (Xg) {
      cudaStreamSynchronize(st);
      cudaFree(Xg);
    }
  }
  if (r == DF_OK && kmax_host) {
    // max|K| of the FP64 build (host side, once)
    std::vector<double> h((size_t)bs);
    if (cudaMemcpyAsync(h.data(), Kfull, sizeof(double) * bs, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      r = DF_ERR_CUDA;
    double mx = 0.0;
    for (double v : h) mx = fmax(mx, fabs(v));
    *kmax_host = mx;
  }
  std::vector<int> sb(nblk);
  std::vector<unsigned long long> eh(nblk);
  for (int s = 1; s <= c->s_max && r == DF_OK; ++s) {
    for (int b = 0; b < nblk; ++b) sb[b] = s;
    r = df_build_K_blocks(c, C, nocc, sb.data(), Kfull, nullptr, stream);
    if (r != DF_OK) break;
    df::ShiftTable tt;
    const long long kb = df::xdigit_ld(nocc);
    for (int q = 0; q <= 8; ++q) tt.v[q] = df::fixed_point_shift(q, kb);
    if (cudaMemsetAsync(err, 0, sizeof(unsigned long long) * nblk, st) != cudaSuccess) {
      r = DF_ERR_CUDA;
      break;
    }
    dim3 grid((nao + 127) / 128, nao, nblk);
    block_error_kernel<<<grid, 128, 0, st>>>(c->Rp, c->eX, c->sblk, tt, K64, nao, nblk, c->nsplit, err);
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyAsync(eh.data(), err, sizeof(unsigned long long) * nblk, cudaMemcpyDeviceToHost, st) !=
            cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
      r = DF_ERR_CUDA;
      break;
    }
    for (int b = 0; b < nblk; ++b) {
      double d;
      std::memcpy(&d, &eh[b], sizeof(double));
      err_host[b * 8 + (s - 1)] = d;
    }
  }
  for (int s = c->s_max + 1; s <= 8 && r == DF_OK; ++s)
    for (int b = 0; b < nblk; ++b) err_host[b * 8 + (s - 1)] = err_host[b * 8 + (c->s_max - 1)];
  cudaStreamSynchronize(st);
  cudaFree(K64);
  cudaFree(Kfull);
  cudaFree(err);
  return r;
}

}  // extern "C"

namespace {

// Table 1's printed accuracy per level (levels 1..4), the tolerance feature.
constexpr double kLevelTau[5] = {0.0, 7.1e-15, 1.8e-12, 4.7e-10, 1.2e-7};

// log2 of the a-priori error bound beta_b(s) of block b's K_b (see
// df_set_predictor): kb 1.01 (s+1) 2^(-8s) (2^(2E) + 2 nao 2^(F+Ec+E)) + kb 2^(2E-52).
double log2_bound(int s, double kb, int nao, int E, int F, int Ec) {
  const double a = 2.0 * E, b = 1.0 + std::log2((double)nao) + F + Ec + E;
  const double hi = std::max(a, b);
  const double trunc = std::log2(1.01 * (s + 1)) - 8.0 * s + hi + std::log2(std::exp2(a - hi) + std::exp2(b - hi));
  const double round = a - 52.0;
  const double top = std::max(trunc, round);
  return std::log2(kb) + top + std::log2(std::exp2(trunc - top) + std::exp2(round - top));
}

df_status cuda_err(cudaError_t e) {
  if (e == cudaSuccess) return DF_OK;
  return e == cudaErrorMemoryAllocation ? DF_ERR_OOM : DF_ERR_CUDA;
}

}  // namespace

namespace df {

df_status build_K_learned(df_ctx *c, const double *C, int nocc, double *K, df_kstats *stats, cudaStream_t st) {
  const int level = c->level;
  const int s_rule = level_count(c, level);
  if (level < 1 || level > 4 || s_rule < 1 || s_rule > c->s_max) return DF_ERR_ARG;
  const int nblk = c->nblk;
  cudaError_t e = cudaSuccess;
  if (!c->lF) e = cudaMalloc(&c->lF, sizeof(float) * 16 * nblk);
  if (e == cudaSuccess && !c->lprobs) e = cudaMalloc(&c->lprobs, sizeof(float) * kOut * nblk);
  if (e == cudaSuccess && !c->lpick) e = cudaMalloc(&c->lpick, sizeof(int) * 2 * nblk);
  if (e == cudaSuccess && !c->lexp) e = cudaMalloc(&c->lexp, sizeof(int) * (2 * nblk + 1));
  if (e == cudaSuccess && !c->lhost) e = cudaMallocHost(&c->lhost, sizeof(int) * (2 * nblk + 1));
  if (e == cudaSuccess && !c->bstats) {
    e = cudaMalloc(&c->bstats, sizeof(double) * 8 * nblk);
    if (e == cudaSuccess) {
      block_stats_kernel<<<nblk, 256, 0, st>>>(c->B, c->eB, c->perm, c->naux, c->nao, c->bstats, c->packed);
      e = cudaGetLastError();
    }
  }
  if (e != cudaSuccess) return cuda_err(e);
  // 1. features -> network -> counts (with the low-confidence fallback)
  block_features_kernel<<<(nblk + 127) / 128, 128, 0, st>>>(c->bstats, nblk, c->naux, c->nao, nocc,
                                                            kLevelTau[level], 0.0, c->dD, c->dE_last, s_rule, c->lF);
  e = cudaGetLastError();
  if (e == cudaSuccess) {
    mlp_forward_kernel<<<(nblk + kRowsPerBlock - 1) / kRowsPerBlock, 256, 0, st>>>(c->pred->P, c->lF, nblk,
                                                                                     c->lprobs);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    pick_slices_kernel<<<(nblk + 127) / 128, 128, 0, st>>>(c->lprobs, nblk, c->min_conf, s_rule, c->s_max,
                                                           c->lpick);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(c->lhost, c->lpick, sizeof(int) * 2 * nblk, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_err(e);
  std::vector<int> sb(c->lhost, c->lhost + nblk);
  int low = 0;
  for (int b = 0; b < nblk; ++b) low += c->lhost[nblk + b];
  // a count above the level's only pays for another below it: with none below,
  // every block takes the level's count
  bool below = false;
  for (int b = 0; b < nblk; ++b) below = below || sb[b] < s_rule;
  if (!below)
    for (int b = 0; b < nblk; ++b) sb[b] = std::min(sb[b], s_rule);
  // 2. first GEMM and X split at the predicted counts (C split deep enough for s_rule)
  df_status r = k_front(c, C, nocc, sb.data(), s_rule, st);
  if (r != DF_OK) return r;
  // 3. the error-bound check from the exponents
  check_exponents_kernel<<<nblk + 1, 256, 0, st>>>(c->eX, c->eB, c->eC, nblk, c->nao, c->naux, nocc, c->lexp);
  e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(c->lhost, c->lexp, sizeof(int) * (2 * nblk + 1), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_err(e);
  const int Ec = c->lhost[2 * nblk];
  std::vector<double> lb_rule(nblk), lb(nblk);
  double ref = -INFINITY;
  for (int b = 0; b < nblk; ++b) {
    const int nP = std::min(kBlock, c->naux - b * kBlock);
    const double kb = (double)nP * nocc;
    lb_rule[b] = log2_bound(s_rule, kb, c->nao, c->lhost[b], c->lhost[nblk + b], Ec);
    lb[b] = log2_bound(sb[b], kb, c->nao, c->lhost[b], c->lhost[nblk + b], Ec);
    ref = std::max(ref, lb_rule[b]);
  }
  // sums of 2^(log2 bound - ref), all <= nblk
  auto total = [&](const std::vector<double> &v) {
    double t = 0.0;
    for (double x : v) t += std::exp2(x - ref);
    return t;
  };
  const double budget = total(lb_rule);
  double have = total(lb);
  int raised = 0;
  while (have > budget * (1.0 + 1e-12)) {
    int pick = -1;
    for (int b = 0; b < nblk; ++b)
      if (sb[b] < s_rule && (pick < 0 || lb[b] > lb[pick])) pick = b;
    if (pick < 0) break;  // cannot happen: every block at >= s_rule meets the budget
    sb[pick] = s_rule;
    lb[pick] = lb_rule[pick];
    ++raised;
    have = total(lb);
  }
  if (raised) {
    // 4. recompute the first GEMM and the X split with the raised counts
    r = k_front(c, C, nocc, sb.data(), s_rule, st);
    if (r != DF_OK) return r;
  }
  r = k_back(c, nocc, K, st);
  if (r != DF_OK) return r;
  if (stats) {
    stats->nblk = nblk;
    long long pairs = 0;
    for (int b = 0; b < nblk; ++b) {
      if (b < 256) stats->slices[b] = sb[b];
      pairs += (long long)sb[b] * (sb[b] + 1) / 2;
    }
    stats->recomputed = raised;
    stats->fallback = 0;
    stats->low_confidence = low;
    stats->level = level;
    stats->slice_pairs = pairs;
    stats->bound_ratio = have / budget;
  }
  return DF_OK;
}

}  // namespace df

extern "C" df_status df_set_predictor(df_ctx *c, df_mlp *net, float min_conf) {
  if (!c || !(min_conf > 0.f && min_conf <= 1.f)) return DF_ERR_ARG;
  c->pred = net;
  c->min_conf = min_conf;
  return DF_OK;
}
