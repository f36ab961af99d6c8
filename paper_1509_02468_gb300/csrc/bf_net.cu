// The learned preconditioner T of the flexible CG and LOBPCG filters (the preconditioner of
// Algorithms 2 and 3, left open by the paper; Section 5's flexible beta admits a variable,
// nonlinear T): a three-layer 3 x 3 conv net on the image-shaped residual r,
//
//   C  = [ (D^-1 r) / rho,  g,  1 / d ],  rho = rms(D^-1 r)
//   A1 = conv(C, W1) (16 ch),  A2 = conv(relu(A1), W2) (16 ch),  O = conv(relu(A2), W3)
//   T(r) = rho O
//
// (cross-correlations without bias, zero outside the image).  Weights are kept in FP32
// (the trained master copy) and used rounded to BF16; every product is accumulated in
// FP32.  Training pairs (r, z) solve (L + sigma I) z = r; the loss of a pair is
// ||T(r) - z||^2 / ||z||^2, its gradient is accumulated by bf_net_accumulate and applied
// by bf_net_adam (Adam, Kingma and Ba).
//
// Kernels work on 32 x 8 pixel tiles with a one-pixel halo staged channel-major in shared
// memory; activations are stored pixel-major [n][16].  Both the layers and the weight
// gradients are bound by shared memory unless a thread reuses what it loads: a thread owns a
// run of four pixels (layers: times four output channels, so 18 loads feed 144 products per
// input channel; gradients: all nine taps of one weight pair).  At 256 x 256 a pair's
// training step took 241 us (layers 16 -> 16 of 20 us, their gradient 52 us, three serial
// sums over the tiles of 33 us each); it takes 116 us now, in nine launches.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <mutex>

#include "bf_internal.cuh"

#define NET_CH 16
#define NET_CIN 3
#define NET_TW 32
#define NET_TH 8
#define NET_HW (NET_TW + 2)
#define NET_HH (NET_TH + 2)
#define NET_XS 36                          // staged row stride (16-byte aligned runs)
#define NET_HP (NET_XS * NET_HH + 4)       // channel stride: 12 banks apart
#define NET_W1 0
#define NET_W2 (NET_CH * NET_CIN * 9)
#define NET_W3 (NET_W2 + NET_CH * NET_CH * 9)
#define NET_NW (NET_W3 + NET_CH * 9)
#define NET_COLS 4                         // columns per pass of bf_net_apply

struct bf_net {
  int device;
  float* w;       // [NET_NW] FP32 master weights
  float* wq;      // [NET_NW] weights rounded to BF16 (as FP32)
  float* m;       // Adam moments
  float* v;
  float* grad;    // [NET_NW] accumulated gradient
  double* loss;   // [1] accumulated loss
  int t;          // Adam steps taken
  void* ws;       // activations, partial sums
  size_t ws_bytes;
};

namespace {

enum { IN_NET = 0, IN_RELU = 1, IN_PLAIN = 2 };
enum { OUT_ACT = 0, OUT_PRECOND = 1, OUT_MASKED = 2 };

struct NetArgs {
  int nx, ny;
  int64_t n;
  const float* r;        // IN_NET: residual columns, r[i * ldr + col]
  int64_t ldr;
  const float* guide;
  const float* d;
  float* rho;            // [cols]
  const double* rpart;   // IN_NET layers: block sums of k_net_sums, [cols][nrp][2]
  int nrp;
  double* zz;            // [1] or NULL
  const float* in;       // [cols][n][cin] activations
  float* out;            // [cols][n][cout]
  const float* mask;     // OUT_MASKED: [cols][n][cout] pre-activations
  float* z;              // OUT_PRECOND: z[i * ldz + col]
  int64_t ldz;
  const float* w;        // layer weights as stored: [cout_l][cin_l][9]
  int transpose;         // use the adjoint (flipped, transposed) weights
  const int* stop;       // optional solver status: nonzero = stopped, skip the work
};

__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// rho[col] = sqrt(mean) and zz = sum z^2 (column 0) from the block sums of k_net_sums, added
// in the same order by every block of the first layer (a launch of its own took longer);
// block (0, 0) of the column keeps them for the kernels after it.
__device__ __forceinline__ float net_rho(const NetArgs& a, int col) {
  __shared__ float sh;
  if (threadIdx.x < 32) {
    double a0 = 0.0, a1 = 0.0;
    for (int b = threadIdx.x; b < a.nrp; b += 32) {
      a0 += a.rpart[((int64_t)col * a.nrp + b) * 2];
      a1 += a.rpart[((int64_t)col * a.nrp + b) * 2 + 1];
    }
    a0 = warp_sum(a0);
    a1 = warp_sum(a1);
    if (threadIdx.x == 0) {
      sh = (float)sqrt(a0 / (double)a.n);
      if (blockIdx.x == 0 && blockIdx.y == 0) {
        a.rho[col] = sh;
        if (a.zz && col == 0) *a.zz = a1;
      }
    }
  }
  __syncthreads();
  return sh;
}

// Stage the input tile (with halo) channel-major: s[c * NET_HP + hp].
template <int CIN, int IN>
__device__ __forceinline__ void net_stage(const NetArgs& a, const float* in, int col, float rh, int bx, int by, float* s) {
  for (int q = threadIdx.x; q < NET_HW * NET_HH; q += NET_TW * NET_TH) {
    const int hy = q / NET_HW, hx = q - hy * NET_HW, hp = hy * NET_XS + hx;
    const int gy = by - 1 + hy, gx = bx - 1 + hx;
    const bool inside = gx >= 0 && gx < a.nx && gy >= 0 && gy < a.ny;
    const int64_t i = (int64_t)gy * a.nx + gx;
    if (IN == IN_NET) {
      float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f;
      if (inside) {
        const float di = a.d[i];
        c0 = rh > 0.0f ? a.r[i * a.ldr + col] / (di * rh) : 0.0f;
        c1 = a.guide[i];
        c2 = 1.0f / di;
      }
      s[0 * NET_HP + hp] = c0;
      s[1 * NET_HP + hp] = c1;
      s[2 * NET_HP + hp] = c2;
    } else {
      const float* src = in + ((int64_t)col * a.n + i) * CIN;
#pragma unroll
      for (int c4 = 0; c4 < CIN; c4 += 4) {
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (inside) {
          if (CIN % 4 == 0) {
            v = *reinterpret_cast<const float4*>(src + c4);
          } else {
            v.x = src[c4];
            if (c4 + 1 < CIN) v.y = src[c4 + 1];
            if (c4 + 2 < CIN) v.z = src[c4 + 2];
            if (c4 + 3 < CIN) v.w = src[c4 + 3];
          }
          if (IN == IN_RELU) {
            v.x = fmaxf(v.x, 0.0f);
            v.y = fmaxf(v.y, 0.0f);
            v.z = fmaxf(v.z, 0.0f);
            v.w = fmaxf(v.w, 0.0f);
          }
        }
        s[(c4 + 0) * NET_HP + hp] = v.x;
        if (c4 + 1 < CIN) s[(c4 + 1) * NET_HP + hp] = v.y;
        if (c4 + 2 < CIN) s[(c4 + 2) * NET_HP + hp] = v.z;
        if (c4 + 3 < CIN) s[(c4 + 3) * NET_HP + hp] = v.w;
      }
    }
  }
}

// The six staged values of one row of a run's window.
__device__ __forceinline__ void net_row(const float* row, float (&x)[6]) {
  const float4 a = *reinterpret_cast<const float4*>(row);
  const float2 b = *reinterpret_cast<const float2*>(row + 4);
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
  x[4] = b.x; x[5] = b.y;
}

// One 3 x 3 conv layer (CIN -> COUT) on a tile; blockIdx.z is the column.  COUT = 16: warp w
// computes output channels 4 (w / 2) .. + 3 of the runs of half a tile.  COUT = 1: the four
// warp pairs each take a quarter of the input channels, and the quarters are added.
template <int CIN, int COUT, int IN, int OUT>
__global__ void __launch_bounds__(NET_TW * NET_TH) k_net_conv(const NetArgs a) {
  static_assert(COUT == NET_CH || (COUT == 1 && CIN % 4 == 0), "layer shapes of the net");
  constexpr int COUTP = (COUT + 3) & ~3;
  __shared__ __align__(16) float sx[CIN * NET_HP];
  __shared__ __align__(16) float sw[CIN * 9 * COUTP];       // [c][tap][o]
  const int col = blockIdx.z;
  const int bx = blockIdx.x * NET_TW, by = blockIdx.y * NET_TH;
  for (int e = threadIdx.x; e < CIN * 9 * COUTP; e += NET_TW * NET_TH) {
    const int o = e % COUTP, ct = e / COUTP, c = ct / 9, t = ct - c * 9;
    float wv = 0.0f;
    if (o < COUT) wv = a.transpose ? a.w[(c * COUT + o) * 9 + (8 - t)] : a.w[(o * CIN + c) * 9 + t];
    sw[e] = wv;
  }
  // the weights do not come from the kernel before this one (and the one that wrote them has
  // finished when that one runs), so they are staged while it does
  bf_pdl_enter();
  if (a.stop && *a.stop != 0) return;
  const float rh = IN == IN_NET ? net_rho(a, col) : 0.0f;
  net_stage<CIN, IN>(a, a.in, col, rh, bx, by, sx);
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, grp = wid >> 1;
  const int lx = 4 * (lane & 7), ly = 4 * (wid & 1) + (lane >> 3);
  if (COUT == 1) {
    constexpr int CQ = CIN / 4;
    __shared__ __align__(16) float red[4][NET_TW * NET_TH];
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int c = grp * CQ; c < (grp + 1) * CQ; ++c) {
#pragma unroll
      for (int ty = 0; ty < 3; ++ty) {
        float x[6];
        net_row(sx + c * NET_HP + (ly + ty) * NET_XS + lx, x);
#pragma unroll
        for (int tx = 0; tx < 3; ++tx) {
          const float w = sw[(c * 9 + 3 * ty + tx) * COUTP];
#pragma unroll
          for (int p = 0; p < 4; ++p) acc[p] = fmaf(w, x[p + tx], acc[p]);
        }
      }
    }
    *reinterpret_cast<float4*>(&red[grp][ly * NET_TW + lx]) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    __syncthreads();
    const int x = bx + (threadIdx.x & 31), y = by + (threadIdx.x >> 5);
    if (x >= a.nx || y >= a.ny) return;
    const float v = (red[0][threadIdx.x] + red[1][threadIdx.x]) + (red[2][threadIdx.x] + red[3][threadIdx.x]);
    const int64_t i = (int64_t)y * a.nx + x;
    if (OUT == OUT_PRECOND) a.z[i * a.ldz + col] = a.rho[col] * v;
    else a.out[(int64_t)col * a.n + i] = v;
    return;
  }
  float acc[4][4];                                          // [pixel][output channel]
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int o = 0; o < 4; ++o) acc[p][o] = 0.0f;
  for (int c = 0; c < CIN; ++c) {
#pragma unroll
    for (int ty = 0; ty < 3; ++ty) {
      float x[6];
      net_row(sx + c * NET_HP + (ly + ty) * NET_XS + lx, x);
#pragma unroll
      for (int tx = 0; tx < 3; ++tx) {
        const float4 w = *reinterpret_cast<const float4*>(sw + (c * 9 + 3 * ty + tx) * COUTP + 4 * grp);
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          acc[p][0] = fmaf(w.x, x[p + tx], acc[p][0]);
          acc[p][1] = fmaf(w.y, x[p + tx], acc[p][1]);
          acc[p][2] = fmaf(w.z, x[p + tx], acc[p][2]);
          acc[p][3] = fmaf(w.w, x[p + tx], acc[p][3]);
        }
      }
    }
  }
  const int y = by + ly;
  if (y >= a.ny) return;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int x = bx + lx + p;
    if (x >= a.nx) continue;
    const int64_t o = ((int64_t)col * a.n + (int64_t)y * a.nx + x) * COUT + 4 * grp;
    float4 v = make_float4(acc[p][0], acc[p][1], acc[p][2], acc[p][3]);
    if (OUT == OUT_MASKED) {
      const float4 m = *reinterpret_cast<const float4*>(a.mask + o);
      v.x = m.x > 0.0f ? v.x : 0.0f;
      v.y = m.y > 0.0f ? v.y : 0.0f;
      v.z = m.z > 0.0f ? v.z : 0.0f;
      v.w = m.w > 0.0f ? v.w : 0.0f;
    }
    *reinterpret_cast<float4*>(a.out + o) = v;
  }
}

// Per-block sums for rho (sum (r/d)^2) and, with z, sum z^2; blockIdx.y is the column.
__global__ void __launch_bounds__(256) k_net_sums(const float* r, int64_t ldr, const float* d, const float* z,
                                                  int64_t n, double* partials, const int* stop) {
  bf_pdl_enter();
  if (stop && *stop != 0) return;
  __shared__ double red[2 * 8];
  const int col = blockIdx.y;
  double s0 = 0.0, s1 = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const float c = r[i * ldr + col] / d[i];
    s0 += (double)(c * c);
    if (z) s1 += (double)z[i] * (double)z[i];
  }
  s0 = warp_sum(s0);
  s1 = warp_sum(s1);
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5] = s0;
    red[8 + (threadIdx.x >> 5)] = s1;
  }
  __syncthreads();
  if (threadIdx.x < 32) {                     // lanes 0 .. 7: the first sums, 8 .. 15: the second
    double v = red[threadIdx.x & 15];
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 23) == 0) partials[((int64_t)col * gridDim.x + blockIdx.x) * 2 + (threadIdx.x >> 3)] = v;
  }
}

// G3 = 2 rho (rho O - z) / zz and per-block sums of (rho O - z)^2.
__global__ void __launch_bounds__(256) k_net_loss(const float* O, const float* z, const float* rho,
                                                  const double* zz, int64_t n, float* G3, double* partials) {
  bf_pdl_enter();
  __shared__ double red[8];
  const float rh = rho[0];
  const float sc = (float)(2.0 * (double)rh / *zz);
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const float e = rh * O[i] - z[i];
    G3[i] = sc * e;
    s += (double)e * (double)e;
  }
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = red[threadIdx.x & 7];
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) partials[blockIdx.x] = v;
  }
}

#define NET_WGRAD_FLOATS (NET_CH * NET_HP + NET_CH * (NET_TW * NET_TH + 4))
// Per-block weight gradient dW[o][c][t] = sum_px G[px][o] X[px + t][c] over the block's
// tile (X staged like a conv input); partials[block][off + (o * CIN + c) * 9 + t].  A thread
// owns the nine taps of one pair (o, c) over a share of the tile's runs of four pixels (each
// sum in two parts, even and odd pixels); the shares are added in order.
template <int CIN, int COUT, int IN>
__device__ __forceinline__ void net_wgrad(const NetArgs& a, const float* in, const float* G, float* partials, int off,
                                          float* sh) {
  constexpr int NP = COUT * CIN, NG = (NET_TW * NET_TH / NP < 16) ? NET_TW * NET_TH / NP : 16;
  constexpr int NRUN = NET_TW * NET_TH / 4, GS = NET_TW * NET_TH + 4;   // gradient channel stride
  constexpr int XF = CIN * NET_HP, GF = COUT * GS, RF = NG > 1 ? NG * NP * 9 : 0;
  static_assert(XF + GF <= NET_WGRAD_FLOATS && RF <= NET_WGRAD_FLOATS, "shared memory of k_net_wgrad");
  float* sx = sh;
  float* sg = sh + XF;                                       // [o][px]
  const int bx = blockIdx.x * NET_TW, by = blockIdx.y * NET_TH;
  net_stage<CIN, IN>(a, in, 0, IN == IN_NET ? a.rho[0] : 0.0f, bx, by, sx);
  {
    const int p = threadIdx.x, x = bx + p % NET_TW, y = by + p / NET_TW;
    const bool in = x < a.nx && y < a.ny;
    const float* src = G + ((int64_t)y * a.nx + x) * COUT;
    if (COUT == 1) {
      sg[p] = in ? *src : 0.0f;
    } else {
#pragma unroll
      for (int o4 = 0; o4 < COUT / 4; ++o4) {
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (in) v = reinterpret_cast<const float4*>(src)[o4];
        sg[(4 * o4) * GS + p] = v.x;
        sg[(4 * o4 + 1) * GS + p] = v.y;
        sg[(4 * o4 + 2) * GS + p] = v.z;
        sg[(4 * o4 + 3) * GS + p] = v.w;
      }
    }
  }
  __syncthreads();
  const int grp = threadIdx.x / NP, pair = threadIdx.x - grp * NP;
  const int o = pair % COUT, c = pair / COUT;
  float s[2][9];
#pragma unroll
  for (int t = 0; t < 9; ++t) s[0][t] = s[1][t] = 0.0f;
  if (grp < NG) {
    for (int r = grp; r < NRUN; r += NG) {
      const int ly = r / (NET_TW / 4), lx = 4 * (r - ly * (NET_TW / 4));
      const float4 g4 = *reinterpret_cast<const float4*>(sg + o * GS + ly * NET_TW + lx);
      const float g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
      for (int ty = 0; ty < 3; ++ty) {
        float x[6];
        net_row(sx + c * NET_HP + (ly + ty) * NET_XS + lx, x);
#pragma unroll
        for (int tx = 0; tx < 3; ++tx)
#pragma unroll
          for (int p = 0; p < 4; ++p) s[p & 1][3 * ty + tx] = fmaf(g[p], x[p + tx], s[p & 1][3 * ty + tx]);
      }
    }
  }
  float* out = partials + (int64_t)(blockIdx.y * gridDim.x + blockIdx.x) * NET_NW + off;
  if (NG == 1) {
#pragma unroll
    for (int t = 0; t < 9; ++t) out[(o * CIN + c) * 9 + t] = s[0][t] + s[1][t];
    return;
  }
  __syncthreads();                                           // the tiles are read
  if (grp < NG) {
#pragma unroll
    for (int t = 0; t < 9; ++t) sh[grp * (NP * 9) + (o * CIN + c) * 9 + t] = s[0][t] + s[1][t];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < NP * 9; e += NET_TW * NET_TH) {
    float v = 0.0f;
    for (int k = 0; k < NG; ++k) v += sh[k * (NP * 9) + e];
    out[e] = v;
  }
}

// The three layers' gradients of a tile in one launch, blockIdx.z the layer (the largest
// first): dW2 = corr(G2, relu(A1)), dW1 = corr(G1, C), dW3 = corr(G3, relu(A2)).
__global__ void __launch_bounds__(NET_TW * NET_TH)
k_net_wgrad(const NetArgs a, const float* A1, const float* A2, const float* G1, const float* G2, const float* G3,
            float* partials) {
  bf_pdl_enter();
  __shared__ __align__(16) float sh[NET_WGRAD_FLOATS];
  if (blockIdx.z == 0) net_wgrad<NET_CH, NET_CH, IN_RELU>(a, A1, G2, partials, NET_W2, sh);
  else if (blockIdx.z == 1) net_wgrad<NET_CIN, NET_CH, IN_NET>(a, nullptr, G1, partials, NET_W1, sh);
  else net_wgrad<NET_CH, 1, IN_RELU>(a, A2, G3, partials, NET_W3, sh);
}

// grad[e] += sum_b partials[b][e] over all layers: 32 entries per block, eight threads each
// taking every eighth tile in FP64 (an FP64 addition is long: one thread per entry took 33 us
// at 256 tiles).
// The block past the entries adds the pair's loss, the sum of k_net_loss's block sums / zz.
__global__ void __launch_bounds__(256) k_net_wgrad_reduce(const float* partials, int nblocks, float* grad,
                                                          const double* lpart, int nl, const double* zz, double* loss) {
  bf_pdl_enter();
  __shared__ double red[8][32];
  if (blockIdx.x == gridDim.x - 1) {
    if (threadIdx.x >= 32) return;
    double t = 0.0;
    for (int b = threadIdx.x; b < nl; b += 32) t += lpart[b];
    t = warp_sum(t);
    if (threadIdx.x == 0) *loss += t / *zz;
    return;
  }
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (e < NET_NW)
    for (int b = part; b < nblocks; b += 8) s += (double)partials[(int64_t)b * NET_NW + e];
  red[part][lane] = s;
  __syncthreads();
  if (part == 0 && e < NET_NW) {
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += red[k][lane];
    grad[e] += (float)t;
  }
}

__global__ void k_net_adam(float* w, float* wq, float* m, float* v, float* grad, int n, float lr, float b1,
                           float b2, float eps, float c1, float c2) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const float g = grad[e];
  const float mm = b1 * m[e] + (1.0f - b1) * g;
  const float vv = b2 * v[e] + (1.0f - b2) * g * g;
  m[e] = mm;
  v[e] = vv;
  const float wn = w[e] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
  w[e] = wn;
  wq[e] = bf16_round(wn);
  grad[e] = 0.0f;
}

__global__ void k_net_scale(float* g, int n, float scale) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) g[e] *= scale;
}

__global__ void k_net_round(const float* w, float* wq, int n) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) wq[e] = bf16_round(w[e]);
}

// ------------------------------------------------------------------ host side
struct Bufs {
  float* A1;        // [cols][n][16]
  float* A2;        // [cols][n][16]
  float* O;         // [n]
  float* G3;        // [n]
  float* G2;        // [n][16]
  float* G1;        // [n][16]
  float* rho;       // [cols]
  double* zz;       // [1]
  double* dpart;    // [cols][nb][2]
  float* wpart;     // [tiles][NET_NW]
};

// blocks of the sums over the pixels: few, as every block of the first layer adds them
int net_sum_blocks(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, 256); }

int net_ws(bf_net* net, const bf_graph* g, int cols, bool train, Bufs* b) {
  const int64_t n = g->n;
  const int nb_red = net_sum_blocks(n);
  auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t act = al((size_t)cols * n * NET_CH * sizeof(float));
  const size_t vec = al((size_t)n * sizeof(float));
  const size_t act1 = al((size_t)n * NET_CH * sizeof(float));
  const size_t ntile = (size_t)((g->nx + NET_TW - 1) / NET_TW) * (size_t)((g->ny + NET_TH - 1) / NET_TH);
  size_t bytes = 2 * act + al(cols * sizeof(float)) + al(sizeof(double)) +
                 al((size_t)cols * nb_red * 2 * sizeof(double));
  if (train) bytes += 2 * vec + 2 * act1 + al(ntile * NET_NW * sizeof(float));
  if (bytes > net->ws_bytes) {
    if (net->ws) cudaFree(net->ws);
    net->ws = nullptr;
    net->ws_bytes = 0;
    cudaError_t e = cudaMalloc(&net->ws, bytes);
    if (e != cudaSuccess) return bf_cuda_fail(e, "cudaMalloc(net workspace)");
    net->ws_bytes = bytes;
  }
  char* p = (char*)net->ws;
  b->A1 = (float*)p; p += act;
  b->A2 = (float*)p; p += act;
  b->rho = (float*)p; p += al(cols * sizeof(float));
  b->zz = (double*)p; p += al(sizeof(double));
  b->dpart = (double*)p; p += al((size_t)cols * nb_red * 2 * sizeof(double));
  b->O = b->G3 = nullptr;
  b->G2 = b->G1 = nullptr;
  b->wpart = nullptr;
  if (train) {
    b->O = (float*)p; p += vec;
    b->G3 = (float*)p; p += vec;
    b->G2 = (float*)p; p += act1;
    b->G1 = (float*)p; p += act1;
    b->wpart = (float*)p;
  }
  return BF_OK;
}

NetArgs net_args(const bf_net* net, const bf_graph* g) {
  NetArgs a;
  memset(&a, 0, sizeof(a));
  a.nx = (int)g->nx;
  a.ny = (int)g->ny;
  a.n = g->n;
  a.guide = (const float*)g->guide;
  a.d = (const float*)g->d;
  (void)net;
  return a;
}

template <int CIN, int COUT, int IN, int OUT>
int launch_conv(const NetArgs& a, int cols, cudaStream_t s) {
  const dim3 grid((unsigned)((a.nx + NET_TW - 1) / NET_TW), (unsigned)((a.ny + NET_TH - 1) / NET_TH), (unsigned)cols);
  BF_LAUNCH_PDL((k_net_conv<CIN, COUT, IN, OUT>), grid, NET_TW * NET_TH, 0, s, a);
  BF_CUDA(cudaGetLastError());
  return BF_OK;
}

// the block sums for rho of `cols` columns of r (and zz of z when given)
int net_sums(const bf_graph* g, const float* r, int64_t ldr, const float* z, int cols, const Bufs& b,
             cudaStream_t s, const int* stop = nullptr) {
  const int64_t n = g->n;
  const int nb = net_sum_blocks(n);
  BF_LAUNCH_PDL(k_net_sums, dim3(nb, cols), 256, 0, s, r, ldr, (const float*)g->d, z, n, b.dpart, stop);
  BF_CUDA(cudaGetLastError());
  return BF_OK;
}

int check_pair(const bf_net* net, const bf_graph* g) {
  if (!net || !g) return bf_fail(BF_EINVAL, "bf_net: NULL argument");
  if (g->esize != 4) return bf_fail(BF_EINVAL, "bf_net: the net works on FP32 graphs");
  if (g->nx > 0x7fffffff / 2 || g->ny > 65535 * NET_TH) return bf_fail(BF_EINVAL, "bf_net: image too large");
  return BF_OK;
}

}  // namespace

// ------------------------------------------------------------------ exported
int bf_net_apply_f32(const bf_net* net_c, const bf_graph* g, const float* R, int64_t ldr, int k, float* Z,
                     int64_t ldz, cudaStream_t s, const int* stop) {
  bf_net* net = const_cast<bf_net*>(net_c);
  int rc = check_pair(net, g);
  if (rc) return rc;
  for (int c0 = 0; c0 < k; c0 += NET_COLS) {
    const int cols = std::min(NET_COLS, k - c0);
    Bufs b;
    rc = net_ws(net, g, cols, false, &b);
    if (rc) return rc;
    rc = net_sums(g, R + c0, ldr, nullptr, cols, b, s, stop);
    if (rc) return rc;
    NetArgs a = net_args(net, g);
    a.stop = stop;
    a.r = R + c0;
    a.ldr = ldr;
    a.rho = b.rho;
    a.rpart = b.dpart;
    a.nrp = net_sum_blocks(g->n);
    a.zz = nullptr;
    a.w = net->wq + NET_W1;
    a.out = b.A1;
    if ((rc = launch_conv<NET_CIN, NET_CH, IN_NET, OUT_ACT>(a, cols, s))) return rc;
    a.in = b.A1;
    a.w = net->wq + NET_W2;
    a.out = b.A2;
    if ((rc = launch_conv<NET_CH, NET_CH, IN_RELU, OUT_ACT>(a, cols, s))) return rc;
    a.in = b.A2;
    a.w = net->wq + NET_W3;
    a.z = Z + c0;
    a.ldz = ldz;
    if ((rc = launch_conv<NET_CH, 1, IN_RELU, OUT_PRECOND>(a, cols, s))) return rc;
  }
  return BF_OK;
}

extern "C" int bf_net_create(const float* w_host, bf_net** out) {
  if (!w_host || !out) return bf_fail(BF_EINVAL, "bf_net_create: NULL argument");
  *out = nullptr;
  bf_net* net = new bf_net();
  memset(net, 0, sizeof(*net));
  BF_CUDA(cudaGetDevice(&net->device));
  const size_t wb = NET_NW * sizeof(float);
  cudaError_t e = cudaMalloc(&net->w, 5 * wb + 256);
  if (e != cudaSuccess) {
    delete net;
    return bf_cuda_fail(e, "cudaMalloc(net)");
  }
  net->wq = net->w + NET_NW;
  net->m = net->wq + NET_NW;
  net->v = net->m + NET_NW;
  net->grad = net->v + NET_NW;
  net->loss = reinterpret_cast<double*>(net->grad + NET_NW + (NET_NW & 1));
  BF_CUDA(cudaMemcpy(net->w, w_host, wb, cudaMemcpyHostToDevice));
  BF_CUDA(cudaMemset(net->m, 0, 3 * wb + 2 * sizeof(double)));
  BF_LAUNCH((k_net_round<<<(NET_NW + 255) / 256, 256>>>(net->w, net->wq, NET_NW)));
  BF_CUDA(cudaDeviceSynchronize());
  *out = net;
  return BF_OK;
}

extern "C" int bf_net_free(bf_net* net) {
  if (!net) return BF_OK;
  if (net->ws) cudaFree(net->ws);
  if (net->w) cudaFree(net->w);
  delete net;
  return BF_OK;
}

extern "C" int bf_net_nweights(void) { return NET_NW; }

extern "C" int bf_net_weights(const bf_net* net, float* w_host, int rounded) {
  if (!net || !w_host) return bf_fail(BF_EINVAL, "bf_net_weights: NULL argument");
  BF_CUDA(cudaMemcpy(w_host, rounded ? net->wq : net->w, NET_NW * sizeof(float), cudaMemcpyDeviceToHost));
  return BF_OK;
}

extern "C" int bf_net_apply(const bf_net* net, const bf_graph* g, const float* R, int64_t ldr, int k, float* Z,
                            int64_t ldz, void* stream) {
  if (!R || !Z) return bf_fail(BF_EINVAL, "bf_net_apply: NULL argument");
  if (k < 1 || ldr < k || ldz < k) return bf_fail(BF_EINVAL, "bf_net_apply: need 1 <= k <= ld");
  return bf_net_apply_f32(net, g, R, ldr, k, Z, ldz, (cudaStream_t)stream, nullptr);
}

extern "C" int bf_net_zero_grad(bf_net* net, void* stream) {
  if (!net) return bf_fail(BF_EINVAL, "bf_net_zero_grad: NULL argument");
  cudaStream_t s = (cudaStream_t)stream;
  BF_CUDA(cudaMemsetAsync(net->grad, 0, NET_NW * sizeof(float), s));
  BF_CUDA(cudaMemsetAsync(net->loss, 0, sizeof(double), s));
  return BF_OK;
}

extern "C" int bf_net_accumulate(bf_net* net, const bf_graph* g, const float* r, const float* z, void* stream) {
  int rc = check_pair(net, g);
  if (rc) return rc;
  if (!r || !z) return bf_fail(BF_EINVAL, "bf_net_accumulate: NULL argument");
  cudaStream_t s = (cudaStream_t)stream;
  Bufs b;
  if ((rc = net_ws(net, g, 1, true, &b))) return rc;
  if ((rc = net_sums(g, r, 1, z, 1, b, s))) return rc;
  NetArgs a = net_args(net, g);
  a.r = r;
  a.ldr = 1;
  a.rho = b.rho;
  a.rpart = b.dpart;
  a.nrp = net_sum_blocks(g->n);
  a.zz = b.zz;
  // forward, keeping the pre-activations
  a.w = net->wq + NET_W1;
  a.out = b.A1;
  if ((rc = launch_conv<NET_CIN, NET_CH, IN_NET, OUT_ACT>(a, 1, s))) return rc;
  a.in = b.A1;
  a.w = net->wq + NET_W2;
  a.out = b.A2;
  if ((rc = launch_conv<NET_CH, NET_CH, IN_RELU, OUT_ACT>(a, 1, s))) return rc;
  a.in = b.A2;
  a.w = net->wq + NET_W3;
  a.out = b.O;
  if ((rc = launch_conv<NET_CH, 1, IN_RELU, OUT_ACT>(a, 1, s))) return rc;
  // loss and dL/dO
  const int64_t n = g->n;
  const int nb = net_sum_blocks(n);
  BF_LAUNCH_PDL(k_net_loss, nb, 256, 0, s, b.O, z, b.rho, b.zz, n, b.G3, b.dpart);
  // backward: G2 = conv^T(G3, W3) * (A2 > 0), G1 = conv^T(G2, W2) * (A1 > 0)
  a.transpose = 1;
  a.in = b.G3;
  a.w = net->wq + NET_W3;
  a.out = b.G2;
  a.mask = b.A2;
  if ((rc = launch_conv<1, NET_CH, IN_PLAIN, OUT_MASKED>(a, 1, s))) return rc;
  a.in = b.G2;
  a.w = net->wq + NET_W2;
  a.out = b.G1;
  a.mask = b.A1;
  if ((rc = launch_conv<NET_CH, NET_CH, IN_PLAIN, OUT_MASKED>(a, 1, s))) return rc;
  a.transpose = 0;
  // weight gradients
  const dim3 tg((unsigned)((a.nx + NET_TW - 1) / NET_TW), (unsigned)((a.ny + NET_TH - 1) / NET_TH));
  const int ntile = (int)(tg.x * tg.y);
  BF_LAUNCH_PDL(k_net_wgrad, dim3(tg.x, tg.y, 3), NET_TW * NET_TH, 0, s, a, b.A1, b.A2, b.G1, b.G2, b.G3, b.wpart);
  BF_LAUNCH_PDL(k_net_wgrad_reduce, (NET_NW + 31) / 32 + 1, 256, 0, s, b.wpart, ntile, net->grad, b.dpart, nb, b.zz,
                net->loss);
  BF_CUDA(cudaGetLastError());
  return BF_OK;
}

extern "C" int bf_net_grad(const bf_net* net, float* grad_host, double* loss_host, void* stream) {
  if (!net) return bf_fail(BF_EINVAL, "bf_net_grad: NULL argument");
  cudaStream_t s = (cudaStream_t)stream;
  if (grad_host) BF_CUDA(cudaMemcpyAsync(grad_host, net->grad, NET_NW * sizeof(float), cudaMemcpyDeviceToHost, s));
  if (loss_host) BF_CUDA(cudaMemcpyAsync(loss_host, net->loss, sizeof(double), cudaMemcpyDeviceToHost, s));
  BF_CUDA(cudaStreamSynchronize(s));
  return BF_OK;
}

extern "C" int bf_net_adam(bf_net* net, float lr, float scale, void* stream) {
  if (!net) return bf_fail(BF_EINVAL, "bf_net_adam: NULL argument");
  if (!(lr >= 0.0f) || !(scale > 0.0f)) return bf_fail(BF_EINVAL, "bf_net_adam: bad lr or scale");
  cudaStream_t s = (cudaStream_t)stream;
  net->t += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f - powf(b1, (float)net->t), c2 = 1.0f - powf(b2, (float)net->t);
  if (scale != 1.0f) {
    // the accumulated gradient is a sum over pairs: scale = 1 / pairs makes it a mean
    BF_LAUNCH((k_net_scale<<<(NET_NW + 255) / 256, 256, 0, s>>>(net->grad, NET_NW, scale)));
  }
  BF_LAUNCH((k_net_adam<<<(NET_NW + 255) / 256, 256, 0, s>>>(net->w, net->wq, net->m, net->v, net->grad, NET_NW, lr,
                                                              b1, b2, 1e-8f, c1, c2)));
  BF_CUDA(cudaMemsetAsync(net->loss, 0, sizeof(double), s));
  BF_CUDA(cudaGetLastError());
  return BF_OK;
}
