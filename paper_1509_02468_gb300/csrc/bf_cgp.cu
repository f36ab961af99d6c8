// Algorithm 2 (Section 5) in ONE cooperative launch, for problems whose vectors fit on the
// chip (152 SMs x 227 KB of shared memory).
//
// One CTA per SM owns a rectangle of the image (or a piece of the signal) and keeps its
// share of x, s, p, q, the degree and the guide (or the weights) in shared memory for the
// whole run.  What bounds such a problem is not arithmetic but the serial chain of an
// iteration: two kernels, each with a launch, a cold staging of its tiles and a last-block
// reduction (14 + 12 us per iteration at 512 x 512 against 1.6 us of arithmetic).  Here an
// iteration is
//   p = s + beta p on the rectangle and its halo (the neighbours' s is read from L2),
//   q = (L + sigma I) p, p^T q  ->  all-reduce, alpha,
//   x += alpha p, s -= alpha T q, the four sums, the frame of s to L2  ->  all-reduce, beta,
// and the all-reduces are the only grid-wide synchronisation: every CTA writes its partial
// sums to a slot of its own and reads all slots, so the sums come with the barrier (one
// write and one polled read of L2 instead of an atomic, a poll and a read).  A double is
// sent as two 64-bit words {epoch, half}, each of which is written and read whole, so a word
// with the awaited epoch carries its data.  All CTAs add the partials in the same order and
// take the same decisions.
//
// Every wait is bounded (1 s by %globaltimer): a CTA that gives up sets the status to
// CG_TIMEOUT; the others see it and leave too.
#include <math.h>

#include <algorithm>

#include "bf_cg.cuh"
#include "bf_run.cuh"

namespace {

#define CGP_T 512                          // threads of an image CTA
#define CGP_TL 256                         // threads of a signal CTA
#define CGP_SLOT 8                         // words of a CTA's slot (four doubles)
#define CGP_MAXC 256                       // most CTAs of a launch
#define CGP_WAIT_NS 1000000000ull
#define CGP_HALO_REGS 4                    // halo pixels a thread can own
typedef unsigned long long u64;

// Words {epoch, payload} of the all-reduce and the scalars every CTA computes for itself.
struct CgpShared {
  double red[4][CGP_T / 32];
  double tot[4];
  double alpha, beta;
  double sr, ss, rr, ref2;
  int status;
};

__device__ __forceinline__ u64 cgp_now() {
  u64 t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// a / b by an FP32 seed and Newton steps in FP64 (a divide is twice as long a chain); the
// last step corrects the quotient, so it is right to the last bit or two.  Values the seed
// cannot hold take the divide.
__device__ __forceinline__ double cgp_div(double a, double b) {
  const double ab = fabs(b);
  if (!(ab > 1e-30 && ab < 1e30)) return a / b;
  double r = (double)__frcp_rn((float)b);
  r = fma(r, fma(-b, r, 1.0), r);
  r = fma(r, fma(-b, r, 1.0), r);
  const double q = a * r;
  return fma(r, fma(-b, q, a), q);
}

// Warp sums of four values at once: 6 additions instead of 20 (an FP64 instruction holds
// the scheduler's FP64 pipe for 64 cycles); value ((lane >> 3) & 3) is returned in a lane.
template <typename T>
__device__ __forceinline__ T cgp_warp4(const T (&v)[4], int lane) {
  const bool h16 = lane & 16, h8 = lane & 8;
  T a = h16 ? v[2] : v[0], b = h16 ? v[3] : v[1];
  a += __shfl_xor_sync(0xffffffffu, h16 ? v[0] : v[2], 16);
  b += __shfl_xor_sync(0xffffffffu, h16 ? v[1] : v[3], 16);
  T c = h8 ? b : a;
  c += __shfl_xor_sync(0xffffffffu, h8 ? a : b, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  return c;
}

// Sums of v over all threads of all CTAs into sh.tot (valid in warps 0 .. NV - 1, value w in
// warp w, lane 0 writes it); a barrier of the grid.  Returns false (in every thread) when a
// wait gave up.  The caller synchronises the CTA before using sh.tot in other warps.
template <int NV, int NT, typename T>
__device__ bool cgp_allreduce(const T (&v)[4], CgpShared& sh, unsigned* words, u64* slots, unsigned epoch,
                              CgState* st) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nc = gridDim.x;
  u64* base = slots + (size_t)(epoch & 1) * CGP_MAXC * CGP_SLOT;
  if (NV == 4) {
    const T w = cgp_warp4<T>(v, lane);
    if ((lane & 7) == 0) sh.red[lane >> 3][wid] = (double)w;
  } else {
    const T w = warp_sum(v[0]);
    if (lane == 0) sh.red[0][wid] = (double)w;
  }
  __syncthreads();
  if (wid < NV) {
    double t = lane < NT / 32 ? sh.red[wid][lane] : 0.0;
#pragma unroll
    for (int o = NT / 64; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane < 2) {
      const u64 bits = (u64)__double_as_longlong(t);
      const u64 word = ((u64)epoch << 32) | (lane ? (bits >> 32) : (bits & 0xffffffffull));
      __threadfence();                     // the CTA's stores before the barrier above come first
      *(volatile u64*)(base + blockIdx.x * CGP_SLOT + 2 * wid + lane) = word;
    }
  }
  // read every CTA's words of these NV values
  int bad = 0;
  for (int w = threadIdx.x; w < nc * 2 * NV; w += NT) {
    const volatile u64* p = base + (w / (2 * NV)) * CGP_SLOT + (w % (2 * NV));
    u64 word = *p;
    if ((unsigned)(word >> 32) != epoch) {
      const u64 t0 = cgp_now();
      for (;;) {
        word = *p;
        if ((unsigned)(word >> 32) == epoch) break;
        if (*(volatile int*)&st->status == CG_TIMEOUT) { bad = 1; break; }
        if (cgp_now() - t0 > CGP_WAIT_NS) {
          atomicExch(&st->status, CG_TIMEOUT);
          bad = 1;
          break;
        }
      }
      if (bad) break;
    }
    words[w] = (unsigned)word;
  }
  __threadfence();                         // later reads see what the others wrote before
  if (__syncthreads_or(bad)) return false;
  if (wid < NV) {
    double t = 0.0;
    for (int c = lane; c < nc; c += 32) {
      const unsigned* p = words + c * 2 * NV + 2 * wid;
      t += __longlong_as_double((long long)(((u64)p[1] << 32) | p[0]));
    }
    t = warp_sum(t);
    if (lane == 0) sh.tot[wid] = t;
  }
  return true;
}

// The scalar steps, by thread 0 of every CTA (all take the same values); CTA 0 keeps the
// history.  Start: the state from the sums s^T r, s^T s, r^T r, x0^T x0.
__device__ void cgp_start_scalars(CgpShared& sh, double shift) {
  sh.sr = sh.tot[0];
  sh.ss = sh.tot[1];
  sh.rr = sh.tot[2];
  const double b2 = shift * shift * sh.tot[3];
  sh.ref2 = b2 > 0.0 ? b2 : sh.tot[2];
  sh.alpha = sh.beta = 0.0;
  sh.status = (isfinite(sh.tot[0]) && isfinite(sh.tot[1]) && isfinite(sh.tot[2])) ? CG_RUN : CG_NONFINITE;
}
// Direction: p^T q in tot[0].
__device__ void cgp_dir_scalars(CgpShared& sh) {
  const double pq = sh.tot[0];
  if (sh.sr == 0.0) sh.status = CG_CONV;
  else if (!isfinite(pq)) sh.status = CG_NONFINITE;
  else if (!(pq > 0.0)) sh.status = CG_BREAK;
  else sh.alpha = cgp_div(sh.sr, pq);
}
// Update: s^T r, s^T q, s^T s, r^T r.
__device__ void cgp_update_scalars(CgpShared& sh, int it, int beta_mode, double tol2, double* hist) {
  if (hist && blockIdx.x == 0) {
    hist[2 * it] = sh.alpha;
    hist[2 * it + 1] = it == 0 ? 0.0 : sh.beta;
  }
  const double den = beta_mode == BF_BETA_PRINTED ? sh.ss : sh.sr;
  sh.beta = cgp_div(-sh.alpha * sh.tot[1], den);
  sh.sr = sh.tot[0];
  sh.ss = sh.tot[2];
  sh.rr = sh.tot[3];
  if (!(isfinite(sh.tot[0]) && isfinite(sh.tot[1]) && isfinite(sh.tot[2]) && isfinite(sh.tot[3])))
    sh.status = CG_NONFINITE;
  else if (tol2 > 0.0 && sh.tot[3] <= tol2 * sh.ref2)
    sh.status = CG_CONV;
}
__device__ void cgp_write_state(const CgpShared& sh, CgState* st, int iters) {
  st->sr = sh.sr;
  st->ss = sh.ss;
  st->rr = sh.rr;
  st->ref2 = sh.ref2;
  st->alpha = sh.alpha;
  st->beta = sh.beta;
  st->iter = iters;
  atomicCAS(&st->status, CG_RUN, sh.status);    // a timeout recorded by another CTA stays
}

// ---------------------------------------------------------------- images
// A CTA's rectangle: W x H pixels (W % 32 == 0, H % 4 == 0) with origin (bx, by).  Tiles with
// halo have row stride xs = W + 2 LP and origin (bx - LP, by - HALO).
struct CgpRect {
  int W, H, ncx;             // rectangle and rectangles per row of the image
};

// The bilateral operator, 7 x 7 window, weights on the fly: the guide's tile beside p's.
struct CgpBilateral {
  static constexpr int HALO = 3, LP = 4;
  RunConst c;
  const float* guide;
  static __host__ __device__ size_t extra(int W, int H) { return (size_t)(W + 2 * LP) * (H + 2 * HALO); }
  __device__ void stage(float* G, int W, int H, int bx, int by, int nx, int ny) const {
    const int xs = W + 2 * LP;
    for (int q = threadIdx.x; q < xs * (H + 2 * HALO); q += CGP_T) {
      const int hy = q / xs, hx = q - hy * xs;
      const int gy = by - HALO + hy, gx = bx - LP + hx;
      const bool in = (unsigned)gx < (unsigned)nx && (unsigned)gy < (unsigned)ny;
      G[q] = in ? (c.use_guide ? guide[(int64_t)gy * nx + gx] : 0.0f) : __int_as_float(0x7f800000);
    }
  }
  __device__ void prepare(const float*, float*, int, int) const {}
  // (L p) of the run at (x, y) of the rectangle
  __device__ void sums(const float* P, const float* G, int W, int H, int x, int y, float (&vi)[RUN_P],
                       float (&acc)[RUN_P]) const {
    const int xs = W + 2 * LP;
    float ws[RUN_P];
    const int o = y * xs + x;
    run_sums<true, false>(c, P + o, G + o, xs, vi, acc, ws);
  }
};

struct CgpImage {
  CgArgs<float> cg;
  CgpRect rc;
  int nx, ny, kmax, vec;
  u64* slots;
};

template <class OP>
__host__ __device__ inline size_t cgp_image_floats(int W, int H) {
  return (size_t)(W + 2 * OP::LP) * (H + 2 * OP::HALO) + OP::extra(W, H) + 4 * (size_t)W * H;
}

// Halo pixel h of the rectangle's frame: rows above and below (full width plus corners),
// then the columns beside it; (tx, ty) relative to the rectangle.
template <int HALO>
__device__ __forceinline__ void cgp_halo_pos(int h, int W, int H, int& tx, int& ty) {
  const int wide = W + 2 * HALO, nrow = HALO * wide;
  if (h < 2 * nrow) {
    const int k = h < nrow ? h : h - nrow;
    const int r = k / wide;
    tx = k - r * wide - HALO;
    ty = h < nrow ? r - HALO : H + r;
  } else {
    const int k = h - 2 * nrow;
    const int r = k / (2 * HALO), c = k - r * (2 * HALO);
    ty = r;
    tx = c < HALO ? c - HALO : W + c - HALO;
  }
}

template <class OP>
__global__ void __launch_bounds__(CGP_T, 1) k_cgp_image(const __grid_constant__ OP op, const __grid_constant__ CgpImage a) {
  constexpr int HALO = OP::HALO, LP = OP::LP;
  extern __shared__ __align__(16) float cgp_smem[];
  __shared__ CgpShared sh;
  __shared__ unsigned words[CGP_MAXC * CGP_SLOT];
  const int W = a.rc.W, H = a.rc.H, xs = W + 2 * LP;
  const int nx = a.nx, ny = a.ny;
  float* P = cgp_smem;
  float* S = P + (size_t)xs * (H + 2 * HALO);
  float* X = S + W * H;
  float* Q = X + W * H;
  float* D = Q + W * H;
  float* EX = D + W * H;
  const int bx = (blockIdx.x % a.rc.ncx) * W, by = (blockIdx.x / a.rc.ncx) * H;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int ux_n = W / 32, nunits = ux_n * (H / 4);
  const int rx = 4 * (lane & 7), ry = lane >> 3;
  const bool jac = a.cg.dinv != nullptr;
  const int beta_mode = a.cg.st->beta_mode;
  const double tol2 = a.cg.st->tol2;
  // ---- x0 on the rectangle and its halo, the operator's tiles, the degree
  for (int q = threadIdx.x; q < xs * (H + 2 * HALO); q += CGP_T) {
    const int hy = q / xs, hx = q - hy * xs;
    const int gy = by - HALO + hy, gx = bx - LP + hx;
    const bool in = (unsigned)gx < (unsigned)nx && (unsigned)gy < (unsigned)ny;
    P[q] = in ? a.cg.x0[(int64_t)gy * nx + gx] : 0.0f;
  }
  op.stage(EX, W, H, bx, by, nx, ny);
  for (int q = threadIdx.x; q < W * H; q += CGP_T) {
    const int y = q / W, x = q - y * W;
    D[q] = (bx + x < nx && by + y < ny) ? a.cg.d[(int64_t)(by + y) * nx + bx + x] : 1.0f;
  }
  __syncthreads();
  // a run's values of s to the frame that the neighbours read
  auto frame = [&](int x, int y, int cnt, const float (&s)[RUN_P]) {
    if (x < 8 || x >= W - 8 || y < HALO || y >= H - HALO)
      run_store(a.cg.s, (int64_t)(by + y) * nx + bx + x, cnt, a.vec, s);
  };
  // ---- r = -L x0, s = T r
  unsigned epoch = 1;
  {
    float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    op.prepare(P, EX, W, H);
    for (int u = wid; u < nunits; u += CGP_T / 32) {
      const int x = (u % ux_n) * 32 + rx, y = (u / ux_n) * 4 + ry;
      const int cnt = run_count(bx + x, by + y, nx, ny);
      float xi[RUN_P], acc[RUN_P], s[RUN_P];
      op.sums(P, EX, W, H, x, y, xi, acc);
#pragma unroll
      for (int j = 0; j < RUN_P; ++j) {
        s[j] = 0.0f;
        if (j < cnt) {
          const float r = -acc[j];
          s[j] = jac ? __fdiv_rn(r, D[y * W + x + j]) : r;
          v[0] = fmaf(s[j], r, v[0]);
          v[1] = fmaf(s[j], s[j], v[1]);
          v[2] = fmaf(r, r, v[2]);
          v[3] = fmaf(xi[j], xi[j], v[3]);
        }
      }
      *reinterpret_cast<float4*>(S + y * W + x) = make_float4(s[0], s[1], s[2], s[3]);
      *reinterpret_cast<float4*>(X + y * W + x) = make_float4(xi[0], xi[1], xi[2], xi[3]);
      if (cnt) frame(x, y, cnt, s);
    }
    if (!cgp_allreduce<4, CGP_T>(v, sh, words, a.slots, epoch, a.cg.st)) return;
    __syncthreads();
    if (threadIdx.x == 0) cgp_start_scalars(sh, (double)a.cg.shift);
    __syncthreads();
  }
  // this thread's halo pixels: offset in the image (-1: outside) and in the tile
  const int nhalo = 2 * HALO * (W + 2 * HALO) + 2 * HALO * H;
  int it = 0;
  for (; it < a.kmax && sh.status == CG_RUN; ++it) {
    const float beta = it ? (float)sh.beta : 0.0f;
    // ---- p = s + beta p
    float hs[CGP_HALO_REGS];
#pragma unroll
    for (int k = 0; k < CGP_HALO_REGS; ++k) {
      const int h = threadIdx.x + k * CGP_T;
      hs[k] = 0.0f;
      if (h < nhalo) {
        int tx, ty;
        cgp_halo_pos<HALO>(h, W, H, tx, ty);
        const int gx = bx + tx, gy = by + ty;
        if ((unsigned)gx < (unsigned)nx && (unsigned)gy < (unsigned)ny)
          hs[k] = __ldcg(a.cg.s + (int64_t)gy * nx + gx);
      }
    }
    for (int u = wid; u < nunits; u += CGP_T / 32) {
      const int x = (u % ux_n) * 32 + rx, y = (u / ux_n) * 4 + ry;
      const float4 s = *reinterpret_cast<const float4*>(S + y * W + x);
      float4* pp = reinterpret_cast<float4*>(P + (y + HALO) * xs + x + LP);
      float4 p = s;
      if (it) {
        const float4 o = *pp;
        p.x = fmaf(beta, o.x, s.x);
        p.y = fmaf(beta, o.y, s.y);
        p.z = fmaf(beta, o.z, s.z);
        p.w = fmaf(beta, o.w, s.w);
      }
      *pp = p;
    }
#pragma unroll
    for (int k = 0; k < CGP_HALO_REGS; ++k) {
      const int h = threadIdx.x + k * CGP_T;
      if (h < nhalo) {
        int tx, ty;
        cgp_halo_pos<HALO>(h, W, H, tx, ty);
        float* pp = P + (ty + HALO) * xs + tx + LP;
        *pp = it ? fmaf(beta, *pp, hs[k]) : hs[k];
      }
    }
    __syncthreads();
    // ---- q = (L + sigma I) p, p^T q
    float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    op.prepare(P, EX, W, H);
    for (int u = wid; u < nunits; u += CGP_T / 32) {
      const int x = (u % ux_n) * 32 + rx, y = (u / ux_n) * 4 + ry;
      const int cnt = run_count(bx + x, by + y, nx, ny);
      float pi[RUN_P], acc[RUN_P], q[RUN_P];
      op.sums(P, EX, W, H, x, y, pi, acc);
#pragma unroll
      for (int j = 0; j < RUN_P; ++j) {
        q[j] = 0.0f;
        if (j < cnt) {
          q[j] = fmaf(a.cg.shift, pi[j], acc[j]);
          v[0] = fmaf(pi[j], q[j], v[0]);
        }
      }
      *reinterpret_cast<float4*>(Q + y * W + x) = make_float4(q[0], q[1], q[2], q[3]);
    }
    if (!cgp_allreduce<1, CGP_T>(v, sh, words, a.slots, ++epoch, a.cg.st)) return;
    if (threadIdx.x == 0) cgp_dir_scalars(sh);
    __syncthreads();
    if (sh.status != CG_RUN) break;
    // ---- x += alpha p, s -= alpha T q, the sums
    const float alpha = (float)sh.alpha;
    v[0] = 0.0f;
    for (int u = wid; u < nunits; u += CGP_T / 32) {
      const int x = (u % ux_n) * 32 + rx, y = (u / ux_n) * 4 + ry;
      const int cnt = run_count(bx + x, by + y, nx, ny);
      const float4 q4 = *reinterpret_cast<const float4*>(Q + y * W + x);
      const float4 p4 = *reinterpret_cast<const float4*>(P + (y + HALO) * xs + x + LP);
      const float4 d4 = *reinterpret_cast<const float4*>(D + y * W + x);
      const float4 x4 = *reinterpret_cast<const float4*>(X + y * W + x);
      const float4 s4 = *reinterpret_cast<const float4*>(S + y * W + x);
      const float q[4] = {q4.x, q4.y, q4.z, q4.w}, p[4] = {p4.x, p4.y, p4.z, p4.w};
      const float d[4] = {d4.x, d4.y, d4.z, d4.w};
      float xv[4] = {x4.x, x4.y, x4.z, x4.w}, s[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
      for (int j = 0; j < RUN_P; ++j) {       // pixels outside the image hold q = s = 0
        xv[j] = fmaf(alpha, p[j], xv[j]);
        s[j] = fmaf(-alpha, jac ? __fdiv_rn(q[j], d[j]) : q[j], s[j]);
        const float r = jac ? d[j] * s[j] : s[j];
        v[0] = fmaf(s[j], r, v[0]);
        v[1] = fmaf(s[j], q[j], v[1]);
        v[2] = fmaf(s[j], s[j], v[2]);
        v[3] = fmaf(r, r, v[3]);
      }
      *reinterpret_cast<float4*>(X + y * W + x) = make_float4(xv[0], xv[1], xv[2], xv[3]);
      *reinterpret_cast<float4*>(S + y * W + x) = make_float4(s[0], s[1], s[2], s[3]);
      if (cnt) frame(x, y, cnt, s);
    }
    if (!cgp_allreduce<4, CGP_T>(v, sh, words, a.slots, ++epoch, a.cg.st)) return;
    __syncthreads();
    if (threadIdx.x == 0) cgp_update_scalars(sh, it, beta_mode, tol2, a.cg.hist);
    __syncthreads();
  }
  for (int u = wid; u < nunits; u += CGP_T / 32) {
    const int x = (u % ux_n) * 32 + rx, y = (u / ux_n) * 4 + ry;
    const int cnt = run_count(bx + x, by + y, nx, ny);
    const float4 x4 = *reinterpret_cast<const float4*>(X + y * W + x);
    const float xv[4] = {x4.x, x4.y, x4.z, x4.w};
    if (cnt) run_store(a.cg.x, (int64_t)(by + y) * nx + bx + x, cnt, a.vec && (((uintptr_t)a.cg.x & 15) == 0), xv);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) cgp_write_state(sh, a.cg.st, it);
}

// ---------------------------------------------------------------- signals
// Any interval window of radius R on a signal: the CTA keeps the weights of its forward
// pairs (i, i + t), t = 1 .. R, i from R samples before its piece to its end, so that an
// iteration has no exponentials (in FP64 they were 9/10 of the arithmetic at 2 FMA per clock
// and SM).  Generic recurrences: r and s = T r are both kept.
template <typename T>
struct CgpLine {
  CgArgs<T> cg;
  T a_r;
  T ls[BF_MAX_R1D + 1];
  int n, R, W, kmax;
  u64* slots;
};

__host__ __device__ inline size_t cgp_line_elems(int W, int R) {
  return (size_t)(W + 2 * R) + 5 * (size_t)W + (size_t)R * (W + R);
}

template <typename T>
__global__ void __launch_bounds__(CGP_TL, 1) k_cgp_line(const __grid_constant__ CgpLine<T> a) {
  extern __shared__ __align__(16) float cgp_smem[];
  __shared__ CgpShared sh;
  __shared__ unsigned words[CGP_MAXC * CGP_SLOT];
  const int W = a.W, R = a.R, n = a.n;
  const int beta_mode = a.cg.st->beta_mode;
  const double tol2 = a.cg.st->tol2;
  T* P = reinterpret_cast<T*>(cgp_smem);       // [W + 2 R], origin b - R
  T* S = P + W + 2 * R;
  T* RR = S + W;
  T* X = RR + W;
  T* Q = X + W;
  T* DI = Q + W;
  T* WF = DI + W;                              // [R][W + R], origin b - R
  const int b = blockIdx.x * W, len = min(W, n - b);
  // ---- x0 with halo, 1 / d, the weights
  for (int q = threadIdx.x; q < W + 2 * R; q += CGP_TL) {
    const int i = b - R + q;
    P[q] = (unsigned)i < (unsigned)n ? a.cg.x0[i] : T(0);
  }
  for (int q = threadIdx.x; q < len; q += CGP_TL) DI[q] = a.cg.dinv ? a.cg.dinv[b + q] : T(1);
  for (int q = threadIdx.x; q < R * (W + R); q += CGP_TL) {
    const int t = q / (W + R), i = b - R + (q - t * (W + R)), j = i + t + 1;
    T w = T(0);
    if (i >= 0 && j < n) {
      if (a.cg.wmode == BF_W_ONTHEFLY) {
        const T dl = a.cg.guide[i] - a.cg.guide[j];
        w = bf_exp_w(fma(-dl * a.a_r, dl, a.ls[t + 1]));
      } else {
        w = (T)ld_weight(a.cg.wf, (int64_t)t * n + i, a.cg.wmode);
      }
    }
    WF[q] = w;
  }
  __syncthreads();
  auto lap = [&](int q) {                      // (L p) of sample q of the piece
    const T pi = P[q + R];
    T acc = T(0);
    for (int t = 1; t <= R; ++t) {
      const T* wt = WF + (t - 1) * (W + R) + q + R;
      acc = fma(wt[0], pi - P[q + R + t], acc);
      acc = fma(wt[-t], pi - P[q + R - t], acc);
    }
    return acc;
  };
  unsigned epoch = 1;
  {
    T v[4] = {T(0), T(0), T(0), T(0)};
    for (int q = threadIdx.x; q < len; q += CGP_TL) {
      const T xi = P[q + R], r = -lap(q), s = a.cg.dinv ? r * DI[q] : r;
      X[q] = xi;
      RR[q] = r;
      S[q] = s;
      if (q < R || q >= len - R) a.cg.s[b + q] = s;
      v[0] = fma(s, r, v[0]);
      v[1] = fma(s, s, v[1]);
      v[2] = fma(r, r, v[2]);
      v[3] = fma(xi, xi, v[3]);
    }
    if (!cgp_allreduce<4, CGP_TL>(v, sh, words, a.slots, epoch, a.cg.st)) return;
    __syncthreads();
    if (threadIdx.x == 0) cgp_start_scalars(sh, (double)a.cg.shift);
    __syncthreads();
  }
  int it = 0;
  for (; it < a.kmax && sh.status == CG_RUN; ++it) {
    const T beta = it ? (T)sh.beta : T(0);
    for (int h = threadIdx.x; h < 2 * R; h += CGP_TL) {        // halo
      const int i = h < R ? b - R + h : b + W + h - R;
      T* pp = P + (h < R ? h : W + h);
      const T s = (unsigned)i < (unsigned)n ? __ldcg(a.cg.s + i) : T(0);
      *pp = it ? fma(beta, *pp, s) : s;
    }
    for (int q = threadIdx.x; q < W; q += CGP_TL) {
      const T s = q < len ? S[q] : T(0);
      P[q + R] = it ? fma(beta, P[q + R], s) : s;
    }
    __syncthreads();
    T v[4] = {T(0), T(0), T(0), T(0)};
    for (int q = threadIdx.x; q < len; q += CGP_TL) {
      const T p = P[q + R], qq = fma(a.cg.shift, p, lap(q));
      Q[q] = qq;
      v[0] = fma(p, qq, v[0]);
    }
    if (!cgp_allreduce<1, CGP_TL>(v, sh, words, a.slots, ++epoch, a.cg.st)) return;
    if (threadIdx.x == 0) cgp_dir_scalars(sh);
    __syncthreads();
    if (sh.status != CG_RUN) break;
    const T alpha = (T)sh.alpha;
    v[0] = T(0);
    for (int q = threadIdx.x; q < len; q += CGP_TL) {
      const T qq = Q[q];
      X[q] = fma(alpha, P[q + R], X[q]);
      const T r = fma(-alpha, qq, RR[q]), s = a.cg.dinv ? r * DI[q] : r;
      RR[q] = r;
      S[q] = s;
      if (q < R || q >= len - R) a.cg.s[b + q] = s;
      v[0] = fma(s, r, v[0]);
      v[1] = fma(s, qq, v[1]);
      v[2] = fma(s, s, v[2]);
      v[3] = fma(r, r, v[3]);
    }
    if (!cgp_allreduce<4, CGP_TL>(v, sh, words, a.slots, ++epoch, a.cg.st)) return;
    __syncthreads();
    if (threadIdx.x == 0) cgp_update_scalars(sh, it, beta_mode, tol2, a.cg.hist);
    __syncthreads();
  }
  for (int q = threadIdx.x; q < len; q += CGP_TL) a.cg.x[b + q] = X[q];
  if (blockIdx.x == 0 && threadIdx.x == 0) cgp_write_state(sh, a.cg.st, it);
}

// ---------------------------------------------------------------- host
#define CGP_SMEM_MAX (214 * 1024)          // dynamic part; the static part is about 9 KB

// CTAs a launch may have: four SMs stay free for one-CTA kernels of other streams (the
// Rayleigh-Ritz solve of a LOBPCG run beside this one), which the cooperative launch would
// otherwise wait for.
int cgp_max_ctas() {
  static int n = 0;
  if (n == 0) {
    int dev = 0, sms = 0, coop = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    n = coop ? std::max(1, std::min(CGP_MAXC, sms - 4)) : -1;
  }
  return n;
}

// The rectangle split of an image with the fewest units of 32 x 4 pixels per scheduler, then
// the smallest halo; false: the image does not fit.
template <class OP>
bool cgp_rect(int nx, int ny, CgpRect* out, int* nreg) {
  const int maxc = cgp_max_ctas();
  long best = -1;
  for (int W = 32; W <= 256; W += 32) {
    const int ncx = (nx + W - 1) / W;
    if (ncx > maxc) continue;
    const int want = std::min(maxc / ncx, (ny + 3) / 4);
    const int H = 4 * ((ny + 4 * want - 1) / (4 * want)), ncy = (ny + H - 1) / H;
    const int nhalo = 2 * OP::HALO * (W + 2 * OP::HALO) + 2 * OP::HALO * H;
    if (cgp_image_floats<OP>(W, H) * 4 > CGP_SMEM_MAX || nhalo > CGP_HALO_REGS * CGP_T) continue;
    const long cost = (long)((W / 32 * (H / 4) + 3) / 4) * 100000 + nhalo;
    if (best < 0 || cost < best) {
      best = cost;
      out->W = W;
      out->H = H;
      out->ncx = ncx;
      *nreg = ncx * ncy;
    }
  }
  return best >= 0;
}

// Samples per CTA of a signal: at least 64 (a smaller piece only adds partial sums to add),
// 0 if it does not fit.
int cgp_line_width(const bf_graph* g) {
  const int maxc = cgp_max_ctas();
  if (maxc < 1) return 0;
  int64_t W = std::max<int64_t>(64, (g->n + maxc - 1) / maxc);
  W = std::max<int64_t>((W + 31) / 32 * 32, 2 * g->rx);
  return cgp_line_elems((int)std::min<int64_t>(W, 1 << 20), g->rx) * g->esize > CGP_SMEM_MAX ? 0 : (int)W;
}

bool cgp_is_line(const bf_graph* g) {
  return g->kind == BF_KIND_BILATERAL && g->p.ndim == 1 && g->ry == 0 && g->n < (1 << 30);
}
bool cgp_is_image(const bf_graph* g) {
  return g->kind == BF_KIND_BILATERAL && fast_shape(g) == FAST_R3_2D && g->p.weight_mode == BF_W_ONTHEFLY;
}

template <class F, class A>
int cgp_coop(F fn, int grid, int threads, size_t smem, cudaStream_t s, A& args) {
  int rc = bf_smem_attr((const void*)fn, CGP_SMEM_MAX, "cudaFuncSetAttribute(k_cgp)");
  if (rc) return rc;
  BF_LAUNCH((void)cudaLaunchCooperativeKernel((const void*)fn, dim3(grid), dim3(threads), args, smem, s));
  BF_CUDA(cudaGetLastError());
  return BF_OK;
}

}  // namespace

size_t cgp_words(const bf_graph* g) {
  if (cgp_max_ctas() < 1) return 0;
  CgpRect rc;
  int nreg = 0;
  bool ok = false;
  if (cgp_is_line(g)) ok = cgp_line_width(g) > 0;
  else if (cgp_is_image(g)) ok = cgp_rect<CgpBilateral>(g->nx, g->ny, &rc, &nreg);
  return ok ? 2 * CGP_MAXC * CGP_SLOT : 0;
}

template <>
int cgp_launch<float>(const bf_graph* g, const CgArgs<float>& cg, int kmax, cudaStream_t s);
template <>
int cgp_launch<double>(const bf_graph* g, const CgArgs<double>& cg, int kmax, cudaStream_t s);

template <typename T>
static int launch_line(const bf_graph* g, const CgArgs<T>& cg, int kmax, cudaStream_t s) {
  CgpLine<T> a;
  memset(&a, 0, sizeof(a));
  const Geom<T>& G = geom_of<T>(g);
  a.cg = cg;
  a.a_r = G.a_r;
  a.n = (int)g->n;
  a.R = g->rx;
  for (int t = 1; t <= g->rx; ++t) a.ls[t] = G.ls[g->rx + t];
  a.W = cgp_line_width(g);
  a.kmax = kmax;
  a.slots = (u64*)cg.partials;
  void* args[] = {&a};
  const int grid = (a.n + a.W - 1) / a.W;
  return cgp_coop(k_cgp_line<T>, grid, CGP_TL, cgp_line_elems(a.W, a.R) * sizeof(T), s, args);
}

template <>
int cgp_launch<double>(const bf_graph* g, const CgArgs<double>& cg, int kmax, cudaStream_t s) {
  return launch_line<double>(g, cg, kmax, s);
}

template <>
int cgp_launch<float>(const bf_graph* g, const CgArgs<float>& cg, int kmax, cudaStream_t s) {
  if (cgp_is_line(g)) return launch_line<float>(g, cg, kmax, s);
  CgpImage a;
  memset(&a, 0, sizeof(a));
  int nreg = 0;
  if (!cgp_rect<CgpBilateral>(g->nx, g->ny, &a.rc, &nreg)) return bf_fail(BF_EINVAL, "cg_filter: image does not fit");
  CgpBilateral op;
  op.c = run_const(g->gf);
  op.guide = cg.guide;
  a.cg = cg;
  a.nx = g->nx;
  a.ny = g->ny;
  a.kmax = kmax;
  a.vec = g->nx % 4 == 0;
  a.slots = (u64*)cg.partials;
  void* args[] = {&op, &a};
  return cgp_coop(k_cgp_image<CgpBilateral>, nreg, CGP_T, cgp_image_floats<CgpBilateral>(a.rc.W, a.rc.H) * 4, s, args);
}
