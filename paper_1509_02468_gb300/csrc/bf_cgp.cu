// Algorithm 2 (Section 5) in ONE cooperative launch, for problems whose vectors fit on the
// chip (152 SMs x 227 KB of shared memory).
//
// One CTA per SM owns a rectangle of the image (or a piece of the signal) and keeps its
// share of x, s, p, q, the degree and the guide (or the weights) in shared memory for the
// whole run.  What bounds such a problem is not arithmetic but the serial chain of an
// iteration: two kernels, each with a launch, a cold staging of its tiles and a last-block
// reduction (14 + 12 us per iteration at 512 x 512 against 1.6 us of arithmetic).  Here an
// iteration is
//   p = s + beta p on the rectangle and its halo (the neighbours' s comes through L2),
//   q = (L + sigma I) p, p^T q  ->  all-reduce, alpha,
//   x += alpha p, s -= alpha T q, the four sums, the frame of s to L2  ->  all-reduce, beta.
// Nothing else synchronises the grid, and nothing needs a fence: what a CTA sends (partial
// sums, frame values) goes out as 64-bit words {epoch, 32 data bits}, each written and read
// whole, and the receiver polls the word until it carries the awaited epoch.  So an
// all-reduce is one write and one polled read of L2, and the halo words, written before it,
// are there when it is done.  (With plain stores, a fence on either side and FP64 additions
// the two all-reduces of an iteration took 17 of its 27 thousand cycles at 512 x 512.)
// All CTAs add the partials alike and take the same decisions; sums and scalars are pairs of
// floats in FP32 runs and FP64 in FP64 runs (see below).  50 iterations of 512 x 512 pixels:
// 436 us (two launches per iteration: 1347, and 1143 with this file's window sums); the
// exchange is 2300 cycles per all-reduce of 144 CTAs with a line of L2 per slot, 3100 with half
// a line, 7200 with slots packed, 2790 with an atomic counter.
//
// Every wait is bounded (1 s by %globaltimer): a CTA that gives up sets the status to
// CG_TIMEOUT; the others see it and leave too, each with its part of x as far as it has come.
#include <math.h>

#include <algorithm>

#include "bf_cg.cuh"
#include "bf_run.cuh"
#include "bf_window_fast.cuh"

namespace {

#define CGP_T 512                          // threads of an image CTA
#define CGP_TL 256                         // threads of a signal CTA
#define CGP_SLOT 16                        // words of a CTA's slot: a line of L2 of its own
#define CGP_MAXC 256                       // most CTAs of a launch
#define CGP_WAIT_NS 1000000000ull
#define CGP_HALO_REGS 4                    // halo pixels a thread can own
typedef unsigned long long u64;

__device__ __forceinline__ u64 cgp_now() {
  u64 t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ---- words in flight
__device__ __forceinline__ u64 cgp_word(unsigned epoch, unsigned data) { return ((u64)epoch << 32) | data; }
__device__ __forceinline__ void cgp_put(u64* p, u64 w) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ u64 cgp_get(const u64* p) {
  u64 w;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ void cgp_get2(const u64* p, u64& a, u64& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
// One more look at the clock and at the others: whether to give up waiting.
__device__ bool cgp_give_up(u64 t0, CgState* st) {
  if (*(volatile int*)&st->status == CG_TIMEOUT) return true;
  if (cgp_now() - t0 <= CGP_WAIT_NS) return false;
  atomicExch(&st->status, CG_TIMEOUT);
  return true;
}
// Poll a word (a pair of words) until it carries `epoch`; false: gave up.
__device__ bool cgp_wait(const u64* p, u64& w, unsigned epoch, CgState* st) {
  const u64 t0 = cgp_now();
  for (unsigned n = 1;; ++n) {
    w = cgp_get(p);
    if ((unsigned)(w >> 32) == epoch) return true;
    if (n % 64 == 0 && cgp_give_up(t0, st)) return false;
  }
}
__device__ bool cgp_wait2(const u64* p, u64& a, u64& b, unsigned epoch, CgState* st) {
  const u64 t0 = cgp_now();
  for (unsigned n = 1;; ++n) {
    cgp_get2(p, a, b);
    if ((unsigned)(a >> 32) == epoch && (unsigned)(b >> 32) == epoch) return true;
    if (n % 64 == 0 && cgp_give_up(t0, st)) return false;
  }
}

// ---- sums and scalars
// A dependent FP64 addition takes about 115 cycles here and holds its scheduler's pipe for
// 64, so FP32 runs carry their sums and scalars as unevaluated pairs of floats h + l (48 bits;
// the terms are FP32 warp sums): an addition (Knuth's two-sum) is a chain of six 4-cycle
// operations.  FP64 runs use FP64.
// Sums are kept times a power of two (exact).  It is taken from the start's sums and again
// from s^T r whenever that has left the range 2^+-CgpRange::BAND (cgp_prepare_beta): the sums
// fall with the square of the residual, far past the range of a float (and, in FP64 runs, to
// where alpha / s^T r overflows), while a run may go on for as long as the FP32 (FP64) terms
// themselves have not vanished.  Scale and beta's factor are made while the update's words are
// on their way: made before it, they cost 512 x 512 pixels 10 to 20 of its 436 us.
struct CgpPair {
  float h, l;
};
__device__ __forceinline__ CgpPair cgp_add(CgpPair a, CgpPair b) {
  const float s = a.h + b.h, t = s - a.h;
  return {s, ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l)};
}
__device__ __forceinline__ double cgp_add(double a, double b) { return a + b; }
__device__ __forceinline__ CgpPair cgp_shfl(CgpPair a, int o) {
  return {__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ double cgp_shfl(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ void cgp_from(float x, CgpPair& r) { r = {x, 0.0f}; }
__device__ __forceinline__ void cgp_from(double x, double& r) { r = x; }
__device__ __forceinline__ void cgp_from(float x, double& r) { r = (double)x; }
__device__ __forceinline__ CgpPair cgp_norm(CgpPair a) {
  const float s = a.h + a.l;
  return {s, a.l - (s - a.h)};
}
__device__ __forceinline__ double cgp_norm(double a) { return a; }
// the two words of a value in flight
__device__ __forceinline__ unsigned cgp_half(CgpPair a, int i) { return __float_as_uint(i ? a.l : a.h); }
__device__ __forceinline__ unsigned cgp_half(double a, int i) {
  const u64 b = (u64)__double_as_longlong(a);
  return i ? (unsigned)(b >> 32) : (unsigned)b;
}
__device__ __forceinline__ void cgp_join(unsigned w0, unsigned w1, CgpPair& r) {
  r = {__uint_as_float(w0), __uint_as_float(w1)};
}
__device__ __forceinline__ void cgp_join(unsigned w0, unsigned w1, double& r) {
  r = __longlong_as_double((long long)(((u64)w1 << 32) | w0));
}
__device__ __forceinline__ CgpPair cgp_mul(CgpPair a, CgpPair b) {
  const float p = a.h * b.h;
  return cgp_norm({p, fmaf(a.h, b.h, -p) + fmaf(a.h, b.l, a.l * b.h)});
}
__device__ __forceinline__ double cgp_mul(double a, double b) { return a * b; }
__device__ __forceinline__ CgpPair cgp_neg(CgpPair a) { return {-a.h, -a.l}; }
__device__ __forceinline__ double cgp_neg(double a) { return -a; }
__device__ __forceinline__ bool cgp_finite(CgpPair a) { return isfinite(a.h) && isfinite(a.l); }
__device__ __forceinline__ bool cgp_finite(double a) { return ((__double_as_longlong(a) >> 52) & 0x7ff) != 0x7ff; }
__device__ __forceinline__ bool cgp_zero(CgpPair a) { return a.h == 0.0f; }
__device__ __forceinline__ bool cgp_zero(double a) { return (__double_as_longlong(a) << 1) == 0; }
__device__ __forceinline__ bool cgp_negative(CgpPair a) { return a.h < 0.0f; }
__device__ __forceinline__ bool cgp_negative(double a) { return __double_as_longlong(a) < 0; }
__device__ __forceinline__ double cgp_double(CgpPair a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ double cgp_double(double a) { return a; }
__device__ __forceinline__ void cgp_set(double x, CgpPair& r) {
  r.h = (float)x;
  r.l = (float)(x - (double)r.h);
}
__device__ __forceinline__ void cgp_set(double x, double& r) { r = x; }
__device__ __forceinline__ float cgp_value(CgpPair a) { return a.h; }
__device__ __forceinline__ double cgp_value(double a) { return a; }

__device__ __forceinline__ CgpPair cgp_times(CgpPair a, float f) { return {a.h * f, a.l * f}; }
__device__ __forceinline__ double cgp_times(double a, double f) { return a * f; }
// exponent of a normal number (below every one of them for 0 and subnormal numbers)
__device__ __forceinline__ int cgp_exponent(float a) { return (int)((__float_as_uint(a) >> 23) & 0xff) - 127; }
__device__ __forceinline__ int cgp_exponent(double a) { return (int)((__double_as_longlong(a) >> 52) & 0x7ff) - 1023; }
__device__ __forceinline__ void cgp_pow2(int k, float& r) { r = __uint_as_float((unsigned)(127 + k) << 23); }
__device__ __forceinline__ void cgp_pow2(int k, double& r) { r = __longlong_as_double((long long)(1023 + k) << 52); }
// Quotient by a reciprocal of the divisor's high part and one residual correction (a Newton
// step); a divisor near the ends of the range, where the reciprocal or the residual would
// leave it, is brought near 1 by a power of two first.
__device__ __forceinline__ CgpPair cgp_div(CgpPair a, CgpPair b) {
  float f = 1.0f;
  const int e = cgp_exponent(b.h);
  if (e < -100 || e > 100) {
    cgp_pow2(max(-126, min(126, -e)), f);
    b = cgp_times(b, f);
  }
  const float r = __frcp_rn(b.h), q = a.h * r;
  const float rem = fmaf(-q, b.h, a.h) + fmaf(-q, b.l, a.l);
  return cgp_times(cgp_norm({q, rem * r}), f);
}
__device__ __forceinline__ double cgp_div(double a, double b) { return a / b; }

template <typename T> struct CgpNum;
template <> struct CgpNum<float> { typedef CgpPair type; };
template <> struct CgpNum<double> { typedef double type; };

// Exponents: s^T r (scaled) stays within 2^+-BAND, the scale within 2^+-LIM.
template <typename T> struct CgpRange;
template <> struct CgpRange<float> { static constexpr int BAND = 20, LIM = 120; };
template <> struct CgpRange<double> { static constexpr int BAND = 200, LIM = 900; };

// What a CTA's threads share: the sums in flight (N) and the scalars of the run, which one
// warp each computes (64 cycles of a scheduler per FP64 instruction and warp) for the others.
template <typename T>
struct CgpShared {
  typedef typename CgpNum<T>::type N;
  T red[4][CGP_T / 32];                    // the warps' sums, unscaled
  union {                                  // the CTAs' partial sums, [CTA][value]
    double d[CGP_MAXC * 4];
    N n[CGP_MAXC * 4];
  } part;
  double tot[4];                           // start: the four sums
  N sr, ss, rr, alpha, beta, cb;           // scaled by `scale`, except the quotients
  double ref2, thr;                        // thr: scaled tol^2 ref^2
  T scale, factor;                         // of the sums (a power of two); its next change
  int fin[4], conv, status;
};
template <typename T> __device__ __forceinline__ double* cgp_part(CgpShared<T>& sh, double*) { return sh.part.d; }
__device__ __forceinline__ CgpPair* cgp_part(CgpShared<float>& sh, CgpPair*) { return sh.part.n; }

// Sums of v (times sh.scale) over all threads of all CTAs, and a barrier of the grid.  Warp
// w < NV gets the total of value w and calls tail(w, total) with all its lanes; what tail
// writes to shared memory is visible to every thread on return.  `during` runs while the
// words of the other CTAs are on their way.  R: representation of the sums.  Returns false
// (in every thread) when a wait gave up.
template <int NV, int NT, typename R, typename T, class During, class Tail>
__device__ __forceinline__ bool cgp_allreduce(const T (&v)[4], CgpShared<T>& sh, u64* slots, unsigned epoch,
                                              CgState* st, During during, Tail tail) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nc = gridDim.x;
  u64* base = slots + (size_t)(epoch & 1) * CGP_MAXC * CGP_SLOT;
  R* part = cgp_part(sh, (R*)nullptr);
  if (NV == 4) {
    const T w = warp_sum4<T>(v, lane);
    if ((lane & 7) == 0) sh.red[lane >> 3][wid] = w;
  } else {
    const T w = warp_sum(v[0]);
    if (lane == 0) sh.red[0][wid] = w;
  }
  __syncthreads();
  if (wid < NV) {
    R t;
    cgp_from(sh.red[wid][lane & (NT / 32 - 1)] * sh.scale, t);
#pragma unroll
    for (int o = NT / 64; o > 0; o >>= 1) t = cgp_add(t, cgp_shfl(t, o));
    t = cgp_norm(t);
    if (lane < 2) cgp_put(base + blockIdx.x * CGP_SLOT + 2 * wid + lane, cgp_word(epoch, cgp_half(t, lane)));
  }
  during();
  // read every CTA's words: first all of this thread's loads, then wait for what is missing
  constexpr int K = (CGP_MAXC * NV + NT - 1) / NT;
  u64 lo[K], hi[K];
  bool ok = true;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int w = threadIdx.x + k * NT;
    if (w < nc * NV) cgp_get2(base + (w / NV) * CGP_SLOT + 2 * (w % NV), lo[k], hi[k]);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int w = threadIdx.x + k * NT;
    if (w < nc * NV && ok) {
      const u64* p = base + (w / NV) * CGP_SLOT + 2 * (w % NV);
      if ((unsigned)(lo[k] >> 32) != epoch || (unsigned)(hi[k] >> 32) != epoch) ok = cgp_wait2(p, lo[k], hi[k], epoch, st);
      cgp_join((unsigned)lo[k], (unsigned)hi[k], part[w]);
    }
  }
  if (__syncthreads_or(!ok)) return false;
  if (wid < NV) {
    R x[CGP_MAXC / 32];
#pragma unroll
    for (int k = 0; k < CGP_MAXC / 32; ++k) {
      const int c = lane + 32 * k;
      cgp_from(T(0), x[k]);
      if (c < nc) x[k] = part[c * NV + wid];
    }
#pragma unroll
    for (int h = 1; h < CGP_MAXC / 32; h <<= 1)
#pragma unroll
      for (int k = 0; k + h < CGP_MAXC / 32; k += 2 * h)
        if (32 * (k + h) < nc) x[k] = cgp_add(x[k], x[k + h]);
    R t = x[0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t = cgp_add(t, cgp_shfl(t, o));
    tail(wid, cgp_norm(t));
  }
  __syncthreads();
  return true;
}

// ---- the scalar steps (tails of the all-reduces; every CTA takes the same ones)
// Start: s^T r, s^T s, r^T r, x0^T x0 in sh.tot; by every thread, after the all-reduce.
template <typename T>
__device__ void cgp_start(CgpShared<T>& sh, double shift, double tol2) {
  if (threadIdx.x == 0) {
    const double sr = sh.tot[0], ss = sh.tot[1], rr = sh.tot[2];
    sh.status = (cgp_finite(sr) && cgp_finite(ss) && cgp_finite(rr)) ? CG_RUN : CG_NONFINITE;
    const double b2 = shift * shift * sh.tot[3];
    sh.ref2 = b2 > 0.0 ? b2 : rr;
    // 2^-exponent of the largest sum, within the scale's range
    const int k = max(-CgpRange<T>::LIM, min(CgpRange<T>::LIM, -cgp_exponent(fmax(fmax(fabs(sr), ss), rr))));
    cgp_pow2(k, sh.scale);
    const double sc = (double)sh.scale;
    cgp_set(sr * sc, sh.sr);
    cgp_set(ss * sc, sh.ss);
    cgp_set(rr * sc, sh.rr);
    sh.thr = tol2 > 0.0 ? tol2 * sh.ref2 * sc : -1.0;
    cgp_set(0.0, sh.alpha);
    cgp_set(0.0, sh.beta);
  }
  __syncthreads();
}
// Direction (warp 0): p^T q -> the breakdown tests and alpha (not finite: the run stops
// before x is touched).
template <typename T>
__device__ __forceinline__ void cgp_direction(CgpShared<T>& sh, typename CgpNum<T>::type pq, int lane) {
  int status = CG_RUN;
  const typename CgpNum<T>::type sr = sh.sr;
  if (cgp_zero(sr)) status = CG_CONV;
  else if (!cgp_finite(pq)) status = CG_NONFINITE;
  else if (cgp_zero(pq) || cgp_negative(pq)) status = CG_BREAK;
  const typename CgpNum<T>::type alpha = cgp_div(sr, pq);
  if (status == CG_RUN && !cgp_finite(alpha)) status = CG_NONFINITE;
  if (lane == 0) {
    sh.status = status;
    if (status == CG_RUN) sh.alpha = alpha;
  }
}
// By the last thread, while the update's words are on their way: beta's factor -alpha / (s^T r or
// s^T s), and the factor of the scale's change (1 until s^T r has left its band).
template <typename T>
__device__ __forceinline__ void cgp_prepare_beta(CgpShared<T>& sh, int beta_mode) {
  if (threadIdx.x != blockDim.x - 1) return;
  constexpr int BAND = CgpRange<T>::BAND, LIM = CgpRange<T>::LIM;
  const int e = cgp_exponent(cgp_value(sh.sr));
  T f = T(1);
  if (e < -BAND || e > BAND) {
    const int cur = cgp_exponent(sh.scale);
    cgp_pow2(max(-LIM, min(LIM, max(-LIM, min(LIM, cur - e)) - cur)), f);
  }
  sh.factor = f;
  sh.cb = cgp_neg(cgp_div(sh.alpha, beta_mode == BF_BETA_PRINTED ? sh.ss : sh.sr));
}
// Update (warps 0 .. 3): s^T r, s^T q, s^T s, r^T r -> beta and the stopping tests, the sums in
// the new scale.
template <typename T>
__device__ __forceinline__ void cgp_update_tail(CgpShared<T>& sh, int w, typename CgpNum<T>::type t, int lane) {
  typename CgpNum<T>::type b = t;
  if (w == 1) b = cgp_mul(sh.cb, t);
  if (lane != 0) return;
  const T f = sh.factor;
  sh.fin[w] = cgp_finite(t);
  if (w == 0) sh.sr = cgp_times(t, f);
  else if (w == 1) sh.beta = b;
  else if (w == 2) sh.ss = cgp_times(t, f);
  else {
    sh.rr = cgp_times(t, f);
    sh.conv = sh.thr >= 0.0 && cgp_double(t) <= sh.thr;
    sh.thr *= (double)f;
    sh.scale *= f;
  }
}
// After the update's all-reduce, by every thread: the status.
template <typename T>
__device__ __forceinline__ int cgp_status(const CgpShared<T>& sh) {
  if (!(sh.fin[0] & sh.fin[1] & sh.fin[2] & sh.fin[3])) return CG_NONFINITE;
  return sh.conv ? CG_CONV : CG_RUN;
}
template <typename T>
__device__ void cgp_history(const CgpShared<T>& sh, double* hist, int it) {
  if (hist && blockIdx.x == 0 && threadIdx.x == blockDim.x - 1) {   // beta: before this update
    hist[2 * it] = cgp_double(sh.alpha);
    hist[2 * it + 1] = it == 0 ? 0.0 : cgp_double(sh.beta);
  }
}
template <typename T>
__device__ void cgp_write_state(const CgpShared<T>& sh, CgState* st, int iters, int status) {
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  const double inv = 1.0 / (double)sh.scale;
  st->sr = cgp_double(sh.sr) * inv;
  st->ss = cgp_double(sh.ss) * inv;
  st->rr = cgp_double(sh.rr) * inv;
  st->ref2 = sh.ref2;
  st->alpha = cgp_double(sh.alpha);
  st->beta = cgp_double(sh.beta);
  st->iter = iters;
  atomicCAS(&st->status, CG_RUN, status);      // a timeout recorded by another CTA stays
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
  __device__ void prepare(const float*, float*, int, int, int, int, int, int) const {}
  // (L p) of the run at (x, y) of the rectangle
  __device__ void sums(const float* P, const float* G, int W, int H, int x, int y, int, int, int, int,
                       float (&vi)[RUN_P], float (&acc)[RUN_P]) const {
    const int xs = W + 2 * LP;
    float ws[RUN_P];
    const int o = y * xs + x;
    run_sums<true, false>(c, P + o, G + o, xs, vi, acc, ws);
  }
};

// The guided filter's operator (Section 3, Eq. 6) of radius R in the difference form of
// bf_guided.cu, by runs of four: stage A gives d_k and a_k of the windows centred on the
// rectangle and R pixels around it, stage B sums the windows that contain a pixel.  Bound by
// shared memory (about 90 wavefronts per 32 pixels) and the FP32 pipe (225 of its cycles per
// scheduler at R = 2).  Rectangles whose halo leaves the image test every member.  50
// iterations of 512 x 512, R = 2: 584 us (five launches per iteration: 2242).
template <int R>
struct CgpGuided {
  static constexpr int HALO = 2 * R, LP = 8;
  const float* guide;
  const float* mu;
  const float* ivar;
  static __host__ __device__ size_t tile(int W, int H) { return (size_t)(W + 2 * LP) * (H + 2 * HALO); }
  static __host__ __device__ size_t extra(int W, int H) { return 5 * tile(W, H); }
  static __device__ float inv_count(int gx, int gy, int nx, int ny) {
    const int cy = min(gy + R, ny - 1) - max(gy - R, 0) + 1, cx = min(gx + R, nx - 1) - max(gx - R, 0) + 1;
    return 1.0f / (float)(cx * cy);
  }
  static __device__ bool border(int W, int H, int bx, int by, int nx, int ny) {
    return bx - HALO < 0 || by - HALO < 0 || bx + W + HALO > nx || by + H + HALO > ny;
  }
  // tiles: guide, mean, 1 / (variance + eps) / N, d_k, a_k
  __device__ void stage(float* EX, int W, int H, int bx, int by, int nx, int ny) const {
    const int xs = W + 2 * LP, nt = (int)tile(W, H);
    for (int q = threadIdx.x; q < nt; q += CGP_T) {
      const int hy = q / xs, hx = q - hy * xs;
      const int gy = by - HALO + hy, gx = bx - LP + hx;
      const bool in = (unsigned)gx < (unsigned)nx && (unsigned)gy < (unsigned)ny;
      const int64_t gp = (int64_t)gy * nx + gx;
      EX[q] = in ? guide[gp] : 0.0f;
      EX[nt + q] = in ? mu[gp] : 0.0f;
      EX[2 * nt + q] = in ? ivar[gp] * inv_count(gx, gy, nx, ny) : 0.0f;
      EX[3 * nt + q] = EX[4 * nt + q] = 0.0f;
    }
  }
  // entry e of 12 values held as pairs
  static __device__ __forceinline__ float at(const run_f2 (&p)[6], int e) { return (e & 1) ? run_hi(p[e / 2]) : run_lo(p[e / 2]); }
  template <bool CHECK>
  __device__ __forceinline__ void stage_a(const float* P, const float* G, const float* MU, int xs, int o, int gx0, int gy,
                                          int nx, int ny, float (&ds)[RUN_P], float (&cs)[RUN_P]) const {
    run_f2 ds2[RUN_P], cs2[RUN_P], xk2[RUN_P], mk2[RUN_P];
#pragma unroll
    for (int j = 0; j < RUN_P; ++j) {
      const float xk = P[o + j], mk = MU[o + j];
      xk2[j] = f2_pack(xk, xk);
      mk2[j] = f2_pack(mk, mk);
      ds2[j] = cs2[j] = 0ull;
      ds[j] = cs[j] = 0.0f;
    }
#pragma unroll
    for (int dy = -R; dy <= R; ++dy) {
      if (CHECK && (unsigned)(gy + dy) >= (unsigned)ny) continue;
      run_f2 xr[6], gr[6];
      run_ld(P + o + dy * xs - 4, xr);
      run_ld(G + o + dy * xs - 4, gr);
#pragma unroll
      for (int j = 0; j < RUN_P; ++j) {
#pragma unroll
        for (int a = 0; a < 6; ++a) {
          const int lo = j + 4 - R, hi = j + 4 + R;
          const bool i0 = 2 * a >= lo && 2 * a <= hi, i1 = 2 * a + 1 >= lo && 2 * a + 1 <= hi;
          if (i0 && i1 && !CHECK) {
            const run_f2 xd = run_sub(xr[a], xk2[j]);
            ds2[j] = run_add(ds2[j], xd);
            cs2[j] = run_fma(run_sub(gr[a], mk2[j]), xd, cs2[j]);
          } else {
#pragma unroll
            for (int b = 0; b < 2; ++b) {
              const int e = 2 * a + b;
              if (!(b ? i1 : i0) || (CHECK && (unsigned)(gx0 + e - 4) >= (unsigned)nx)) continue;
              const float xd = at(xr, e) - run_lo(xk2[j]);
              ds[j] += xd;
              cs[j] = fmaf(at(gr, e) - run_lo(mk2[j]), xd, cs[j]);
            }
          }
        }
      }
    }
#pragma unroll
    for (int j = 0; j < RUN_P; ++j) {
      ds[j] += run_lo(ds2[j]) + run_hi(ds2[j]);
      cs[j] += run_lo(cs2[j]) + run_hi(cs2[j]);
    }
  }
  __device__ void prepare(const float* P, float* EX, int W, int H, int bx, int by, int nx, int ny) const {
    const int xs = W + 2 * LP, nt = (int)tile(W, H), per = W / 4 + 2;
    const float *G = EX, *MU = EX + nt, *IV = EX + 2 * nt;
    float *DK = EX + 3 * nt, *AK = EX + 4 * nt;
    const bool chk = border(W, H, bx, by, nx, ny);
    for (int r = threadIdx.x; r < per * (H + 2 * R); r += CGP_T) {
      const int ry = r / per, x = 4 * (r - ry * per) - 4, y = ry - R;     // windows (x .. x + 3, y)
      const int o = (y + HALO) * xs + x + LP;
      float ds[RUN_P], cs[RUN_P];
      if (chk) stage_a<true>(P, G, MU, xs, o, bx + x, by + y, nx, ny, ds, cs);
      else stage_a<false>(P, G, MU, xs, o, bx + x, by + y, nx, ny, ds, cs);
#pragma unroll
      for (int j = 0; j < RUN_P; ++j) {
        const int gx = bx + x + j, gy = by + y;
        const bool in = !chk || ((unsigned)gx < (unsigned)nx && (unsigned)gy < (unsigned)ny);
        const float inv = chk ? (in ? inv_count(gx, gy, nx, ny) : 0.0f) : 1.0f / (float)((2 * R + 1) * (2 * R + 1));
        DK[o + j] = in ? ds[j] * inv : 0.0f;
        AK[o + j] = in ? cs[j] * IV[o + j] : 0.0f;
      }
    }
    __syncthreads();
  }
  template <bool CHECK>
  __device__ __forceinline__ void stage_b(const float* P, const float* EX, int nt, int xs, int o, int gx0, int gy, int nx,
                                          int ny, float (&vi)[RUN_P], float (&acc)[RUN_P]) const {
    const float *G = EX, *MU = EX + nt, *DK = EX + 3 * nt, *AK = EX + 4 * nt;
    run_f2 xi2[RUN_P], gi2[RUN_P], l2[RUN_P];
#pragma unroll
    for (int j = 0; j < RUN_P; ++j) {
      vi[j] = P[o + j];
      const float gi = G[o + j];
      xi2[j] = f2_pack(vi[j], vi[j]);
      gi2[j] = f2_pack(gi, gi);
      l2[j] = 0ull;
      acc[j] = 0.0f;
    }
#pragma unroll
    for (int dy = -R; dy <= R; ++dy) {
      if (CHECK && (unsigned)(gy + dy) >= (unsigned)ny) continue;
      run_f2 xr[6], mr[6], dr[6], ar[6];
      const int ro = o + dy * xs - 4;
      run_ld(P + ro, xr);
      run_ld(MU + ro, mr);
      run_ld(DK + ro, dr);
      run_ld(AK + ro, ar);
#pragma unroll
      for (int j = 0; j < RUN_P; ++j) {
#pragma unroll
        for (int a = 0; a < 6; ++a) {
          const int lo = j + 4 - R, hi = j + 4 + R;
          const bool i0 = 2 * a >= lo && 2 * a <= hi, i1 = 2 * a + 1 >= lo && 2 * a + 1 <= hi;
          if (i0 && i1 && !CHECK) {
            const run_f2 t = run_sub(run_sub(xi2[j], xr[a]), dr[a]);
            l2[j] = run_add(l2[j], run_fma(run_sub(mr[a], gi2[j]), ar[a], t));
          } else {
#pragma unroll
            for (int b = 0; b < 2; ++b) {
              const int e = 2 * a + b;
              if (!(b ? i1 : i0) || (CHECK && (unsigned)(gx0 + e - 4) >= (unsigned)nx)) continue;
              const float t = (vi[j] - at(xr, e)) - at(dr, e);
              acc[j] += fmaf(at(mr, e) - run_lo(gi2[j]), at(ar, e), t);
            }
          }
        }
      }
    }
#pragma unroll
    for (int j = 0; j < RUN_P; ++j) acc[j] += run_lo(l2[j]) + run_hi(l2[j]);
  }
  __device__ void sums(const float* P, const float* EX, int W, int H, int x, int y, int bx, int by, int nx, int ny,
                       float (&vi)[RUN_P], float (&acc)[RUN_P]) const {
    const int xs = W + 2 * LP, nt = (int)tile(W, H), o = (y + HALO) * xs + x + LP;
    if (border(W, H, bx, by, nx, ny)) stage_b<true>(P, EX, nt, xs, o, bx + x, by + y, nx, ny, vi, acc);
    else stage_b<false>(P, EX, nt, xs, o, bx + x, by + y, nx, ny, vi, acc);
  }
};

struct CgpImage {
  CgArgs<float> cg;
  CgpRect rc;
  int nx, ny, kmax, vec;
  u64* slots;                // [2][CGP_MAXC][CGP_SLOT], by epoch parity
  u64* frames;               // [n]: s of the rectangles' frames
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

// x of the rectangle to the image, at the end and when a wait gives up (as far as the run has
// come).  Not inlined: with the store in place and breaks out of the loop to it, 512 x 512 pixels
// take 30 us more (the window sums are the same code; where it lies is not).
__device__ __noinline__ void cgp_store_x(const CgpImage& a, const float* X) {
  const int W = a.rc.W, H = a.rc.H;
  const int bx = (blockIdx.x % a.rc.ncx) * W, by = (blockIdx.x / a.rc.ncx) * H;
  const bool vec = a.vec && ((uintptr_t)a.cg.x & 15) == 0;
  __syncthreads();
  for (int q = threadIdx.x; q < W * H / 4; q += CGP_T) {
    const int y = 4 * q / W, x = 4 * q - y * W;
    const int cnt = run_count(bx + x, by + y, a.nx, a.ny);
    const float4 x4 = *reinterpret_cast<const float4*>(X + 4 * q);
    const float xv[4] = {x4.x, x4.y, x4.z, x4.w};
    if (cnt) run_store(a.cg.x, (int64_t)(by + y) * a.nx + bx + x, cnt, vec, xv);
  }
}

template <class OP>
__global__ void __launch_bounds__(CGP_T, 1) k_cgp_image(const __grid_constant__ OP op, const __grid_constant__ CgpImage a) {
  constexpr int HALO = OP::HALO, LP = OP::LP;
  extern __shared__ __align__(16) float cgp_smem[];
  typedef CgpPair N;
  __shared__ CgpShared<float> sh;
  if ((int)blockIdx.x == a.cg.absent) return;
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
  if (threadIdx.x == 0) sh.scale = 1.0f;
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
  // a run's values of s that the neighbours read
  auto frame = [&](int x, int y, int cnt, const float (&s)[RUN_P], unsigned tag) {
    const bool rows = y < HALO || y >= H - HALO;
    u64* f = a.frames + (int64_t)(by + y) * nx + bx + x;
#pragma unroll
    for (int j = 0; j < RUN_P; ++j)
      if (j < cnt && (rows || x + j < HALO || x + j >= W - HALO)) cgp_put(f + j, cgp_word(tag, __float_as_uint(s[j])));
  };
  // this thread's halo pixels: tile offset, and index in the image (-1: none or outside)
  const int nhalo = 2 * HALO * (W + 2 * HALO) + 2 * HALO * H;
  int htile[CGP_HALO_REGS], himg[CGP_HALO_REGS];
  u64 hw[CGP_HALO_REGS];
#pragma unroll
  for (int k = 0; k < CGP_HALO_REGS; ++k) {
    const int h = threadIdx.x + k * CGP_T;
    himg[k] = htile[k] = -1;
    hw[k] = 0ull;
    if (h < nhalo) {
      int tx, ty;
      cgp_halo_pos<HALO>(h, W, H, tx, ty);
      const int gx = bx + tx, gy = by + ty;
      htile[k] = (ty + HALO) * xs + tx + LP;
      if ((unsigned)gx < (unsigned)nx && (unsigned)gy < (unsigned)ny) himg[k] = gy * nx + gx;
    }
  }
  // the halo words: loads issued ...
  auto halo_get = [&]() {
#pragma unroll
    for (int k = 0; k < CGP_HALO_REGS; ++k)
      if (himg[k] >= 0) hw[k] = cgp_get(a.frames + himg[k]);
  };
  // ... and awaited
  auto halo_wait = [&](unsigned tag) {
    bool ok = true;
#pragma unroll
    for (int k = 0; k < CGP_HALO_REGS; ++k)
      if (himg[k] >= 0 && (unsigned)(hw[k] >> 32) != tag && ok) ok = cgp_wait(a.frames + himg[k], hw[k], tag, a.cg.st);
    return ok;
  };
  // ---- r = -L x0, s = T r
  unsigned epoch = 1;
  {
    float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    op.prepare(P, EX, W, H, bx, by, nx, ny);
    for (int u = wid; u < nunits; u += CGP_T / 32) {
      const int x = (u % ux_n) * 32 + rx, y = (u / ux_n) * 4 + ry;
      const int cnt = run_count(bx + x, by + y, nx, ny);
      float xi[RUN_P], acc[RUN_P], s[RUN_P];
      op.sums(P, EX, W, H, x, y, bx, by, nx, ny, xi, acc);
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
      if (cnt) frame(x, y, cnt, s, 1u);
    }
    if (!cgp_allreduce<4, CGP_T, double>(v, sh, a.slots, epoch, a.cg.st, halo_get, [&](int w, double t) {
          if (lane == 0) sh.tot[w] = t;
        }))
      return cgp_store_x(a, X);
    cgp_start(sh, (double)a.cg.shift, tol2);
  }
  int it = 0, status = sh.status;
  for (; it < a.kmax && status == CG_RUN; ++it) {
    const float beta = cgp_value(sh.beta);     // 0 before the first step
    // ---- p = s + beta p
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
    const bool ok = halo_wait((unsigned)it + 1u);
#pragma unroll
    for (int k = 0; k < CGP_HALO_REGS; ++k)
      if (htile[k] >= 0) {
        const float s = himg[k] >= 0 ? __uint_as_float((unsigned)hw[k]) : 0.0f;
        P[htile[k]] = it ? fmaf(beta, P[htile[k]], s) : s;
      }
    if (__syncthreads_or(!ok)) return cgp_store_x(a, X);
    // ---- q = (L + sigma I) p, p^T q
    float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    op.prepare(P, EX, W, H, bx, by, nx, ny);
    for (int u = wid; u < nunits; u += CGP_T / 32) {
      const int x = (u % ux_n) * 32 + rx, y = (u / ux_n) * 4 + ry;
      const int cnt = run_count(bx + x, by + y, nx, ny);
      float pi[RUN_P], acc[RUN_P], q[RUN_P];
      op.sums(P, EX, W, H, x, y, bx, by, nx, ny, pi, acc);
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
    if (!cgp_allreduce<1, CGP_T, N>(v, sh, a.slots, ++epoch, a.cg.st, [] {},
                                    [&](int, N t) { cgp_direction(sh, t, lane); }))
      return cgp_store_x(a, X);
    status = sh.status;
    if (status != CG_RUN) break;
    // ---- x += alpha p, s -= alpha T q, the sums
    const float alpha = cgp_value(sh.alpha);
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
      if (cnt) frame(x, y, cnt, s, (unsigned)it + 2u);
    }
    auto during = [&] {
      halo_get();
      cgp_prepare_beta(sh, beta_mode);
      cgp_history(sh, a.cg.hist, it);
    };
    if (!cgp_allreduce<4, CGP_T, N>(v, sh, a.slots, ++epoch, a.cg.st, during,
                                    [&](int w, N t) { cgp_update_tail(sh, w, t, lane); }))
      return cgp_store_x(a, X);
    status = cgp_status(sh);
  }
  cgp_store_x(a, X);
  cgp_write_state(sh, a.cg.st, it, status);
}

// ---------------------------------------------------------------- signals
// Any interval window of radius R on a signal: the CTA keeps the weights of its forward
// pairs (i, i + t), t = 1 .. R, i from R samples before its piece to its end, so that an
// iteration has no exponentials (in FP64 they were 9/10 of the arithmetic at 2 FMA per clock
// and SM).  Generic recurrences: r and s = T r are both kept.  4096 samples, FP64, 11 taps, 20
// iterations: 160 us (two launches per iteration on 16 CTAs: 725).
template <typename T>
struct CgpLine {
  CgArgs<T> cg;
  T a_r;
  T ls[BF_MAX_R1D + 1];
  int n, R, W, kmax;
  u64* slots;
  u64* frames;                                 // [n] words (FP64: [n][2]): s at the pieces' ends
};

__host__ __device__ inline size_t cgp_line_elems(int W, int R) {
  return (size_t)(W + 2 * R) + 5 * (size_t)W + (size_t)R * (W + R);
}

// x of the piece to the signal.
template <typename T>
__device__ __noinline__ void cgp_store_x(const CgpLine<T>& a, const T* X) {
  const int b = blockIdx.x * a.W, len = min(a.W, a.n - b);
  __syncthreads();
  for (int q = threadIdx.x; q < len; q += CGP_TL) a.cg.x[b + q] = X[q];
}

template <typename T>
__global__ void __launch_bounds__(CGP_TL, 1) k_cgp_line(const __grid_constant__ CgpLine<T> a) {
  extern __shared__ __align__(16) float cgp_smem[];
  typedef typename CgpNum<T>::type N;
  __shared__ CgpShared<T> sh;
  if ((int)blockIdx.x == a.cg.absent) return;
  const int lane = threadIdx.x & 31;
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
  if (threadIdx.x == 0) sh.scale = T(1);
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
    T acc[4] = {T(0), T(0), T(0), T(0)};       // four chains: an FP64 FMA is long
    for (int t = 1; t <= R; ++t) {
      const T* wt = WF + (t - 1) * (W + R) + q + R;
      const T f = pi - P[q + R + t], g = pi - P[q + R - t];
      if (t & 1) {
        acc[0] = fma(wt[0], f, acc[0]);
        acc[1] = fma(wt[-t], g, acc[1]);
      } else {
        acc[2] = fma(wt[0], f, acc[2]);
        acc[3] = fma(wt[-t], g, acc[3]);
      }
    }
    return (acc[0] + acc[1]) + (acc[2] + acc[3]);
  };
  // s at the ends of the piece, for the neighbours, and the halo
  auto frame = [&](int q, T s, unsigned tag) {
    if (q >= R && q < len - R) return;
    if (sizeof(T) == 4) {
      cgp_put(a.frames + b + q, cgp_word(tag, __float_as_uint((float)s)));
    } else {
      const u64 bits = (u64)__double_as_longlong((double)s);
      cgp_put(a.frames + 2 * (int64_t)(b + q), cgp_word(tag, (unsigned)bits));
      cgp_put(a.frames + 2 * (int64_t)(b + q) + 1, cgp_word(tag, (unsigned)(bits >> 32)));
    }
  };
  static_assert(2 * BF_MAX_R1D <= CGP_TL, "one halo sample per thread");
  const int hi_ = threadIdx.x < R ? b - R + threadIdx.x : b + W + threadIdx.x - R;
  const bool halo = threadIdx.x < 2 * R, hin = halo && (unsigned)hi_ < (unsigned)n;
  T* hp = P + (threadIdx.x < R ? threadIdx.x : W + threadIdx.x);
  u64 hw[2] = {0ull, 0ull};
  auto halo_get = [&]() {
    if (hin) {
      if (sizeof(T) == 4) hw[0] = cgp_get(a.frames + hi_);
      else cgp_get2(a.frames + 2 * (int64_t)hi_, hw[0], hw[1]);
    }
  };
  auto halo_wait = [&](unsigned tag) {
    bool ok = true;
    if (hin) {
      if ((unsigned)(hw[0] >> 32) != tag) ok = cgp_wait(a.frames + (sizeof(T) / 4) * (int64_t)hi_, hw[0], tag, a.cg.st);
      if (ok && sizeof(T) == 8 && (unsigned)(hw[1] >> 32) != tag)
        ok = cgp_wait(a.frames + 2 * (int64_t)hi_ + 1, hw[1], tag, a.cg.st);
    }
    return ok;
  };
  unsigned epoch = 1;
  {
    T v[4] = {T(0), T(0), T(0), T(0)};
    for (int q = threadIdx.x; q < len; q += CGP_TL) {
      const T xi = P[q + R], r = -lap(q), s = a.cg.dinv ? r * DI[q] : r;
      X[q] = xi;
      RR[q] = r;
      S[q] = s;
      frame(q, s, 1u);
      v[0] = fma(s, r, v[0]);
      v[1] = fma(s, s, v[1]);
      v[2] = fma(r, r, v[2]);
      v[3] = fma(xi, xi, v[3]);
    }
    if (!cgp_allreduce<4, CGP_TL, double>(v, sh, a.slots, epoch, a.cg.st, halo_get, [&](int w, double t) {
          if (lane == 0) sh.tot[w] = t;
        }))
      return cgp_store_x(a, X);
    cgp_start(sh, (double)a.cg.shift, tol2);
  }
  int it = 0, status = sh.status;
  for (; it < a.kmax && status == CG_RUN; ++it) {
    const T beta = (T)cgp_value(sh.beta);      // 0 before the first step
    for (int q = threadIdx.x; q < W; q += CGP_TL) {
      const T s = q < len ? S[q] : T(0);
      P[q + R] = it ? fma(beta, P[q + R], s) : s;
    }
    const bool ok = halo_wait((unsigned)it + 1u);
    if (halo) {
      const T s = !hin ? T(0)
                       : (sizeof(T) == 4 ? (T)__uint_as_float((unsigned)hw[0])
                                         : (T)__longlong_as_double((long long)((hw[1] << 32) | (hw[0] & 0xffffffffull))));
      *hp = it ? fma(beta, *hp, s) : s;
    }
    if (__syncthreads_or(!ok)) return cgp_store_x(a, X);
    T v[4] = {T(0), T(0), T(0), T(0)};
    for (int q = threadIdx.x; q < len; q += CGP_TL) {
      const T p = P[q + R], qq = fma(a.cg.shift, p, lap(q));
      Q[q] = qq;
      v[0] = fma(p, qq, v[0]);
    }
    if (!cgp_allreduce<1, CGP_TL, N>(v, sh, a.slots, ++epoch, a.cg.st, [] {},
                                    [&](int, N t) { cgp_direction(sh, t, lane); }))
      return cgp_store_x(a, X);
    status = sh.status;
    if (status != CG_RUN) break;
    const T alpha = (T)cgp_value(sh.alpha);
    v[0] = T(0);
    for (int q = threadIdx.x; q < len; q += CGP_TL) {
      const T qq = Q[q];
      X[q] = fma(alpha, P[q + R], X[q]);
      const T r = fma(-alpha, qq, RR[q]), s = a.cg.dinv ? r * DI[q] : r;
      RR[q] = r;
      S[q] = s;
      frame(q, s, (unsigned)it + 2u);
      v[0] = fma(s, r, v[0]);
      v[1] = fma(s, qq, v[1]);
      v[2] = fma(s, s, v[2]);
      v[3] = fma(r, r, v[3]);
    }
    auto during = [&] {
      halo_get();
      cgp_prepare_beta(sh, beta_mode);
      cgp_history(sh, a.cg.hist, it);
    };
    if (!cgp_allreduce<4, CGP_TL, N>(v, sh, a.slots, ++epoch, a.cg.st, during,
                                    [&](int w, N t) { cgp_update_tail(sh, w, t, lane); }))
      return cgp_store_x(a, X);
    status = cgp_status(sh);
  }
  cgp_store_x(a, X);
  cgp_write_state(sh, a.cg.st, it, status);
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
// the smallest halo; false: the image does not fit.  Where one unit per scheduler is enough,
// rectangles of four units (32 x 16) do the same on a quarter of the CTAs: they leave the others
// to runs on other streams and have shorter all-reduces.  30 steps of 128 x 128 pixels: 172 us
// (192 with 128 CTAs of one unit); on 8 streams 44 us a run (186; 111 to 147 with two launches
// per iteration, which overlap).  Fewer than 17 CTAs stay as they are (32 x 32, guided, radius 3:
// 251 us against 257), and larger rectangles have no such choice: 256 x 256 pixels take 128 CTAs
// and run one after the other (189 us each; 122 to 147 on 8 streams with two launches).
template <class OP>
bool cgp_rect(int nx, int ny, CgpRect* out, int* nreg) {
  const int maxc = cgp_max_ctas();
  long best = -1;
  auto take = [&](int W, int H, long cost) {
    best = cost;
    out->W = W;
    out->H = H;
    out->ncx = (nx + W - 1) / W;
    *nreg = out->ncx * ((ny + H - 1) / H);
  };
  for (int W = 32; W <= 256; W += 32) {
    const int ncx = (nx + W - 1) / W;
    if (ncx > maxc) continue;
    const int want = std::min(maxc / ncx, (ny + 3) / 4);
    const int H = 4 * ((ny + 4 * want - 1) / (4 * want));
    const int nhalo = 2 * OP::HALO * (W + 2 * OP::HALO) + 2 * OP::HALO * H;
    if (cgp_image_floats<OP>(W, H) * 4 > CGP_SMEM_MAX || nhalo > CGP_HALO_REGS * CGP_T) continue;
    const long cost = (long)((W / 32 * (H / 4) + 3) / 4) * 100000 + nhalo;
    if (best < 0 || cost < best) take(W, H, cost);
  }
  const int four = ((nx + 31) / 32) * ((ny + 15) / 16);
  if (best >= 0 && best < 200000 && *nreg > 16 && 2 * four <= *nreg) take(32, 16, best);
  return best >= 0;
}

// Samples per CTA of a signal: at least 128 (4096 samples in FP64, 20 steps: 160 us; 256: 185),
// 0 if it does not fit.  FP32 runs that would take more than half of the SMs so and not with 256
// samples leave them to runs on other streams where it costs nothing (30 steps of 15000, radius 5:
// 133 us either way, on 8 streams 31 us a run against 75; radius 20: 146 us against 139).
int cgp_line_width(const bf_graph* g) {
  const int maxc = cgp_max_ctas();
  if (maxc < 1) return 0;
  const bool half = g->esize == 4 && g->rx <= 8 && g->n > 64 * (int64_t)maxc && g->n <= 128 * (int64_t)maxc;
  int64_t W = std::max<int64_t>(half ? 256 : 128, (g->n + maxc - 1) / maxc);
  W = std::max<int64_t>((W + 31) / 32 * 32, 2 * g->rx);
  return cgp_line_elems((int)std::min<int64_t>(W, 1 << 20), g->rx) * g->esize > CGP_SMEM_MAX ? 0 : (int)W;
}

bool cgp_is_line(const bf_graph* g) {
  return g->kind == BF_KIND_BILATERAL && g->p.ndim == 1 && g->ry == 0 && g->n < (1 << 28);
}
bool cgp_is_image(const bf_graph* g) {
  return g->kind == BF_KIND_BILATERAL && fast_shape(g) == FAST_R3_2D && g->p.weight_mode == BF_W_ONTHEFLY;
}
// guided images of radius 1 .. 3 in FP32: the radius, else 0
int cgp_guided(const bf_graph* g) {
  return g->kind == BF_KIND_GUIDED && g->esize == 4 && g->ry > 0 && g->rx <= 3 ? g->rx : 0;
}
bool cgp_split(const bf_graph* g, CgpRect* rc, int* nreg) {
  if (cgp_is_image(g)) return cgp_rect<CgpBilateral>(g->nx, g->ny, rc, nreg);
  switch (cgp_guided(g)) {
    case 1: return cgp_rect<CgpGuided<1>>(g->nx, g->ny, rc, nreg);
    case 2: return cgp_rect<CgpGuided<2>>(g->nx, g->ny, rc, nreg);
    case 3: return cgp_rect<CgpGuided<3>>(g->nx, g->ny, rc, nreg);
  }
  return false;
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
  const bool ok = cgp_is_line(g) ? cgp_line_width(g) > 0 : cgp_split(g, &rc, &nreg);
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
  a.frames = (u64*)cg.p_old;
  void* args[] = {&a};
  const int grid = (a.n + a.W - 1) / a.W;
  return cgp_coop(k_cgp_line<T>, grid, CGP_TL, cgp_line_elems(a.W, a.R) * sizeof(T), s, args);
}

template <class OP>
static int cgp_image(OP op, CgpImage& a, int nreg, cudaStream_t s) {
  void* args[] = {&op, &a};
  return cgp_coop(k_cgp_image<OP>, nreg, CGP_T, cgp_image_floats<OP>(a.rc.W, a.rc.H) * 4, s, args);
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
  if (!cgp_split(g, &a.rc, &nreg)) return bf_fail(BF_EINVAL, "cg_filter: image does not fit");
  a.cg = cg;
  a.nx = g->nx;
  a.ny = g->ny;
  a.kmax = kmax;
  a.vec = g->nx % 4 == 0;
  a.slots = (u64*)cg.partials;
  a.frames = (u64*)cg.p_old;
  if (cgp_is_image(g)) {
    CgpBilateral op;
    op.c = run_const(g->gf);
    op.guide = cg.guide;
    return cgp_image(op, a, nreg, s);
  }
  switch (cgp_guided(g)) {
    case 1: return cgp_image(CgpGuided<1>{cg.guide, (const float*)g->gmu, (const float*)g->givar}, a, nreg, s);
    case 2: return cgp_image(CgpGuided<2>{cg.guide, (const float*)g->gmu, (const float*)g->givar}, a, nreg, s);
  }
  return cgp_image(CgpGuided<3>{cg.guide, (const float*)g->gmu, (const float*)g->givar}, a, nreg, s);
}
