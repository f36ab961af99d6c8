// Window sums of the 7 x 7 image window for one column of values (k = 1) with weights
// recomputed from the guide, by horizontal runs in packed arithmetic: the inner loop of the
// CG filter (Algorithm 2, q = L p), of bf_apply at k = 1, of the bilateral step D^-1 W x and
// of the degree.
//
// A thread owns a run of RUN_P = 4 consecutive pixels of one row.  For each of the 7 window
// rows it reads the 12 staged values around its run as three 16-byte vectors, i.e. as six
// aligned register pairs; a pair holds two neighbouring taps, and for every pixel of the run
// three aligned pairs and one single value cover the 7 taps of the row.  So all but one tap
// of a row go through two-lane instructions (f32x2): per two taps
//   dl = g_i - g_j, t = dl * (-a_r), e = t * dl + ls, (w = 2^e each), df = v_i - v_j,
//   acc += w * df
// are 5 issue slots and 2 exponentials instead of 10 and 2.  The FP32 pipe runs two-lane
// instructions at half rate, so what is saved is issue slots: one pixel per thread and
// scalar instructions needed 473 issue slots per pixel of which 240 were FP32 arithmetic;
// here the 48 taps take about 190 slots, and the bound is the FP32 pipe itself (240 cycles
// per 32 pixels and scheduler; the exponentials take 192 of the SFU beside it).
//
// A neighbour outside the image does not exist.  The guide is staged as +inf there, which
// makes the exponent -inf and the weight exactly 0, so no tile needs coordinate tests.  For
// sigma_r = inf (a_r = 0) the guide is staged as 0 inside the image and -1 takes the place
// of -a_r: the exponent is ls inside and -inf outside.
//
// Measured (GB300, 2070 MHz): 430 cycles per 32 pixels and scheduler in the kernels that use
// it; all taps in scalar instructions 472; two, three or four CTAs per SM alike.
#pragma once

#include "bf_internal.cuh"
#include "bf_window_fast.cuh"

#define RUN_P 4
#define RUN_R 3
#define RUN_TW 64
#define RUN_TH 16
#define RUN_THREADS (RUN_TW * RUN_TH / RUN_P)
#define RUN_XS (RUN_TW + 8)                    // staged columns bx - 4 .. bx + 67
#define RUN_HH (RUN_TH + 2 * RUN_R)            // staged rows by - 3 .. by + 18
#define RUN_HP (RUN_HH * RUN_XS)

typedef unsigned long long run_f2;             // two FP32 lanes

// Exponent constants of the window: -a_r, and ls by |dy| for the tap pairs that start at
// dx = -3 .. 2 and for the single taps at dx = +-3.
struct RunConst {
  float2 pair[RUN_R + 1][6];
  float one[RUN_R + 1];                        // |dx| = 3
  float one1;                                  // (0, +-1)
  float nar;
  int use_guide;                               // 0: a_r = 0
};

inline RunConst run_const(const Geom<float>& g) {
  RunConst c;
  for (int ady = 0; ady <= RUN_R; ++ady) {
    const float* ls = g.ls + (ady + RUN_R) * 7 + RUN_R;
    for (int p = 0; p < 6; ++p) c.pair[ady][p] = make_float2(ls[p - 3], ls[p - 2]);
    c.one[ady] = ls[3];
  }
  c.one1 = g.ls[RUN_R * 7 + RUN_R + 1];
  c.use_guide = g.a_r > 0.0f;
  c.nar = c.use_guide ? -g.a_r : -1.0f;
  return c;
}

__device__ __forceinline__ run_f2 run_sub(run_f2 a, run_f2 b) {
  run_f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ run_f2 run_add(run_f2 a, run_f2 b) {
  run_f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ run_f2 run_mul(run_f2 a, run_f2 b) {
  run_f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ run_f2 run_fma(run_f2 a, run_f2 b, run_f2 c) {
  run_f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ float run_ex2(float a) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ float run_lo(run_f2 v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float run_hi(run_f2 v) { return __uint_as_float((unsigned)(v >> 32)); }

// The sums of one thread's run, in three parts per pixel (two lanes and the single taps).
template <bool NEED_V, bool NEED_W>
struct RunAcc {
  run_f2 a2[RUN_P], w2[RUN_P];
  float a1[RUN_P], w1[RUN_P];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < RUN_P; ++j) {
      a2[j] = w2[j] = 0ull;
      a1[j] = w1[j] = 0.0f;
    }
  }
  __device__ __forceinline__ float sum(int j) const { return (run_lo(a2[j]) + run_hi(a2[j])) + a1[j]; }
  __device__ __forceinline__ float wsum(int j) const { return (run_lo(w2[j]) + run_hi(w2[j])) + w1[j]; }
};

// 12 staged values as six pairs.
__device__ __forceinline__ void run_ld(const float* row, run_f2 (&p)[6]) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(row + 4 * q);
    p[2 * q] = t.x;
    p[2 * q + 1] = t.y;
  }
}

// One window row (|dy| = ADY) of the run: gp, vp the row's pairs; gi2, vi2 the run's own
// guide and values, each twice.  Entry e of the 12 staged values is the tap dx = e - 4 - j
// of pixel j.
template <int ADY, bool NEED_V, bool NEED_W>
__device__ __forceinline__ void run_row(const RunConst& c, run_f2 nar2, const run_f2 (&gp)[6], const run_f2 (&vp)[6],
                                        const run_f2 (&gi2)[RUN_P], const run_f2 (&vi2)[RUN_P],
                                        RunAcc<NEED_V, NEED_W>& s) {
#pragma unroll
  for (int j = 0; j < RUN_P; ++j) {
    const int a0 = (j + 2) / 2;                // first pair that lies in the window
    const int d0 = 2 * a0 - 4 - j;             // its first dx: -2 (j even) or -3 (j odd)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int a = a0 + q, dx = d0 + 2 * q;
      if (ADY == 0 && (dx == 0 || dx == -1)) { // the pair with the pixel itself: its other tap
        const float gj = dx == 0 ? run_hi(gp[a]) : run_lo(gp[a]);
        const float dl = run_lo(gi2[j]) - gj;
        const float w = run_ex2(fmaf(dl * c.nar, dl, c.one1));
        if (NEED_V) s.a1[j] = fmaf(w, run_lo(vi2[j]) - (dx == 0 ? run_hi(vp[a]) : run_lo(vp[a])), s.a1[j]);
        if (NEED_W) s.w1[j] += w;
        continue;
      }
      const run_f2 dl = run_sub(gi2[j], gp[a]);
      const float2 lsf = c.pair[ADY][dx + 3];
      const run_f2 e = run_fma(run_mul(dl, nar2), dl, f2_pack(lsf.x, lsf.y));
      const run_f2 w = f2_pack(run_ex2(run_lo(e)), run_ex2(run_hi(e)));
      if (NEED_V) s.a2[j] = run_fma(w, run_sub(vi2[j], vp[a]), s.a2[j]);
      if (NEED_W) s.w2[j] = run_add(s.w2[j], w);
    }
    // the single tap: dx = -3 (j even, entry j + 1) or dx = 3 (j odd, entry j + 7)
    const int e1 = (j & 1) ? j + 7 : j + 1;
    const float gj = (e1 & 1) ? run_hi(gp[e1 / 2]) : run_lo(gp[e1 / 2]);
    const float dl = run_lo(gi2[j]) - gj;
    const float w = run_ex2(fmaf(dl * c.nar, dl, c.one[ADY]));
    if (NEED_V) s.a1[j] = fmaf(w, run_lo(vi2[j]) - ((e1 & 1) ? run_hi(vp[e1 / 2]) : run_lo(vp[e1 / 2])), s.a1[j]);
    if (NEED_W) s.w1[j] += w;
  }
}

// acc[j] = sum_{j' != i} w (v_i - v_j'), ws[j] = sum w for the run whose window's top left
// staged vector (row dy = -3, column x0 - 4) is at sv, sg; row stride xs floats (a multiple
// of 4).  vi returns the run's own values.
template <bool NEED_V, bool NEED_W>
__device__ __forceinline__ void run_sums(const RunConst& c, const float* sv, const float* sg, int xs,
                                         float (&vi)[RUN_P], float (&acc)[RUN_P], float (&ws)[RUN_P]) {
  RunAcc<NEED_V, NEED_W> s;
  s.clear();
  run_f2 gi2[RUN_P], vi2[RUN_P], gp[6], vp[6];
  const run_f2 nar2 = f2_pack(c.nar, c.nar);
  run_ld(sg + RUN_R * xs, gp);
  if (NEED_V) run_ld(sv + RUN_R * xs, vp);
#pragma unroll
  for (int j = 0; j < RUN_P; ++j) {
    const float gj = (j & 1) ? run_hi(gp[2 + j / 2]) : run_lo(gp[2 + j / 2]);
    gi2[j] = f2_pack(gj, gj);
    vi[j] = 0.0f;
    if (NEED_V) vi[j] = (j & 1) ? run_hi(vp[2 + j / 2]) : run_lo(vp[2 + j / 2]);
    vi2[j] = f2_pack(vi[j], vi[j]);
  }
  run_row<0, NEED_V, NEED_W>(c, nar2, gp, vp, gi2, vi2, s);
#define RUN_ROWS(A)                                                      \
  run_ld(sg + (RUN_R - A) * xs, gp);                                     \
  if (NEED_V) run_ld(sv + (RUN_R - A) * xs, vp);                         \
  run_row<A, NEED_V, NEED_W>(c, nar2, gp, vp, gi2, vi2, s);              \
  run_ld(sg + (RUN_R + A) * xs, gp);                                     \
  if (NEED_V) run_ld(sv + (RUN_R + A) * xs, vp);                         \
  run_row<A, NEED_V, NEED_W>(c, nar2, gp, vp, gi2, vi2, s);
  RUN_ROWS(1)
  RUN_ROWS(2)
  RUN_ROWS(3)
#undef RUN_ROWS
#pragma unroll
  for (int j = 0; j < RUN_P; ++j) {
    acc[j] = NEED_V ? s.sum(j) : 0.0f;
    ws[j] = NEED_W ? s.wsum(j) : 0.0f;
  }
}

// ---- tiles --------------------------------------------------------------------------------
__host__ __device__ inline int run_tiles_x(int nx) { return (nx + RUN_TW - 1) / RUN_TW; }
__host__ __device__ inline int run_tiles_y(int ny) { return (ny + RUN_TH - 1) / RUN_TH; }

// Arrays of a stage: src[a][gp * ld[a]] (NULL: not staged); array 0 holds the values, array
// NA - 1 the guide (+inf outside the image, see RunConst::use_guide; the others are 0 there).
template <int NA>
struct RunSrc {
  const float* p[NA];
  int64_t ld[NA];
  int vec;                                     // rows are whole aligned 16-byte vectors
};

template <int NA>
inline void run_src_vec(RunSrc<NA>& s, int nx) {
  s.vec = nx % 4 == 0;
  for (int a = 0; a < NA; ++a) {
    if (s.p[a] && (s.ld[a] != 1 || ((uintptr_t)s.p[a] & 15))) s.vec = 0;
  }
}

template <int NA>
__device__ __forceinline__ void run_issue(const RunConst& c, int bx, int by, int nx, int ny, const RunSrc<NA>& src,
                                          float* stage) {
  const unsigned base = (unsigned)__cvta_generic_to_shared(stage);
  const float inf = __int_as_float(0x7f800000);
  if (src.vec) {                               // a group of four columns is in the image or not
    for (int q = threadIdx.x; q < RUN_HH * (RUN_XS / 4); q += RUN_THREADS) {
      const int hy = q / (RUN_XS / 4), h4 = q - hy * (RUN_XS / 4);
      const int gy = by - RUN_R + hy, gx = bx - 4 + 4 * h4;
      const bool in = (unsigned)gx < (unsigned)nx && (unsigned)gy < (unsigned)ny;
      const int64_t gp = in ? (int64_t)gy * nx + gx : 0;
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        if (!src.p[a]) continue;
        if (a == NA - 1 && !in) {
          *reinterpret_cast<float4*>(stage + a * RUN_HP + 4 * q) = make_float4(inf, inf, inf, inf);
        } else {
          const bool rd = in && (a < NA - 1 || c.use_guide);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(base + 4u * (unsigned)(a * RUN_HP + 4 * q)),
                       "l"(src.p[a] + gp), "r"(rd ? 16 : 0) : "memory");
        }
      }
    }
  } else {
    for (int hy = threadIdx.x >> 5; hy < RUN_HH; hy += RUN_THREADS / 32) {
#pragma unroll
      for (int h0 = 0; h0 < RUN_XS; h0 += 32) {
        const int hx = h0 + (threadIdx.x & 31);
        if (hx >= RUN_XS) continue;
        const int q = hy * RUN_XS + hx;
        const int gy = by - RUN_R + hy, gx = bx - 4 + hx;
        const bool in = (unsigned)gx < (unsigned)nx && (unsigned)gy < (unsigned)ny;
        const int64_t gp = in ? (int64_t)gy * nx + gx : 0;
#pragma unroll
        for (int a = 0; a < NA; ++a) {
          if (!src.p[a]) continue;
          if (a == NA - 1 && !in) {
            stage[a * RUN_HP + q] = inf;
          } else {
            const bool rd = in && (a < NA - 1 || c.use_guide);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(base + 4u * (unsigned)(a * RUN_HP + q)),
                         "l"(src.p[a] + gp * src.ld[a]), "r"(rd ? 4 : 0) : "memory");
          }
        }
      }
    }
  }
}

// Walk this CTA's 64 x 16 tiles (grid-stride) with the next tile's copies in flight.
// combine(stage) runs between a tile's arrival and its sums when COMBINE (it may rewrite
// array 0 from the others, RUN_HP floats apart); epi(x0, y, vi, acc, ws) consumes the sums
// of the thread's run (first pixel (x0, y), which may lie outside the image).  A warp covers
// 32 x 4 pixels.  Dynamic shared memory: run_smem(NA).
__host__ __device__ constexpr int run_smem(int na) { return 2 * na * RUN_HP * 4; }

template <int NA, bool NEED_V, bool NEED_W, bool COMBINE, class Combine, class Epi>
__device__ __forceinline__ void run_tiles(const RunConst& c, int nx, int ny, const RunSrc<NA>& src, Combine combine,
                                          Epi epi) {
  extern __shared__ __align__(16) float run_stage[];
  const int ntx = run_tiles_x(nx), ntiles = ntx * run_tiles_y(ny);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int cx = 32 * (wid & 1) + 4 * (lane & 7), ry = 4 * (wid >> 1) + (lane >> 3);
  int t = blockIdx.x;
  if (t < ntiles) run_issue<NA>(c, (t % ntx) * RUN_TW, (t / ntx) * RUN_TH, nx, ny, src, run_stage);
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int b = 0; t < ntiles; t += gridDim.x, b ^= 1) {
    const int tn = t + gridDim.x;
    float* cur = run_stage + b * NA * RUN_HP;
    if (tn < ntiles)
      run_issue<NA>(c, (tn % ntx) * RUN_TW, (tn / ntx) * RUN_TH, nx, ny, src, run_stage + (b ^ 1) * NA * RUN_HP);
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    if (COMBINE) {
      combine(cur);
      __syncthreads();
    }
    float vi[RUN_P], acc[RUN_P], ws[RUN_P];
    const float* top = cur + ry * RUN_XS + cx;
    run_sums<NEED_V, NEED_W>(c, top, top + (NA - 1) * RUN_HP, RUN_XS, vi, acc, ws);
    epi((t % ntx) * RUN_TW + cx, (t / ntx) * RUN_TH + ry, vi, acc, ws);
    __syncthreads();                           // the stage is refilled in the next iteration
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// The run's pixels in the image: 0 .. RUN_P.
__device__ __forceinline__ int run_count(int x0, int y, int nx, int ny) {
  if (y >= ny || x0 >= nx) return 0;
  return min(RUN_P, nx - x0);
}

// Store a run of 4 values at p[i0 ..] (cnt of them in the image).
__device__ __forceinline__ void run_store(float* p, int64_t i0, int cnt, bool vec, const float (&v)[RUN_P]) {
  if (vec && cnt == RUN_P) {
    *reinterpret_cast<float4*>(p + i0) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int j = 0; j < RUN_P; ++j)
      if (j < cnt) p[i0 + j] = v[j];
  }
}
// Load a run (0 past the image).
__device__ __forceinline__ void run_load(const float* p, int64_t i0, int cnt, bool vec, float (&v)[RUN_P]) {
  if (vec && cnt == RUN_P) {
    const float4 t = *reinterpret_cast<const float4*>(p + i0);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else {
#pragma unroll
    for (int j = 0; j < RUN_P; ++j) v[j] = j < cnt ? p[i0 + j] : 0.0f;
  }
}
