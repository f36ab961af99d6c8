// What the CG translation units share: the scalar state of a run and the arguments of its
// kernels.
#pragma once

#include "bf_internal.cuh"

enum { CG_RUN = 0, CG_CONV = 1, CG_BREAK = 2, CG_NONFINITE = 3, CG_TIMEOUT = 4 };

struct CgState {
  double sr;        // s^T r of the current residual
  double ss;        // s^T s
  double rr;        // r^T r
  double pq;        // p^T q
  double alpha;
  double beta;      // beta to use in the next direction update
  double ref2;      // ||b||^2 (or ||r_0||^2 when b = 0)
  double tol2;
  int status;
  int iter;         // completed iterations
  int beta_mode;
  int pad;
  unsigned int counter;
  unsigned int pad2;
};

template <typename T>
struct CgArgs {
  const T* x0;
  T* x;
  T* r;
  T* s;
  T* q;
  const T* p_old;
  T* p_new;
  const T* guide;
  const T* dinv;       // Jacobi preconditioner (NULL: identity)
  const T* d;          // degree (the 7 x 7 paths divide by it)
  const void* wf;
  int wmode;
  int64_t n;
  T shift;
  int first;           // first iteration: p = s
  double* partials;
  CgState* st;
  double* hist;        // [2 kmax] or NULL
  int absent;          // testing: the CTA of a one-launch run that leaves before it sends anything (-1: none)
};

// The whole run in one cooperative launch with its vectors on the chip (bf_cgp.cu).
// cgp_words: 64-bit words of exchange area a run needs at a.partials, 0 when the graph does
// not fit; it also exchanges vector frames in a.p_old (8 bytes per sample, 16 in FP64: both
// direction buffers, which must be contiguous).  Both areas hold zeros before the launch
// (k_cg_state_init).  cgp_launch: BF_OK after enqueuing it.
size_t cgp_words(const bf_graph* g);
template <typename T>
int cgp_launch(const bf_graph* g, const CgArgs<T>& a, int kmax, cudaStream_t s);
