// scalars.cuh - device-resident COCG scalars and deterministic grid reductions.
//
// COCG (van der Vorst & Melissen; the solver of Section 1 and Section 3) needs
// two global reductions per iteration: mu = p^T B p, and rho' = r^T r with
// ||r||^2 for the stop test ||r|| / ||RHS|| (Section 4).  The kernels that
// produce the vectors also produce per-block partial sums; the last block to
// finish (an atomic arrival counter, no waiting) adds the partials in a fixed
// order and updates the scalars below on the device, so the host never sits
// in the iteration loop and the result does not depend on block timing.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "passes.cuh"   // warp sums

namespace ori {

enum { FIN_NONE = 0,    // no reduction
       FIN_ALPHA = 1,   // mu = sum p^T q; alpha = rho / mu
       FIN_SUM = 2,     // sum -> sc->sum (generic)
       FIN_UPDATE = 3,  // rho' and ||r||^2 -> beta, stop test
       FIN_INIT = 4 };  // rho and ||r||^2 of the initial residual

enum { DONE_RUNNING = 0, DONE_CONVERGED = 1, DONE_BREAKDOWN = 2,
       DONE_NONFINITE = 3, DONE_MAXIT = 4 };

constexpr int kHistMax = 512;

struct alignas(16) Scalars {
  double2 rho;       // r^T r (unconjugated) of the current residual
  double2 mu;        // p^T q
  double2 alpha;     // rho / mu
  double2 beta;      // rho' / rho
  double2 sum;       // result of FIN_SUM
  double rnorm2;     // ||r||^2 (conjugated) of the current residual
  double rnorm2_0;   // ||r_0||^2
  double target2;    // stop when rnorm2 <= target2
  double tol;        // relative tolerance for FIN_INIT
  int done;          // DONE_*
  int iter;          // iterations finished
  int maxit;
  unsigned count;    // arrival counter of the last-block protocol
  double hist[kHistMax];  // ||r||^2 after each iteration (first kHistMax)
};

__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  const double den = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / den, (a.y * b.x - a.x * b.y) / den);
}

__device__ __forceinline__ bool isfinite2(double2 v) { return isfinite(v.x) && isfinite(v.y); }

// Every block calls this after writing its partial(s).  Returns true in the
// block that arrived last.
__device__ __forceinline__ bool last_block_arrives(Scalars* sc, int& s_last) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned prev = atomicAdd(&sc->count, 1u);
    s_last = (prev == gridDim.x - 1) ? 1 : 0;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}

// Sum of the partials over i in [0, nparts) in a fixed order: partials[i]
// -> a, or with PAIRS partials[2 i] -> a and partials[2 i + 1] -> b in one
// sweep.  Called by all threads of the last block (whole warps); valid in
// thread 0.
template <bool PAIRS>
__device__ __forceinline__ void reduce_partials(const double2* partials, int nparts, double2* red, double2& a,
                                                double2& b) {
  a = make_double2(0.0, 0.0);
  b = make_double2(0.0, 0.0);
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) {
    const double2 v = __ldcg(partials + (PAIRS ? 2LL * i : i));
    a.x += v.x;
    a.y += v.y;
    if (PAIRS) {
      const double2 w = __ldcg(partials + 2LL * i + 1);
      b.x += w.x;
      b.y += w.y;
    }
  }
  if (PAIRS) warp_sum4(a, b);
  else a = warp_sum2(a);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  // the caller's scratch holds 32 double2: pairs take two rounds of it
  for (int which = 0; which < (PAIRS ? 2 : 1); ++which) {
    __syncthreads();
    if (lane == 0) red[w] = which == 0 ? a : b;
    __syncthreads();
    if (threadIdx.x == 0) {
      double2 t = make_double2(0.0, 0.0);
      for (int i = 0; i < nw; ++i) { t.x += red[i].x; t.y += red[i].y; }
      if (which == 0) a = t;
      else b = t;
    }
  }
  __syncthreads();
}

// Scalar update by the last block.  Partials hold one double2 per block
// (FIN_ALPHA, FIN_SUM) or two (FIN_UPDATE, FIN_INIT: r^T r, then (||r||^2, 0)).
__device__ __forceinline__ void finalize(Scalars* sc, const double2* partials, int nparts, int fin,
                                         double2* red) {
  if (fin == FIN_ALPHA || fin == FIN_SUM) {
    double2 s, none;
    reduce_partials<false>(partials, nparts, red, s, none);
    if (threadIdx.x == 0) {
      if (fin == FIN_SUM) {
        sc->sum = s;
      } else {
        sc->mu = s;
        if (!isfinite2(s)) {
          sc->done = DONE_NONFINITE;
        } else if (s.x == 0.0 && s.y == 0.0) {
          sc->done = DONE_BREAKDOWN;
        } else {
          sc->alpha = cdiv(sc->rho, s);
          if (!isfinite2(sc->alpha)) sc->done = DONE_BREAKDOWN;
        }
      }
      sc->count = 0;
    }
    return;
  }
  double2 rr, nn;
  reduce_partials<true>(partials, nparts, red, rr, nn);
  if (threadIdx.x == 0) {
    const double rn2 = nn.x;
    if (fin == FIN_INIT) {
      sc->rho = rr;
      sc->rnorm2 = rn2;
      sc->rnorm2_0 = rn2;
      sc->target2 = sc->tol * sc->tol * rn2;
      sc->iter = 0;
      sc->beta = make_double2(0.0, 0.0);
      // a residual that already meets the target needs no iteration; a nonzero
      // residual with r^T r = 0 cannot start COCG (rho is the divisor of beta)
      sc->done = (!isfinite(rn2) || !isfinite2(rr)) ? DONE_NONFINITE
               : ((rn2 == 0.0 || rn2 <= sc->target2) ? DONE_CONVERGED
               : ((rr.x == 0.0 && rr.y == 0.0) ? DONE_BREAKDOWN : DONE_RUNNING));
    } else {
      const int it = sc->iter + 1;
      sc->iter = it;
      sc->rnorm2 = rn2;
      if (it <= kHistMax) sc->hist[it - 1] = rn2;
      if (!isfinite(rn2) || !isfinite2(rr)) {
        sc->done = DONE_NONFINITE;
      } else if (rn2 <= sc->target2) {
        sc->done = DONE_CONVERGED;
      } else if (rr.x == 0.0 && rr.y == 0.0) {
        sc->done = DONE_BREAKDOWN;
      } else if (it >= sc->maxit) {
        sc->done = DONE_MAXIT;
      }
      sc->beta = cdiv(rr, sc->rho);
      // beta = rho' / rho: a vanished rho (or a rho' at rounding level over it)
      // is a breakdown, not a NaN to carry into p
      if (sc->done == DONE_RUNNING && !isfinite2(sc->beta)) sc->done = DONE_BREAKDOWN;
      sc->rho = rr;
    }
    sc->count = 0;
  }
}

}  // namespace ori
