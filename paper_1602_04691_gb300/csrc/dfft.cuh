// dfft.cuh - shared-memory-resident FFTs for the paired-FP32 (double-float)
// passes, and for the FP64 passes at the lengths without a register split.
// Paired-FP32 arithmetic costs about ten FP32 instructions per operation, so
// these passes are bound by instruction issue, not memory; fully unrolled
// register transforms of 32 points made the code too large for the
// instruction cache.  Here a tile of C columns x L points sits in shared
// memory and is transformed in place in three stages of radices 8, r2 and r3
// (two stages, 8 and r3, at L = 64 and 128):
//
//   forward: decimation in frequency, natural order in, digit-reversed out
//   inverse: decimation in time, digit-reversed in, natural order out
//
// The callers fuse the outer stages with what surrounds them: the first with
// the global loads, the last (blocks of r3 neighbouring points, no twiddles)
// with the global stores, and the Z pass its last forward stage, the spectrum
// product and its first inverse stage, which all work on the same r3 points.
// A tile so makes two round trips through shared memory per transform and
// three per Z pass beside the middle stage's.  The inverse X and Y passes,
// whose input comes in natural order from global memory, run the DIF stages
// with the inverse sign instead.
#pragma once

#include "dfloat.cuh"

namespace ori {

// Radices of the second and third stage.
template <int L, bool MIXED = is_mixed_len(L)>
struct SRad {
  static constexpr int r3 = L == 256 ? 4 : (L == 128 || L >= 1024) ? 16 : 8;
  static constexpr int r2 = L / 8 / r3;
};
template <int L>
struct SRad<L, true> {
  static constexpr int r2 = MixRad<L>::r2, r3 = MixRad<L>::r3;
};

// After the stages position p = (t1 r2 + t2) r3 + t3 holds frequency
// k = t1 + 8 (t2 + r2 t3): block b = t1 r2 + t2 holds the frequencies
// freq_of_block(b) + (L / r3) t3.
template <int L>
__device__ __forceinline__ int freq_of_block(int b) {
  constexpr int r2 = SRad<L>::r2;
  const int t1 = b / r2;
  return t1 + 8 * (b - t1 * r2);
}
template <int L>
__device__ __forceinline__ int block_of_freq(int k0) {   // k0 < L / r3
  return (k0 & 7) * SRad<L>::r2 + (k0 >> 3);
}

// Layout of a tile in shared memory: idx(j, c, q) is the place of point j of
// column c, q = j / (L / 8); item(g) splits a work item of `per` items a column.
// Columns (Y and Z passes): rows of C columns, neighbouring threads on
// neighbouring columns, the column index swizzled by the row so that both
// row-wise and column-wise warp accesses avoid bank conflicts.
template <int L, int C>
struct ColTile {
  static constexpr int ELEMS = L * C;
  __device__ __forceinline__ static int idx(int j, int c, int) { return j * C + (c ^ (j & (C - 1))); }
  template <int PER>
  __device__ __forceinline__ static void item(int g, int& c, int& i) { c = g % C; i = g / C; }
};
// Lines (X passes): every line on its own, neighbouring threads along the line.
// The last stage takes consecutive frequencies, whose points lie L / 8 apart:
// one element of padding every L / 8 points puts them on different banks (in
// rows of columns 77% of the X passes' shared loads were conflicts).
template <int L, int C>
struct LineTile {
  static constexpr int ELEMS = (L + 8) * C;
  __device__ __forceinline__ static int idx(int j, int c, int q) { return c * (L + 8) + j + q; }
  template <int PER>
  __device__ __forceinline__ static void item(int g, int& c, int& i) { c = g / PER; i = g - c * PER; }
};

// One in-place decimation-in-frequency stage of radix R on all C columns:
// blocks of M points, span s = M / R; outputs multiplied by w_M^(j t').
template <int R, int M, int SIGN, int L, int C, template <int, int> class Lay, class T>
__device__ __forceinline__ void dif_stage(cpx<T>* X, const cpx<T>* tw, int tid, int nt) {
  static_assert(M == L / 8, "the middle stage: one block per eighth of the points");
  constexpr int s = M / R, step = L / M;
  for (int g = tid; g < C * (L / R); g += nt) {
    int c, bi;
    Lay<L, C>::template item<L / R>(g, c, bi);
    const int blk = bi / s, j = bi - blk * s;
    const int base = blk * M + j;
    cpx<T> v[R];
#pragma unroll
    for (int t = 0; t < R; ++t) v[t] = ld_stage(X + Lay<L, C>::idx(base + t * s, c, blk));
    dft<R, SIGN, false>(v);
#pragma unroll
    for (int t = 1; t < R; ++t) v[t] = twL_mul<SIGN>(v[t], tw, j * t * step);   // j t < M
#pragma unroll
    for (int t = 0; t < R; ++t) st_stage(X + Lay<L, C>::idx(base + t * s, c, blk), settle(v[t]));
  }
}

// One in-place decimation-in-time stage: inputs multiplied by w_M^(j t), then
// the radix-R butterfly.
template <int R, int M, int SIGN, int L, int C, template <int, int> class Lay, class T>
__device__ __forceinline__ void dit_stage(cpx<T>* X, const cpx<T>* tw, int tid, int nt) {
  static_assert(M == L / 8, "the middle stage: one block per eighth of the points");
  constexpr int s = M / R, step = L / M;
  for (int g = tid; g < C * (L / R); g += nt) {
    int c, bi;
    Lay<L, C>::template item<L / R>(g, c, bi);
    const int blk = bi / s, j = bi - blk * s;
    const int base = blk * M + j;
    cpx<T> v[R];
#pragma unroll
    for (int t = 0; t < R; ++t) v[t] = ld_stage(X + Lay<L, C>::idx(base + t * s, c, blk));
#pragma unroll
    for (int t = 1; t < R; ++t) v[t] = twL_mul<SIGN>(v[t], tw, j * t * step);   // j t < M
    dft<R, SIGN, false>(v);
#pragma unroll
    for (int t = 0; t < R; ++t) st_stage(X + Lay<L, C>::idx(base + t * s, c, blk), settle(v[t]));
  }
}

// The middle stage (radix r2), forward (DIF, either sign) and inverse (DIT).
template <int L, int C, int SIGN = -1, template <int, int> class Lay = ColTile, class T>
__device__ __forceinline__ void dif_middle(cpx<T>* X, const cpx<T>* tw, int tid, int nt) {
  if constexpr (SRad<L>::r2 > 1) {
    dif_stage<SRad<L>::r2, L / 8, SIGN, L, C, Lay>(X, tw, tid, nt);
    __syncthreads();
  }
}
template <int L, int C, template <int, int> class Lay = ColTile, class T>
__device__ __forceinline__ void dit_middle(cpx<T>* X, const cpx<T>* tw, int tid, int nt) {
  if constexpr (SRad<L>::r2 > 1) {
    dit_stage<SRad<L>::r2, L / 8, +1, L, C, Lay>(X, tw, tid, nt);
    __syncthreads();
  }
}

// The last DIF stage of block `blk` of column c, in registers: v[t] is the
// transform at frequency freq_of_block(blk) + (L / r3) t.
template <int L, int C, int SIGN, template <int, int> class Lay = ColTile, class T>
__device__ __forceinline__ void dif_last(const cpx<T>* X, int blk, int c, cpx<T> (&v)[SRad<L>::r3]) {
  constexpr int r3 = SRad<L>::r3;
#pragma unroll
  for (int t = 0; t < r3; ++t) v[t] = ld_stage(X + Lay<L, C>::idx(blk * r3 + t, c, blk / SRad<L>::r2));
  dft<r3, SIGN, false>(v);
}

// Threads of a tile of C columns, between most / 2 and most: the multiple of 32
// that wastes the fewest thread-points over the three stages.  With `ctas` > 0,
// the few CTAs that shared memory lets on an SM, the warps they make count too:
// W of them hide latency like W / (W + 12) (paired-FP32 Z pass at n = 200, 400
// points: 1.69 ms with two CTAs of 160 threads and the least waste, 1.54 with
// two of 224; at n = 400 12.2 ms with 320 threads, 11.8 with 416; both before
// the renormalisations inside the stages, with which they are 1.61 and 12.7).
template <int L>
constexpr int stage_threads(int C, int most, int ctas = 0) {
  int best = most;
  double best_cost = 1e30;
  for (int nt = (most / 2 + 31) / 32 * 32; nt <= most; nt += 32) {
    double cost = 0;
    for (int r : {8, SRad<L>::r2, SRad<L>::r3}) {
      const int items = C * (L / r);
      if (r > 1) cost += double((items + nt - 1) / nt) * nt * r;
    }
    if (ctas > 0) cost *= 1 + 12.0 / (ctas * (nt / 32));
    if (cost <= best_cost) {
      best_cost = cost;
      best = nt;
    }
  }
  return best;
}

}  // namespace ori
