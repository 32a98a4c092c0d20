// passes.cuh - the FFT passes of the padded 3D convolution (Section 3).
//
// The matvec y = x + K(s x) (K = c_S |Delta| G_off, s = h N or sqrt(h N)) runs
// as five passes over two scratch cubes, each pass an FFT of length L along
// one axis, pruned by the zero padding (Section 3: u is padded with zeros,
// and entries past the n-th are discarded after the inverse transform):
//
//   X fwd : x[z][y][0..n)  --(prologue: scale, COCG update)-->  T1[z][y][0..L)
//   Y fwd : T1[z][0..n)[kx]                                 ->  T2[z][0..L)[kx]
//   Z conv: T2[0..n)[ky][kx] -> FFT -> * Ghat -> IFFT -> keep z < n (in place)
//   Y inv : T2[z][0..L)[kx]                                 ->  T1[z][0..n)[kx]
//   X inv : T1[z][y][0..L) -> keep x < n --(epilogue: y = x + s conv, dots)--> y
//
// T1 is [n][n][L] (C-order, x fastest).  T2 holds its [z][ky][kx] points in
// blocks of B = yblk(L) values of ky, [ky / B][z][ky % B][kx] (below L = 256
// B = L, the plain order).  The Y passes walk ky at a fixed z and the Z pass z
// at a fixed ky; in the plain order a Z tile's n rows lie L^2 points apart
// (8 MB at L = 1024), every one in another page, and the address translation
// was what a tile of narrow rows waited for (8-column Z tiles, n = 512: 3.59 ms
// plain, 3.13 ms in blocks of 128; n = 288: 0.58 and 0.52 ms).  The spectrum is
// stored once for the (L/2+1)^3 distinct entries (the kernel cube is even
// along each axis); column (kx, ky, kz) reads entry (m(kz), m(ky), m(kx)),
// m(k) = min(k, L - k), and already carries c_S |Delta| / L^3.
//
// Every pass computes length-L DFTs on a tile of C lines held by one CTA as
// L = L1 * L2: a length-L1 DFT in registers over j1 (j = j1 L2 + j2), the
// twiddle exp(-2 pi i j2 k1 / L), one exchange through shared memory, and a
// length-L2 DFT over j2 giving X[k1 + L1 k2].  The inverse runs the same two
// stages in the opposite order, so a forward transform followed by an
// inverse (the Z pass) needs no exchange in between.
#pragma once

#include "common.cuh"

#include <cuda.h>   // CUtensorMap (the type only; maps are encoded through the runtime's driver entry point)

#include <algorithm>
#include <initializer_list>

namespace ori {

// Layout of the lines a CTA works on.
enum { LAYOUT_STRIDED = 0,     // C consecutive columns, points at a stride
       LAYOUT_CONTIG = 1 };    // C whole lines, points contiguous (X passes)

enum { SMODE_FWD = 0,          // forward transform, store n_out points
       SMODE_INV = 1,          // inverse transform of L points, store n_out
       SMODE_ZCONV = 2 };      // forward, * spectrum, inverse, store n_out

// Prologue of the X forward pass (value fed at cell (line, j), j < n).
enum { PRO_SCALE = 0,          // v = s[i] * x[i]           (x of type T)
       PRO_SCALE_D = 1,        // v = s[i] * x[i]           (x complex128, cast)
       PRO_COCG_FIRST = 2,     // p = r;          v = s[i] * p
       PRO_COCG = 3,           // p = r + beta p; v = s[i] * p
       PRO_KERNEL = 4 };       // v = G(d |signed offset|) (plan; FP64 only)

// Epilogue of the X inverse pass (conv value v at cell i = line*n + x).
enum { EPI_PLUS = 0,           // y = x + v                   (A form)
       EPI_PLUS_S = 1,         // y = x + s v                 (B form)
       EPI_PLUS_D = 2,         // y = x + v, x,y complex128   (A form, FP32 math)
       EPI_PLUS_S_D = 3,       // y = x + s v, x,y complex128 (B form, FP32 math)
       EPI_COCG = 4,           // q = p + s v; partial sum p^T q
       EPI_RESID = 5,          // r = b - (w + s v); partial sum ||r||^2
       EPI_RECOVER = 6,        // u = w / s, or b - v where s == 0
       EPI_RUPDATE = 7 };      // r -= c (d + s v), r complex128; partial ||r||^2

struct XArgs {
  // prologue
  const void* x;        // input vector (T or double), or r for COCG
  void* p;              // COCG search direction (read/write)
  const void* scale;    // complex scale s (T), n^3
  const void* beta;     // device double2 (COCG)
  // kernel-cube generation (PRO_KERNEL)
  double d, k;
  // epilogue
  const void* xin;      // x (EPI_PLUS*), p (EPI_COCG), w (EPI_RESID/RECOVER)
  const void* bvec;     // b (EPI_RESID, EPI_RECOVER); r (EPI_RUPDATE, in place)
  double coef;          // c of EPI_RUPDATE
  void* out;            // y / q / r / u
  double2* partials;    // per-block partial sums
  // geometry
  const void* in;       // FFT input (T1 for the inverse pass)
  void* fft_out;        // FFT output (T1 for the forward pass)
  int n;                // cells per axis
  int nlines;           // number of lines
  int n_in;             // valid input points (forward)
  int line_len_in;      // elements between lines in the input
  int line_len_out;     // elements between lines in the output
  int lines_per_plane;  // PRO_KERNEL: lines of one z plane (L, or the L/2 + 1 of the even half)
  int plane0;           // PRO_KERNEL: z index of the first plane of the launch
  int mode;             // PRO_* or EPI_*
  const void* twL;      // twiddle table for length L
  const int* done;      // solver flag: the pass returns at once if *done != 0
  // batch of right-hand sides: blockIdx.y selects one; each per-RHS pointer
  // moves by its byte stride (scale, the medium, is shared by all)
  long long bs_x, bs_p, bs_xin, bs_out, bs_bvec, bs_in, bs_fft;
  long long bs_beta;    // bytes between the beta of consecutive RHS
  int done_stride;      // bytes between the flags of consecutive RHS
  const double* coefs;  // EPI_RUPDATE: per-RHS coefficient (overrides coef when set)
  int nrhs;             // right-hand sides in the batch (gridDim.y)
  int sm_count;         // persistent kernels: SMs of the device
  int* err;             // set to 1 by a kernel whose bounded wait on a bulk copy gave up
};

struct SArgs {
  const void* in;
  void* out;
  long long in_outer, out_outer;   // elements between outer indices
  long long in_pt, out_pt;         // elements between points of a line
  // elements between blocks of yblk(L): of the output points of a forward
  // pass, the input points of an inverse pass, the outer index of the Z pass
  long long in_blk, out_blk;
  int ncols;                       // columns per outer index (stride 1)
  int col_blocks;                  // ceil(ncols / C)
  int n_in, n_out;
  int nouter;
  const void* twL;
  const void* ghat;                // spectrum, H^3 entries (SMODE_ZCONV)
  const void* ghatZ;               // FP32 spectrum in Z-tile order [my][kx/W][mz][W], W = zgroup(L)
  int H;                           // L/2 + 1
  const int* done;
  int sm_count;                    // persistent kernels: CTAs to launch
  // batch of right-hand sides (blockIdx.y): byte strides of in/out per RHS,
  // and of the spectra, one spectrum per wave number for rhs_per_ghat RHS
  int nrhs;
  long long bs_in, bs_out, bs_ghat, bs_ghatZ;
  int rhs_per_ghat;
  int done_stride;
  int mirror_in;                   // forward transform of an even sequence stored up to L/2:
                                   // input row j > L/2 is read from row L - j
  // launch schedule of the FP32 Y-forward and Z passes (chosen by the plan's
  // autotuner): SCHED_PERSISTENT = the pipelined persistent kernel
  // with at most cta_cap resident CTAs per SM (0 = as many as fit);
  // SCHED_TILES = one CTA per tile of columns
  int sched;
  int cta_cap;
  int variant;                     // pipelined FP32 kernels: launch variant (has_pipe_variants)
  // FP32 Z and Y passes with 16-column tiles: the input rows of a tile
  // arrive by TMA (cp.async.bulk.tensor) through this map of the input cube:
  // Z pass, dims (kx, ky % B, z, ky / B, right-hand side) of T2 and box
  // (16, 1, zbox, 1, 1); Y forward, dims (kx, y, z, right-hand side) of T1 and box
  // (16, zbox, 1, 1); Y inverse, dims (kx, ky % B, ky / B, z, right-hand side)
  // of T2 and box (16, B, zbox / B, 1, 1); zrows_ok = 0 keeps cp.async
  CUtensorMap zrows;
  int zrows_ok;
  int zbox;
  int* err;                        // set to 1 when a bounded wait on a copy gave up
};

enum { SCHED_PERSISTENT = 0, SCHED_TILES = 1 };

// Columns per group of the Z-tile-ordered FP32 spectrum [my][kx / W][mz][W]: W = kZGroup,
constexpr int kZGroup = 16;
// ... at transform length L, where the Z pass works in groups of fewer columns
// (zconv_groups): their number.
constexpr int zgroup(int L) { return is_mixed_len(L) || L == 1024 ? 8 : kZGroup; }

// Transform length of a grid: the smallest instantiated length >= 2n.  Any
// length >= 2n - 1 gives the same operator, and the work of a pass grows with
// its square, so the lengths between the powers of two pay for themselves
// even though a power of two is 10-20% faster per point (FP32 operator, n =
// 260: 4.72 ms at 1024, 1.17 at 576; n = 200: 0.68 ms at 512, 0.42 at 400; n =
// 100: 0.115 ms at 256, 0.069 at 200).  Below 144 the passes are launch-bound
// and the power of two stays.
constexpr int transform_length(int n, int pow2) {
  for (int m : {144, 200, 288, 400, 576, 800})
    if (m >= 2 * n && m > pow2 / 2 && m < pow2) return m;
  return pow2;
}

// Values of ky per block of T2 at transform length L.  Narrow Z tiles want few
// (rows of a tile within tens of pages), the Y passes many: n = 512, Y forward +
// Z + Y inverse 1.01 + 2.86 + 1.05 ms in blocks of 32, 1.10 + 2.98 + 1.05 in
// blocks of 128; n = 400: 0.67 + 1.73 + 0.59 in blocks of 40, 0.67 + 1.84 + 0.59
// plain; n = 260: what the Z pass gains (0.55 -> 0.53) the Y passes lose.
constexpr int yblk(int L) {
  if (L < 256) return L;
  if (is_mixed_len(L)) return L == 800 ? 40 : L;
  return L == 256 ? 64 : 32;
}
// Offset of point k of a line laid out in blocks: `blk` elements between blocks, `pt` between points of one.
template <int L>
__device__ __forceinline__ long long blk_off(int k, long long blk, long long pt) {
  constexpr int B = yblk(L);
  static_assert(L % B == 0, "whole blocks");
  return (long long)(k / B) * blk + (long long)(k % B) * pt;
}

// Offset of point k + STEP t from that of point k < STEP (`at` = blk_off<L>(k)):
// the block and the place in it move by compile-time amounts when STEP is
// whole blocks or divides one.
template <int L, int STEP>
__device__ __forceinline__ long long blk_at(long long at, int k, int t, long long blk, long long pt) {
  constexpr int B = yblk(L);
  if constexpr (B == L) return at + t * (STEP * pt);
  else if constexpr (STEP % B == 0) return at + t * (STEP / B * blk);
  else if constexpr (B % STEP == 0) return at + (STEP * t / B) * blk + (STEP * t % B) * pt;
  else return blk_off<L>(k + STEP * t, blk, pt);
}

// Rows of one TMA box when boxes of equal size cover exactly `rows` staged rows (at most 256 each).
constexpr int even_box(int rows) {
  int q = (rows + 255) / 256;
  while (rows % q != 0) ++q;
  return rows / q;
}

// ---------------------------------------------------------------------------
// Dependent launches (programmatic stream serialization).  The passes of an
// operator are short kernels one after another: a launch made with this
// attribute brings its CTAs onto SMs that the previous kernel leaves, runs its
// prologue there (the twiddle table in shared memory, barrier set-up) and
// waits in dep_wait until the previous kernel has completed and its writes
// are visible.  Every kernel launched this way calls dep_wait before it
// touches anything another kernel writes or reads (all but the plan's
// twiddle tables), in every thread.  Such a kernel is alive while its
// predecessor still writes, so it reads what a predecessor writes by coherent
// loads only: no __ldg, and no `const __restrict__` parameter, which lets the
// compiler take non-coherent loads, for which nothing may write the data while
// the kernel lives and which dep_wait need not hold back.  __restrict__ stays
// on the arrays of the medium and the caller's right-hand side, complete
// before the chain of launches starts, and on a kernel's own outputs.
// The successor's launch is not triggered
// early: CTAs waiting on an SM from the start of their predecessor cost more
// than the overlap gives (n = 400: FP32 operator 4.14 ms with an early trigger,
// 3.92 without, 3.93 with plain launches; n = 128: 0.112, 0.103 and 0.118 ms).
// FP32 operator (five passes) at n = 100: 79.9 -> 66.7 us; FP64 operator at
// n = 12: 44.0 -> 34.4 us; mixed solve at n = 20: 0.83 -> 0.72 ms, and with the
// solver's vector and control kernels launched the same way 0.73 -> 0.68 ms
// (n = 40: 1.01 -> 0.94; three runs of each side in turn, within 0.002).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class... P, class... A>
inline cudaError_t launch_dep(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                              const A&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Move a pointer by `bytes` (null stays null).
__device__ __forceinline__ const void* bmove(const void* p, long long bytes) {
  return p == nullptr ? p : static_cast<const void*>(static_cast<const char*>(p) + bytes);
}
__device__ __forceinline__ void* bmove(void* p, long long bytes) {
  return p == nullptr ? p : static_cast<void*>(static_cast<char*>(p) + bytes);
}
__device__ __forceinline__ const int* bflag(const int* f, int stride, int rhs) {
  return f == nullptr ? f : reinterpret_cast<const int*>(reinterpret_cast<const char*>(f) + (long long)stride * rhs);
}

// The view of the arguments seen by right-hand side `rhs` of a batch.
__device__ __forceinline__ XArgs x_for_rhs(XArgs a, int rhs) {
  if (a.coefs != nullptr) a.coef = a.coefs[rhs];
  if (rhs == 0) return a;
  a.x = bmove(a.x, a.bs_x * rhs);
  a.p = bmove(a.p, a.bs_p * rhs);
  a.beta = bmove(a.beta, a.bs_beta * rhs);
  a.xin = bmove(a.xin, a.bs_xin * rhs);
  a.bvec = bmove(a.bvec, a.bs_bvec * rhs);
  a.out = bmove(a.out, a.bs_out * rhs);
  a.in = bmove(a.in, a.bs_fft * rhs);
  a.fft_out = bmove(a.fft_out, a.bs_fft * rhs);
  a.done = bflag(a.done, a.done_stride, rhs);
  return a;
}
__device__ __forceinline__ SArgs s_for_rhs(SArgs a, int rhs) {
  if (rhs == 0) return a;
  a.in = bmove(a.in, a.bs_in * rhs);
  a.out = bmove(a.out, a.bs_out * rhs);
  const int g = a.rhs_per_ghat > 0 ? rhs / a.rhs_per_ghat : 0;
  a.ghat = bmove(a.ghat, a.bs_ghat * g);
  a.ghatZ = bmove(a.ghatZ, a.bs_ghatZ * g);
  a.done = bflag(a.done, a.done_stride, rhs);
  return a;
}

// Launch variants of the pipelined FP32 Y-forward, Z and Y-inverse passes at
// the padded lengths where the autotuner chooses among them:
//   0: the default tile (16 columns) and split L = L1 * L2 of Split<L>;
//   1: 8-column tiles, same split;
//   2: 16-column tiles, first stage of radix 2 * L1 (second of L2 / 2).
constexpr bool has_pipe_variants(int L) { return L >= 256 && L <= 1024; }
constexpr int pipe_variants(int L) { return has_pipe_variants(L) ? 3 : 1; }

template <int L, int C, class T, int L1X = Split<L>::L1>
struct Tile {
  static constexpr int L1 = L1X;
  static constexpr int L2 = L / L1X;
  static constexpr int NT = C * L2;            // threads per CTA
  static constexpr int PK = L2 + 1;            // forward exchange [c][k1][j2]
  static constexpr int PC = (L1 * PK) | 1;
  static constexpr int PKI = L1 + 1;           // inverse exchange [c][ja][k1]
  static constexpr int PCI = (L2 * PKI) | 1;
  static constexpr int SMEM_ELEMS = (C * PC > C * PCI) ? C * PC : C * PCI;
  static constexpr size_t SMEM_BYTES = size_t(SMEM_ELEMS) * sizeof(cpx<T>);
  // The FP32 X passes are latency bound: three resident CTAs per SM (the
  // exchange buffer allows it) keep more loads in flight (measured: the X
  // passes gain 20%, the strided Y passes do not, so only the X passes use it).
  static constexpr int MINB = (sizeof(T) == 4 && NT == 256 && SMEM_BYTES <= 72 * 1024) ? 3 : 1;
};

// ---------------------------------------------------------------------------
// Stage helpers shared by both layouts
// ---------------------------------------------------------------------------

// thread t -> (line c, j2) of the first forward stage / second inverse stage
template <int LAYOUT, int C, int L2>
__device__ __forceinline__ void map_t(int t, int& c, int& j) {
  if (LAYOUT == LAYOUT_STRIDED) { c = t % C; j = t / C; }
  else { j = t % L2; c = t / L2; }
}
// item s -> (line c, k1) of the second forward stage / first inverse stage
template <int LAYOUT, int C, int L1>
__device__ __forceinline__ void map_s(int s, int& c, int& k) {
  if (LAYOUT == LAYOUT_STRIDED) { c = s % C; k = s / C; }
  else { k = s % L1; c = s / L1; }
}

// ---------------------------------------------------------------------------
// Warp + block reduction of a double2 partial into partials[blockIdx.x]
// ---------------------------------------------------------------------------
// FP64 additions run at 2 lanes a cycle and SM, so a block's reductions cost
// more than its loads when every lane carries every value through all five
// butterfly steps.  Here the values are split over the lanes first: half the
// lanes go on with one value, half with the other (5 additions a warp for two
// values, 6 for four, instead of 10 and 20).
__device__ __forceinline__ double warp_sum_tail(double v, int from) {
  for (int o = from; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double2 warp_sum2(double2 v) {
  const bool up = (threadIdx.x & 16) != 0;
  double k = up ? v.y : v.x;
  k += __shfl_xor_sync(0xffffffffu, up ? v.x : v.y, 16);
  k = warp_sum_tail(k, 8);
  return make_double2(__shfl_sync(0xffffffffu, k, 0), __shfl_sync(0xffffffffu, k, 16));
}
// Sums of a and b over the warp, valid in every lane.
__device__ __forceinline__ void warp_sum4(double2& a, double2& b) {
  const bool up = (threadIdx.x & 16) != 0, odd = (threadIdx.x & 8) != 0;
  double2 k = up ? b : a;
  const double2 s = up ? a : b;
  k.x += __shfl_xor_sync(0xffffffffu, s.x, 16);
  k.y += __shfl_xor_sync(0xffffffffu, s.y, 16);
  double v = odd ? k.y : k.x;
  v += __shfl_xor_sync(0xffffffffu, odd ? k.x : k.y, 8);
  v = warp_sum_tail(v, 4);
  a = make_double2(__shfl_sync(0xffffffffu, v, 0), __shfl_sync(0xffffffffu, v, 8));
  b = make_double2(__shfl_sync(0xffffffffu, v, 16), __shfl_sync(0xffffffffu, v, 24));
}

// All threads of the block must call it.  Uses 32 double2 of scratch smem.
__device__ __forceinline__ void block_partial(double2 v, double2* red, double2* partials) {
  v = warp_sum2(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double2 s = make_double2(0.0, 0.0);
    for (int i = 0; i < nw; ++i) { s.x += red[i].x; s.y += red[i].y; }
    partials[blockIdx.x] = s;
  }
}

// Like block_partial, but v is already reduced over the warp (valid in lane 0).
__device__ __forceinline__ void block_partial_lane0(double2 v, double2* red, double2* partials) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double2 s = make_double2(0.0, 0.0);
    for (int i = 0; i < nw; ++i) { s.x += red[i].x; s.y += red[i].y; }
    partials[blockIdx.x] = s;
  }
}

// ---------------------------------------------------------------------------
// Pass launchers.  Each arithmetic T (float, double, dfl) and each part (the
// X passes, the strided forward and inverse passes, the Z pass) is explicitly
// instantiated in a translation unit of its own (passes_inst.cu compiled once
// per pair), so that the library builds in parallel.
// ---------------------------------------------------------------------------
struct Scalars;
template <class T> cudaError_t run_xfwd(int L, bool half, const XArgs& a, cudaStream_t s, bool setup);
template <class T> cudaError_t run_xinv(int L, const XArgs& a, Scalars* sc, int fin, cudaStream_t s, bool setup,
                                        unsigned* nblocks);
template <class T> cudaError_t run_strided_fwd(int L, bool half, const SArgs& a, cudaStream_t s, bool setup);
template <class T> cudaError_t run_strided_inv(int L, const SArgs& a, cudaStream_t s, bool setup);
template <class T> cudaError_t run_zconv(int L, const SArgs& a, cudaStream_t s, bool setup);

// One strided pass (SMODE_FWD, SMODE_INV or SMODE_ZCONV) at padded length L.
template <class T>
inline cudaError_t run_strided(int L, int smode, bool half, const SArgs& a, cudaStream_t s, bool setup) {
  if (smode == SMODE_FWD) return run_strided_fwd<T>(L, half, a, s, setup);
  if (smode == SMODE_INV) return run_strided_inv<T>(L, a, s, setup);
  return run_zconv<T>(L, a, s, setup);
}

}  // namespace ori
