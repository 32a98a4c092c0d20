// common.cuh - complex arithmetic, twiddle factors and in-register DFTs for
// the FFT passes of the convolution matvec (Section 3, Eq. 3.3.8).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace ori {

// ---------------------------------------------------------------------------
// Complex numbers (interleaved re, im; 8 bytes for float, 16 for double)
// ---------------------------------------------------------------------------
template <class T>
struct alignas(2 * sizeof(T)) cpx {
  T x, y;
};

template <class T>
__host__ __device__ __forceinline__ cpx<T> mkc(T a, T b) { return cpx<T>{a, b}; }
template <class T>
__device__ __forceinline__ cpx<T> operator+(cpx<T> a, cpx<T> b) { return {a.x + b.x, a.y + b.y}; }
template <class T>
__device__ __forceinline__ cpx<T> operator-(cpx<T> a, cpx<T> b) { return {a.x - b.x, a.y - b.y}; }
// FP32 complex sums as one packed two-lane instruction (add/sub.rn.f32x2,
// sm_100 and later): the same rounding per lane as two scalar operations,
// half the issue slots.  The FFT passes are bound by instruction issue, and
// their butterflies are mostly complex additions.
__device__ __forceinline__ unsigned long long pack2(cpx<float> a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ cpx<float> unpack2(unsigned long long v) {
  cpx<float> r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
template <>
__device__ __forceinline__ cpx<float> operator+(cpx<float> a, cpx<float> b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
template <>
__device__ __forceinline__ cpx<float> operator-(cpx<float> a, cpx<float> b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}

template <class T>
__device__ __forceinline__ cpx<T> cmul(cpx<T> a, cpx<T> b) {
  return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <class T>
__device__ __forceinline__ cpx<T> cscale(cpx<T> a, T s) { return {a.x * s, a.y * s}; }
template <class T>
__device__ __forceinline__ cpx<T> czero() { return {T(0), T(0)}; }

template <class D, class S>
__device__ __forceinline__ cpx<D> ccast(cpx<S> a) { return {D(a.x), D(a.y)}; }

// ---------------------------------------------------------------------------
// Twiddles.  cos/sin of 2 pi j / M are evaluated at compile time from their
// Taylor series on [0, pi/4] after an exact reduction by octant symmetry.
// ---------------------------------------------------------------------------
constexpr double kPi = 3.14159265358979323846264338327950288;

constexpr double taylor_sin(double x) {
  double t = x, s = x;
  for (int i = 1; i < 16; ++i) {
    t *= -x * x / double((2 * i) * (2 * i + 1));
    s += t;
  }
  return s;
}
constexpr double taylor_cos(double x) {
  double t = 1.0, s = 1.0;
  for (int i = 1; i < 16; ++i) {
    t *= -x * x / double((2 * i - 1) * (2 * i));
    s += t;
  }
  return s;
}

// (cos, sin) of 2 pi j / M for M divisible by 8.
struct CosSin {
  double c, s;
};
constexpr CosSin turn_cos_sin(long long j, long long M) {
  long long jm = ((j % M) + M) % M;
  const long long m8 = M / 8;
  const long long oct = jm / m8, rem = jm % m8;
  const double step = 2.0 * kPi / double(M);
  const double phi = double(rem) * step;          // in [0, pi/4)
  const double phr = double(m8 - rem) * step;     // in (0, pi/4]
  const double cp = taylor_cos(phi), sp = taylor_sin(phi);
  const double cr = taylor_cos(phr), sr = taylor_sin(phr);
  switch (oct) {
    case 0: return {cp, sp};
    case 1: return {sr, cr};
    case 2: return {-sp, cp};
    case 3: return {-cr, sr};
    case 4: return {-cp, -sp};
    case 5: return {-sr, -cr};
    case 6: return {sp, -cp};
    default: return {cr, -sr};
  }
}

// cos/sin of 2 pi j / 64 for the in-register DFTs (radix up to 64).
struct Tw64 {
  double c[64];
  double s[64];
  float cf[64];
  float sf[64];
};
constexpr Tw64 make_tw64() {
  Tw64 t{};
  for (int j = 0; j < 64; ++j) {
    CosSin v = turn_cos_sin(j, 64);
    t.c[j] = v.c;
    t.s[j] = v.s;
    t.cf[j] = float(v.c);
    t.sf[j] = float(v.s);
  }
  return t;
}

__constant__ Tw64 c_tw64 = make_tw64();

template <class T>
__device__ __forceinline__ T tw64c(int i);
template <>
__device__ __forceinline__ float tw64c<float>(int i) { return c_tw64.cf[i]; }
template <>
__device__ __forceinline__ double tw64c<double>(int i) { return c_tw64.c[i]; }
template <class T>
__device__ __forceinline__ T tw64s(int i);
template <>
__device__ __forceinline__ float tw64s<float>(int i) { return c_tw64.sf[i]; }
template <>
__device__ __forceinline__ double tw64s<double>(int i) { return c_tw64.s[i]; }

// z * exp(SIGN * 2 pi i idx / 64); idx is a compile-time constant after
// unrolling, so trivial factors cost nothing and the others read the
// constant bank directly.
template <int SIGN, class T>
__device__ __forceinline__ cpx<T> tw64_mul(cpx<T> z, int idx) {
  idx &= 63;
  if (idx == 0) return z;
  if (idx == 32) return {-z.x, -z.y};
  if (idx == 16) return SIGN > 0 ? cpx<T>{-z.y, z.x} : cpx<T>{z.y, -z.x};
  if (idx == 48) return SIGN > 0 ? cpx<T>{z.y, -z.x} : cpx<T>{-z.y, z.x};
  const T c = tw64c<T>(idx);
  const T s = SIGN > 0 ? tw64s<T>(idx) : -tw64s<T>(idx);
  return cmul(z, cpx<T>{c, s});
}

// Read-only cached loads of one complex number.
__device__ __forceinline__ cpx<float> ldgc(const cpx<float>* p) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(p));
  return {v.x, v.y};
}
__device__ __forceinline__ cpx<double> ldgc(const cpx<double>* p) {
  const double2 v = __ldg(reinterpret_cast<const double2*>(p));
  return {v.x, v.y};
}

// Load and store of one complex value as the FFT stages keep it in shared
// memory and as the twiddle tables hold it: T's own layout here; paired FP32
// specialises the pair (dfloat.cuh).
template <class T> __device__ __forceinline__ cpx<T> ld_stage(const cpx<T>* p) { return *p; }
template <class T> __device__ __forceinline__ void st_stage(cpx<T>* p, cpx<T> v) { *p = v; }

// z * exp(SIGN * 2 pi i m / L) from a table tab[m] = (cos, sin)(2 pi m / L).
template <int SIGN, class T>
__device__ __forceinline__ cpx<T> twL_mul(cpx<T> z, const cpx<T>* __restrict__ tab, int m) {
  // generic load: the table may sit in global memory or in shared memory
  const cpx<T> w = ld_stage(tab + m);
  return cmul(z, cpx<T>{w.x, SIGN > 0 ? w.y : -w.y});
}

constexpr int bitrev(int i, int R) {
  int r = 0;
  for (int b = 1; b < R; b <<= 1) {
    r = (r << 1) | (i & 1);
    i >>= 1;
  }
  return r;
}

// z * (SIGN i): a quarter turn, no arithmetic.
template <int SIGN, class T>
__device__ __forceinline__ cpx<T> mul_i(cpx<T> z) {
  return SIGN > 0 ? cpx<T>{-z.y, z.x} : cpx<T>{z.y, -z.x};
}

// In-register DFT of size R (power of two, R <= 64):
//   a[k] <- sum_j a[j] exp(SIGN 2 pi i j k / R).
// Decimation in frequency, then the bit-reversal permutation (free: all
// indices are compile-time constants).  The stages go two at a time as
// radix-4 butterflies, a final radix-2 stage when log2 R is odd.  A radix-4
// butterfly leaves the array exactly as the two radix-2 stages it replaces
// (spans s and s/2 of a block of M = 2s points, w = exp(SIGN 2 pi i / M)):
// for x0..x3 = a[j], a[j + s/2], a[j + s], a[j + 3s/2] and
// t0 = x0 + x2, t1 = x0 - x2, t2 = x1 + x3, t3 = SIGN i (x1 - x3),
//   a[j] = t0 + t2,           a[j + s/2] = (t0 - t2) w^2j,
//   a[j + s] = (t1 + t3) w^j, a[j + 3s/2] = (t1 - t3) w^3j,
// since w^(s/2) = SIGN i; it needs three twiddle products where the two
// radix-2 stages need four (34 -> 28 nontrivial products at R = 32, measured:
// the FP32 Z pass 3.43 -> 3.36 ms at n = 512).  HALF: a[j] = 0 for j >= R/2
// on input (the zero padding of Section 3), so the first butterflies have
// x2 = x3 = 0.
// Radix-2 form of the same transform (every stage span s = R/2, R/4, ..., 1;
// the outputs multiplied by w^j of their block): the small transforms (R <= 8,
// the radix-8 stages of the paired-FP32 passes), where the radix-4 form
// saves no twiddle product.
template <int R, int SIGN, bool HALF, class T>
__device__ __forceinline__ void dft_radix2(cpx<T> (&a)[R]) {
#pragma unroll
  for (int s = R / 2; s >= 1; s >>= 1) {
#pragma unroll
    for (int b = 0; b < R; b += 2 * s) {
#pragma unroll
      for (int j = 0; j < s; ++j) {
        const int idx = j * (64 / (2 * s));
        const cpx<T> u = a[b + j];
        if (HALF && s == R / 2) {
          a[b + j + s] = tw64_mul<SIGN>(u, idx);
        } else {
          const cpx<T> v = a[b + j + s];
          a[b + j] = u + v;
          a[b + j + s] = tw64_mul<SIGN>(u - v, idx);
        }
      }
    }
  }
  cpx<T> t[R];
#pragma unroll
  for (int i = 0; i < R; ++i) t[i] = a[bitrev(i, R)];
#pragma unroll
  for (int i = 0; i < R; ++i) a[i] = t[i];
}

// ---------------------------------------------------------------------------
// Sizes with a factor 3 or 5 (R = P Q, P a power of two, Q = 3 or 5): the
// in-register transforms of the padded lengths between powers of two.
// ---------------------------------------------------------------------------
constexpr bool is_pow2(int v) { return (v & (v - 1)) == 0; }
constexpr int pow2_part(int v) { return (v & 1) ? 1 : 2 * pow2_part(v / 2); }

// cos/sin of 2 pi j / M, M divisible by 8, rounded from a double-double
// evaluation (error-free sums and products of Knuth and Dekker): the angle
// 2 pi j / M of a length that is no power of two is itself rounded, and with the
// angle and the series in plain FP64 the values were up to two units off, the
// cos of 2 pi / 3 among them.  For compile time only: a fused multiply-add would
// spoil the error-free sums.
struct DD {
  double h, l;
};
constexpr DD dd_sum(double a, double b) {
  const double s = a + b, bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
constexpr DD dd_prod(double a, double b) {
  const double p = a * b, ca = 134217729.0 * a, cb = 134217729.0 * b;   // halves of 26 bits
  const double ah = ca - (ca - a), bh = cb - (cb - b), al = a - ah, bl = b - bh;
  return {p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr DD operator+(DD a, DD b) {
  const DD s = dd_sum(a.h, b.h);
  return dd_sum(s.h, s.l + (a.l + b.l));
}
constexpr DD operator*(DD a, DD b) {
  const DD p = dd_prod(a.h, b.h);
  return dd_sum(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr DD operator/(DD a, double n) {
  const double q = a.h / n;
  const DD p = dd_prod(q, n);
  return dd_sum(q, ((a.h - p.h) - p.l + a.l) / n);
}
constexpr CosSin precise_cos_sin(long long j, long long M) {
  const long long jm = ((j % M) + M) % M, m8 = M / 8, oct = jm / m8, rem = jm % m8;
  const DD two_pi = {6.283185307179586, 2.4492935982947064e-16};
  double c[2] = {0, 0}, s[2] = {0, 0};   // of rem and of m8 - rem, both in [0, pi/4]
  for (int v = 0; v < 2; ++v) {
    const DD x = two_pi * DD{double(v == 0 ? rem : m8 - rem), 0.0} / double(M), x2 = x * x;
    DD tc = {1.0, 0.0}, ts = x, sc = tc, ss = x;
    for (int i = 1; i < 15; ++i) {
      tc = tc * x2 / double(-(2 * i - 1) * (2 * i));
      ts = ts * x2 / double(-(2 * i) * (2 * i + 1));
      sc = sc + tc;
      ss = ss + ts;
    }
    c[v] = sc.h;
    s[v] = ss.h;
  }
  switch (oct) {
    case 0: return {c[0], s[0]};
    case 1: return {s[1], c[1]};
    case 2: return {-s[0], c[0]};
    case 3: return {-c[1], s[1]};
    case 4: return {-c[0], -s[0]};
    case 5: return {-s[1], -c[1]};
    case 6: return {s[0], -c[0]};
    default: return {c[1], -s[1]};
  }
}

// cos/sin of 2 pi j / R as a compile-time constant of type T (paired FP32
// specialises it in dfloat.cuh).
template <int R, class T>
struct TwR {
  static constexpr T c(int j) { return T(precise_cos_sin(8LL * j, 8LL * R).c); }
  static constexpr T s(int j) { return T(precise_cos_sin(8LL * j, 8LL * R).s); }
};

template <int R>
struct TwTab {
  double c[R], s[R];
};
template <int R>
constexpr TwTab<R> make_twtab() {
  TwTab<R> t{};
  for (int j = 0; j < R; ++j) {
    const CosSin v = precise_cos_sin(8LL * j, 8LL * R);
    t.c[j] = v.c;
    t.s[j] = v.s;
  }
  return t;
}

// a + s t and m + SIGN i n (a quarter turn folded into the sums).
template <class T>
__device__ __forceinline__ cpx<T> axpy_r(T s, cpx<T> t, cpx<T> a) { return {a.x + s * t.x, a.y + s * t.y}; }
template <int SIGN, class T>
__device__ __forceinline__ cpx<T> add_i(cpx<T> m, cpx<T> n) {
  return SIGN > 0 ? cpx<T>{m.x - n.y, m.y + n.x} : cpx<T>{m.x + n.y, m.y - n.x};
}

// Paired FP32 renormalises (settle, dfloat.cuh; nothing in the other
// arithmetics) the sums that go into a product here, the outputs of the
// P-point transforms in dft_pfa and those of the first radix-4 stage of a
// 16-point transform: a pair then goes through no more additions between two
// renormalisations than in a radix-8 stage.  Error against 64 bits of a
// convolution alone, root mean square of 24 media, without and with them: 10.0
// and 9.1e-15 at n = 72, 10.2 and 9.4 at n = 144, 10.2 and 9.6 at n = 200, 10.4
// and 9.4 at n = 280.  (It falls with the padding: at 256 points 6.5 at n = 68,
// 7.8 at n = 100, 9.5 at n = 128.)  Cost: operator at n = 144 0.89 -> 0.95 ms,
// n = 200 2.80 -> 2.94, n = 400 22.3 both.
template <int SIGN, class T>
__device__ __forceinline__ void dft3(cpx<T>& a, cpx<T>& b, cpx<T>& c) {
  constexpr T half = TwR<3, T>::c(1), sn = TwR<3, T>::s(1);   // cos = -1/2
  const cpx<T> t = settle(b + c), d = settle(b - c);
  const cpx<T> m = axpy_r(half, t, a);
  a = a + t;
  if constexpr (std::is_floating_point<T>::value) {   // m +- i s d with the products fused into the sums
    constexpr T s = SIGN > 0 ? sn : -sn;
    b = {m.x - s * d.y, m.y + s * d.x};
    c = {m.x + s * d.y, m.y - s * d.x};
  } else {
    const cpx<T> n = {sn * d.x, sn * d.y};
    b = add_i<SIGN>(m, n);
    c = add_i<-SIGN>(m, n);
  }
}

template <int SIGN, class T>
__device__ __forceinline__ void dft5(cpx<T>& a, cpx<T>& b, cpx<T>& c, cpx<T>& d, cpx<T>& e) {
  constexpr T c1 = TwR<5, T>::c(1), c2 = TwR<5, T>::c(2), s1 = TwR<5, T>::s(1), s2 = TwR<5, T>::s(2);
  const cpx<T> t1 = settle(b + e), t2 = settle(c + d), t3 = settle(b - e), t4 = settle(c - d);
  const cpx<T> m1 = axpy_r(c2, t2, axpy_r(c1, t1, a)), m2 = axpy_r(c1, t2, axpy_r(c2, t1, a));
  const cpx<T> n1 = axpy_r(s2, t4, cpx<T>{s1 * t3.x, s1 * t3.y});
  const cpx<T> n2 = axpy_r(-s1, t4, cpx<T>{s2 * t3.x, s2 * t3.y});
  a = a + (t1 + t2);
  b = add_i<SIGN>(m1, n1);
  e = add_i<-SIGN>(m1, n1);
  c = add_i<SIGN>(m2, n2);
  d = add_i<-SIGN>(m2, n2);
}

template <int R, int SIGN, bool HALF, class T>
__device__ __forceinline__ void dft(cpx<T> (&a)[R]);

// z * exp(SIGN 2 pi i j / R), j and R compile-time constants.
template <int R, int SIGN, class T>
__device__ __forceinline__ cpx<T> twR_mul(cpx<T> z, int j) {
  if (j == 0) return z;
  constexpr TwTab<R> t = make_twtab<R>();
  const T c = T(t.c[j]), s = T(t.s[j]);
  return cmul(z, cpx<T>{c, SIGN > 0 ? s : -s});
}

// Prime-factor form (Good 1958): with n = Q n1 + P n2 (mod R) and k read mod P
// and mod Q, w_R^(nk) = w_P^(n1 k) w_Q^(n2 k): P-point and Q-point transforms
// with no twiddles between them.
template <int R, int SIGN, class T>
__device__ __forceinline__ void dft_pfa(cpx<T> (&a)[R]) {
  constexpr int P = pow2_part(R), Q = R / P;
  static_assert(Q == 3 || Q == 5, "one odd factor, 3 or 5");
  cpx<T> t[Q][P];
#pragma unroll
  for (int n2 = 0; n2 < Q; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < P; ++n1) t[n2][n1] = a[(Q * n1 + P * n2) % R];
    if constexpr (P > 1) dft<P, SIGN, false>(t[n2]);
    if constexpr (P > 1 && !std::is_floating_point<T>::value) {
#pragma unroll
      for (int n1 = 0; n1 < P; ++n1) t[n2][n1] = settle(t[n2][n1]);
    }
  }
#pragma unroll
  for (int k = 0; k < P; ++k) {
    if constexpr (Q == 3) dft3<SIGN>(t[0][k], t[1][k], t[2][k]);
    else dft5<SIGN>(t[0][k], t[1][k], t[2][k], t[3][k], t[4][k]);
  }
#pragma unroll
  for (int k = 0; k < R; ++k) a[k] = t[k % Q][k % P];
}

// HALF for a composite R: the even outputs are the R/2-point transform of the
// nonzero half, the odd ones that of the half times w^j.
template <int R, int SIGN, class T>
__device__ __forceinline__ void dft_half_in(cpx<T> (&a)[R]) {
  constexpr int M = R / 2;
  cpx<T> e[M], o[M];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    e[j] = a[j];
    o[j] = twR_mul<R, SIGN>(a[j], j);
  }
  dft_pfa<M, SIGN>(e);
  dft_pfa<M, SIGN>(o);
#pragma unroll
  for (int k = 0; k < M; ++k) {
    a[2 * k] = e[k];
    a[2 * k + 1] = o[k];
  }
}

template <int R, int SIGN, bool HALF, class T>
__device__ __forceinline__ void dft(cpx<T> (&a)[R]) {
  if constexpr (!is_pow2(R)) {
    if constexpr (HALF) dft_half_in<R, SIGN>(a);
    else dft_pfa<R, SIGN>(a);
  } else if constexpr (R > 1 && R <= 8) {
    dft_radix2<R, SIGN, HALF>(a);
  } else if constexpr (R > 1) {
    bool first = true;
    int s = R / 2;
#pragma unroll
    for (; s >= 2; s /= 4) {
#pragma unroll
      for (int b = 0; b < R; b += 2 * s) {
#pragma unroll
        for (int j = 0; j < s / 2; ++j) {
          const int idx = j * (64 / (2 * s));   // w^j in 64ths of a turn
          const int h = s / 2;
          cpx<T> t0, t1, t2, t3;
          if (HALF && first) {
            t0 = a[b + j];
            t1 = a[b + j];
            t2 = a[b + j + h];
            t3 = mul_i<SIGN>(a[b + j + h]);
          } else {
            const cpx<T> x0 = a[b + j], x1 = a[b + j + h], x2 = a[b + j + s], x3 = a[b + j + 3 * h];
            t0 = x0 + x2;
            t1 = x0 - x2;
            t2 = x1 + x3;
            t3 = mul_i<SIGN>(x1 - x3);
          }
          a[b + j] = t0 + t2;
          a[b + j + h] = tw64_mul<SIGN>(t0 - t2, 2 * idx);
          a[b + j + s] = tw64_mul<SIGN>(t1 + t3, idx);
          a[b + j + 3 * h] = tw64_mul<SIGN>(t1 - t3, 3 * idx);
        }
      }
      first = false;
      // paired FP32: at most three halvings between renormalisations, as in a radix-8 stage
      if constexpr (!std::is_floating_point<T>::value) {
        if (s >= 4) {
#pragma unroll
          for (int i = 0; i < R; ++i) a[i] = settle(a[i]);
        }
      }
    }
    if (s == 1) {   // the last radix-2 stage (span 1: no twiddles)
#pragma unroll
      for (int b = 0; b < R; b += 2) {
        const cpx<T> u = a[b];
        if (HALF && first) {
          a[b + 1] = u;
        } else {
          const cpx<T> v = a[b + 1];
          a[b] = u + v;
          a[b + 1] = u - v;
        }
      }
    }
    cpx<T> t[R];
#pragma unroll
    for (int i = 0; i < R; ++i) t[i] = a[bitrev(i, R)];
#pragma unroll
    for (int i = 0; i < R; ++i) a[i] = t[i];
  }
}

// The same transform when only the outputs k < R/2 are used (the rows an
// inverse pass keeps).  A composite R combines two R/2-point transforms for
// those outputs alone; a power of two leaves the pruning to the compiler.
template <int R, int SIGN, class T>
__device__ __forceinline__ void dft_low(cpx<T> (&a)[R]) {
  if constexpr (is_pow2(R)) {
    dft<R, SIGN, false>(a);
  } else {
    constexpr int M = R / 2;
    cpx<T> e[M], o[M];
#pragma unroll
    for (int j = 0; j < M; ++j) {
      e[j] = a[2 * j];
      o[j] = a[2 * j + 1];
    }
    dft_pfa<M, SIGN>(e);
    dft_pfa<M, SIGN>(o);
#pragma unroll
    for (int j = 0; j < M; ++j) a[j] = e[j] + twR_mul<R, SIGN>(o[j], j);
  }
}

// Transform lengths with a factor 9 or 25, for grids whose power of two would
// be mostly padding (transform_length).  Every one is 8 r2 r3 (the stages of
// the shared-memory transforms, MixRad) and L1 L2 with L1 a multiple of an
// even L2 (the two register stages, Split).
constexpr bool is_mixed_len(int L) { return !is_pow2(L); }
template <int L> struct MixRad;
template <> struct MixRad<144> { static constexpr int r2 = 6, r3 = 3, L1 = 12; };
template <> struct MixRad<200> { static constexpr int r2 = 5, r3 = 5, L1 = 20; };
template <> struct MixRad<288> { static constexpr int r2 = 6, r3 = 6, L1 = 24; };
template <> struct MixRad<400> { static constexpr int r2 = 10, r3 = 5, L1 = 20; };
template <> struct MixRad<576> { static constexpr int r2 = 6, r3 = 12, L1 = 24; };
template <> struct MixRad<800> { static constexpr int r2 = 10, r3 = 10, L1 = 40; };

// Split of the padded length L = L1 * L2 into two in-register stages.
constexpr int ilog2(int v) { return v <= 1 ? 0 : 1 + ilog2(v >> 1); }
template <int L, bool MIXED = is_mixed_len(L)>
struct Split {
  static constexpr int lg = ilog2(L);
  static constexpr int L1 = 1 << ((lg + 1) / 2);
  static constexpr int L2 = L / L1;
};

template <int L>
struct Split<L, true> {
  static constexpr int L1 = MixRad<L>::L1;
  static constexpr int L2 = L / L1;
  static_assert(L1 % L2 == 0 && L2 % 2 == 0 && L % 8 == 0, "mixed transform length");
};

}  // namespace ori
