// Discrete Fourier transforms of one short column held in registers, with
// the sign of e^{+2 pi i n k / N} (both uses here -- states to real space and
// pair products to the response set -- have that sign).  N is a compile-time
// size with factors 2, 3 and 5; every index is a constant, so a column is N
// complex registers and the transform runs without shared memory, barriers or
// twiddle loads.  Coprime factors combine by the prime-factor map (no
// twiddles: 24 = 3 x 8 takes 264 real additions and multiply-adds, where the
// 13 outputs of a 24-point response column by direct sums take 1248), equal
// primes by Cooley-Tukey with constant twiddles.
// (I. J. Good, J. R. Stat. Soc. B 20, 361 (1958); J. W. Cooley and
// J. W. Tukey, Math. Comp. 19, 297 (1965).)
#pragma once

#include <cuda_runtime.h>

#include <type_traits>
#include <utility>

namespace chi0 {
namespace fft {

template <int B, int E, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(std::forward<F>(f));
  }
}

// cos and sin of 2 pi p / q at compile time: Taylor series after reduction to
// the first octant (remainder below 1e-20 there).
constexpr double series_sin(double x) {
  double t = x, s = x;
  for (int k = 1; k < 12; ++k) {
    t *= -x * x / ((2 * k) * (2 * k + 1));
    s += t;
  }
  return s;
}
constexpr double series_cos(double x) {
  double t = 1.0, s = 1.0;
  for (int k = 1; k < 12; ++k) {
    t *= -x * x / ((2 * k - 1) * (2 * k));
    s += t;
  }
  return s;
}
constexpr double kPi = 3.14159265358979323846264338327950288;
constexpr double cos_frac(int p, int q);
constexpr double sin_frac(int p, int q) {  // sin(2 pi p / q)
  p %= q;
  if (2 * p > q) return -sin_frac(q - p, q);                     // (pi, 2 pi)
  if (4 * p > q) return sin_frac(q - 2 * p, 2 * q);              // (pi/2, pi]: sin(pi - x)
  if (8 * p > q) return cos_frac(q - 4 * p, 4 * q);              // (pi/4, pi/2]: cos(pi/2 - x)
  return series_sin(2.0 * kPi * p / q);
}
constexpr double cos_frac(int p, int q) {
  p %= q;
  if (2 * p > q) return cos_frac(q - p, q);
  if (4 * p > q) return -cos_frac(q - 2 * p, 2 * q);
  if (8 * p > q) return sin_frac(q - 4 * p, 4 * q);
  return series_cos(2.0 * kPi * p / q);
}

template <typename C>
__device__ __forceinline__ C cadd(const C a, const C b) {
  C r;
  r.x = a.x + b.x;
  r.y = a.y + b.y;
  return r;
}
template <typename C>
__device__ __forceinline__ C csub(const C a, const C b) {
  C r;
  r.x = a.x - b.x;
  r.y = a.y - b.y;
  return r;
}
template <typename C>  // a + i b
__device__ __forceinline__ C cadd_i(const C a, const C b) {
  C r;
  r.x = a.x - b.y;
  r.y = a.y + b.x;
  return r;
}
template <typename C>  // a - i b
__device__ __forceinline__ C csub_i(const C a, const C b) {
  C r;
  r.x = a.x + b.y;
  r.y = a.y - b.x;
  return r;
}
template <typename C, typename T>  // a + s b, s real
__device__ __forceinline__ C cfma(const C a, const T s, const C b) {
  C r;
  r.x = fma(s, b.x, a.x);
  r.y = fma(s, b.y, a.y);
  return r;
}
template <typename C, typename T>  // a + i s b, s real
__device__ __forceinline__ C cfma_i(const C a, const T s, const C b) {
  C r;
  r.x = fma(-s, b.y, a.x);
  r.y = fma(s, b.x, a.y);
  return r;
}

// A constant of the transforms with the part that its rounding to T drops (0 in
// FP64).  In FP32 the few constants of a column act on every transition alike,
// so their rounding (up to 3e-8 each) would not average out: nine columns make
// up a rho, and the gain of a 24-point one is 1e-8 off with rounded constants,
// 1e-10 with these (extrapolar chi0 of N_G = 220 against 64 bits: 1.3e-7 -> 5e-8
// for 2% of its time).  sum() is c a + s b with one rounding of the rest.
template <typename T>
struct Const {
  T hi, lo;
  constexpr Const(double v) : hi((T)v), lo((T)(v - (double)(T)v)) {}
};
template <typename T>
__device__ __forceinline__ T times(const Const<T> c, const T a) {
  if constexpr (sizeof(T) == 4) return fma(c.hi, a, c.lo * a);
  else return c.hi * a;
}
template <typename T>
__device__ __forceinline__ T sum(const Const<T> c, const T a, const Const<T> s, const T b) {
  if constexpr (sizeof(T) == 4) return fma(c.hi, a, fma(s.hi, b, fma(c.lo, a, s.lo * b)));
  else return fma(c.hi, a, s.hi * b);
}

// a e^{2 pi i P / Q}
template <int P, int Q, typename C>
__device__ __forceinline__ C twiddle(const C a) {
  using T = decltype(a.x);
  constexpr int p = P % Q;
  C r;
  if constexpr (p == 0) {
    r = a;
  } else if constexpr (4 * p == Q) {
    r.x = -a.y;
    r.y = a.x;
  } else if constexpr (2 * p == Q) {
    r.x = -a.x;
    r.y = -a.y;
  } else if constexpr (4 * p == 3 * Q) {
    r.x = a.y;
    r.y = -a.x;
  } else if constexpr (sizeof(T) == 4 && 8 * p % Q == 0) {   // |cos| = |sin|
    constexpr Const<std::remove_const_t<T>> c(cos_frac(p, Q));
    constexpr bool same = 8 * p == Q || 8 * p == 5 * Q;
    r.x = times(c, same ? a.x - a.y : a.x + a.y);
    r.y = times(c, same ? a.y + a.x : a.y - a.x);
  } else {
    constexpr Const<std::remove_const_t<T>> c(cos_frac(p, Q)), s(sin_frac(p, Q)), ms(-sin_frac(p, Q));
    r.x = sum(c, a.x, ms, a.y);
    r.y = sum(c, a.y, s, a.x);
  }
  return r;
}

template <int N>
struct Split;  // N = R * M, and whether R and M are coprime
#define CHI0_FFT_SPLIT(n, r)                                        \
  template <>                                                       \
  struct Split<n> {                                                 \
    static constexpr int R = r, M = n / r;                          \
  }
CHI0_FFT_SPLIT(6, 2);
CHI0_FFT_SPLIT(8, 2);
CHI0_FFT_SPLIT(9, 3);
CHI0_FFT_SPLIT(10, 2);
CHI0_FFT_SPLIT(12, 3);
CHI0_FFT_SPLIT(15, 3);
CHI0_FFT_SPLIT(16, 4);
CHI0_FFT_SPLIT(18, 2);
CHI0_FFT_SPLIT(20, 4);
CHI0_FFT_SPLIT(24, 3);
CHI0_FFT_SPLIT(30, 5);
CHI0_FFT_SPLIT(32, 4);
CHI0_FFT_SPLIT(36, 4);
#undef CHI0_FFT_SPLIT

constexpr int gcd(int a, int b) { return b == 0 ? a : gcd(b, a % b); }
constexpr int inverse_mod(int a, int m) {
  for (int x = 1; x < m; ++x)
    if ((a % m) * x % m == 1) return x;
  return 0;
}

// a[k] <- sum_n a[n] e^{2 pi i n k / N}, natural order in and out
template <int N, typename C>
__device__ __forceinline__ void column(C (&a)[N]) {
  using T = std::remove_const_t<decltype(a[0].x)>;
  if constexpr (N == 1) {
  } else if constexpr (N == 2) {
    const C b = a[1];
    a[1] = csub(a[0], b);
    a[0] = cadd(a[0], b);
  } else if constexpr (N == 3) {
    constexpr Const<T> s(sin_frac(1, 3));
    const C t = cadd(a[1], a[2]), d = csub(a[1], a[2]);
    const C m = cfma(a[0], (T)-0.5, t);
    a[0] = cadd(a[0], t);
    if constexpr (sizeof(T) == 4) {
      C e;
      e.x = times(s, d.x);
      e.y = times(s, d.y);
      a[1] = cadd_i(m, e);
      a[2] = csub_i(m, e);
    } else {
      a[1] = cfma_i(m, s.hi, d);
      a[2] = cfma_i(m, -s.hi, d);
    }
  } else if constexpr (N == 4) {
    const C s02 = cadd(a[0], a[2]), d02 = csub(a[0], a[2]);
    const C s13 = cadd(a[1], a[3]), d13 = csub(a[1], a[3]);
    a[0] = cadd(s02, s13);
    a[1] = cadd_i(d02, d13);
    a[2] = csub(s02, s13);
    a[3] = csub_i(d02, d13);
  } else if constexpr (N == 5) {
    constexpr Const<T> c1(cos_frac(1, 5)), c2(cos_frac(2, 5));
    constexpr Const<T> s1(sin_frac(1, 5)), s2(sin_frac(2, 5)), ms1(-sin_frac(1, 5));
    const C t1 = cadd(a[1], a[4]), t2 = cadd(a[2], a[3]), d1 = csub(a[1], a[4]), d2 = csub(a[2], a[3]);
    C m1, m2, e1, e2;
    if constexpr (sizeof(T) == 4) {
      m1.x = a[0].x + sum(c1, t1.x, c2, t2.x);
      m1.y = a[0].y + sum(c1, t1.y, c2, t2.y);
      m2.x = a[0].x + sum(c2, t1.x, c1, t2.x);
      m2.y = a[0].y + sum(c2, t1.y, c1, t2.y);
    } else {
      m1 = cfma(cfma(a[0], c1.hi, t1), c2.hi, t2);
      m2 = cfma(cfma(a[0], c2.hi, t1), c1.hi, t2);
    }
    e1.x = sum(s1, d1.x, s2, d2.x);
    e1.y = sum(s1, d1.y, s2, d2.y);
    e2.x = sum(s2, d1.x, ms1, d2.x);
    e2.y = sum(s2, d1.y, ms1, d2.y);
    a[0] = cadd(a[0], cadd(t1, t2));
    a[1] = cadd_i(m1, e1);
    a[4] = csub_i(m1, e1);
    a[2] = cadd_i(m2, e2);
    a[3] = csub_i(m2, e2);
  } else {
    constexpr int R = Split<N>::R, M = Split<N>::M;
    constexpr bool coprime = gcd(R, M) == 1;
    // rows: coprime n = M n1 + R n2 (mod N); otherwise n = M n1 + n2
    C t[N];  // t[n2 * R + k1]
    static_for<0, M>([&](auto n2c) {
      constexpr int n2 = decltype(n2c)::value;
      C v[R];
      static_for<0, R>([&](auto n1c) {
        constexpr int n1 = decltype(n1c)::value;
        constexpr int n = coprime ? (M * n1 + R * n2) % N : M * n1 + n2;
        v[n1] = a[n];
      });
      column<R>(v);
      static_for<0, R>([&](auto k1c) {
        constexpr int k1 = decltype(k1c)::value;
        if constexpr (coprime)
          t[n2 * R + k1] = v[k1];
        else
          t[n2 * R + k1] = twiddle<n2 * k1, N>(v[k1]);
      });
    });
    static_for<0, R>([&](auto k1c) {
      constexpr int k1 = decltype(k1c)::value;
      C v[M];
      static_for<0, M>([&](auto n2c) {
        constexpr int n2 = decltype(n2c)::value;
        v[n2] = t[n2 * R + k1];
      });
      column<M>(v);
      static_for<0, M>([&](auto k2c) {
        constexpr int k2 = decltype(k2c)::value;
        // coprime: k = k1 mod R and k2 mod M; otherwise k = k1 + R k2
        constexpr int k = coprime ? (k1 * M * inverse_mod(M, R) + k2 * R * inverse_mod(R, M)) % N : k1 + R * k2;
        a[k] = v[k2];
      });
    });
  }
}

}  // namespace fft
}  // namespace chi0
