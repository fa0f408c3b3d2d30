// dft_small.cuh - forward DFTs of 1 to 32 points held in registers.
//
// 2, 4, 8: dft_reg (fft_core.cuh); 16 and 32: 4 x 4 and 4 x 8.  Odd primes: the symmetric form
//   X_q, X_(p-q) = (v_0 + sum_m cos(2 pi q m / p) s_m) -+ i sum_m sin(2 pi q m / p) d_m,
//   s_m, d_m = v_m +- v_(p-m), 1 <= m <= (p - 1) / 2.
// Products of coprime factors A B: Good's prime-factor mapping
//   n = B n1 + A n2, k = B (B^-1 mod A) k1 + A (A^-1 mod B) k2  (mod A B),
// which needs no twiddles; the other products: Cooley-Tukey.  The roots are formed at
// compile time in float64 from the Taylor series on [0, pi/4] and rounded once.
#pragma once

#include <type_traits>

#include "fft_core.cuh"

namespace shl {
namespace gen {

// f(integral_constant<int, i>) for i = LO .. HI - 1: loop bodies whose index is a
// constant expression, so that the roots below are immediates.
template <int LO, int HI, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (LO < HI) {
    f(std::integral_constant<int, LO>{});
    static_for<LO + 1, HI>(f);
  }
}

constexpr double TWO_PI = 6.283185307179586476925286766559;

constexpr double series_cos(double x) {
  double t = 1.0, s = 1.0;
  for (int i = 1; i <= 10; ++i) {
    t *= -x * x / ((2.0 * i - 1.0) * (2.0 * i));
    s += t;
  }
  return s;
}
constexpr double series_sin(double x) {
  double t = x, s = x;
  for (int i = 1; i <= 10; ++i) {
    t *= -x * x / ((2.0 * i) * (2.0 * i + 1.0));
    s += t;
  }
  return s;
}
// cos(2 pi k / n), the angle reduced to [0, pi/4] in integers first
constexpr double cos_turn(long long k, long long n) {
  k = ((k % n) + n) % n;
  if (2 * k > n) k = n - k;
  if (4 * k > n) return -cos_turn(n - 2 * k, 2 * n);
  if (8 * k > n) return series_sin(TWO_PI * (double)(n - 4 * k) / (double)(4 * n));
  return series_cos(TWO_PI * (double)k / (double)n);
}
constexpr double sin_turn(long long k, long long n) { return cos_turn(4 * k - n, 4 * n); }

constexpr int pow2_part(int r) { return r % 2 ? 1 : 2 * pow2_part(r / 2); }
constexpr bool is_prime(int r) {
  for (int f = 2; f * f <= r; ++f)
    if (r % f == 0) return false;
  return r > 1;
}
constexpr int smallest_factor(int r) {
  for (int f = 2; f * f <= r; ++f)
    if (r % f == 0) return f;
  return r;
}
// First factor of the split of a composite R that is no power of two.
constexpr int split_factor(int r) {
  if (r % 2 == 0) return pow2_part(r);
  const int p = smallest_factor(r);
  int a = p;
  while ((r / a) % p == 0 && r / a > p) a *= p;      // 27 = 9 * 3; 9 and 25: p * p
  return a;
}
constexpr int gcd_of(int a, int b) { return b ? gcd_of(b, a % b) : a; }
constexpr int inverse_mod(int a, int m) {
  for (int x = 1; x < m; ++x)
    if (a * x % m == 1) return x;
  return 0;
}

template <int R>
__device__ __forceinline__ void dft_n(float2 (&v)[R]);

template <int R>
__device__ __forceinline__ void dft_prime(float2 (&v)[R]) {
  constexpr int H = (R - 1) / 2;
  float2 s[H], d[H];
#pragma unroll
  for (int m = 1; m <= H; ++m) {
    s[m - 1] = caddp(v[m], v[R - m]);
    d[m - 1] = csubp(v[m], v[R - m]);
  }
  const float2 v0 = v[0];
#pragma unroll
  for (int m = 0; m < H; ++m) v[0] = caddp(v[0], s[m]);
  static_for<1, H + 1>([&](auto qi) {
    constexpr int q = decltype(qi)::value;
    float2 a = v0, b = make_float2(0.f, 0.f);
    static_for<1, H + 1>([&](auto mi) {
      constexpr int m = decltype(mi)::value;
      constexpr float c = (float)cos_turn(q * m, R), w = (float)sin_turn(q * m, R);
      a.x = fmaf(c, s[m - 1].x, a.x);
      a.y = fmaf(c, s[m - 1].y, a.y);
      b.x = m == 1 ? w * d[0].x : fmaf(w, d[m - 1].x, b.x);
      b.y = m == 1 ? w * d[0].y : fmaf(w, d[m - 1].y, b.y);
    });
    v[q] = make_float2(a.x + b.y, a.y - b.x);          // a - i b
    v[R - q] = make_float2(a.x - b.y, a.y + b.x);
  });
}

template <int R, int A>
__device__ __forceinline__ void dft_split(float2 (&v)[R]) {
  constexpr int B = R / A;
  constexpr bool COPRIME = gcd_of(A, B) == 1;
  constexpr int KA = COPRIME ? B * inverse_mod(B % A, A) % R : 1;
  constexpr int KB = COPRIME ? A * inverse_mod(A % B, B) % R : A;
  float2 t[A][B];
  static_for<0, B>([&](auto ni) {
    constexpr int n2 = decltype(ni)::value;
    float2 a[A];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) a[n1] = v[(B * n1 + (COPRIME ? A : 1) * n2) % R];
    dft_n<A>(a);
    static_for<0, A>([&](auto ki) {
      constexpr int k1 = decltype(ki)::value;
      if constexpr (!COPRIME && k1 * n2 != 0) {
        constexpr float c = (float)cos_turn(k1 * n2, R), s = (float)-sin_turn(k1 * n2, R);
        t[k1][n2] = make_float2(fmaf(a[k1].x, c, -a[k1].y * s), fmaf(a[k1].x, s, a[k1].y * c));
      } else {
        t[k1][n2] = a[k1];
      }
    });
  });
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    dft_n<B>(t[k1]);
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) v[(KA * k1 + KB * k2) % R] = t[k1][k2];
  }
}

// v[k] <- sum_n v[n] exp(-2 pi i n k / R), natural order in and out.
template <int R>
__device__ __forceinline__ void dft_n(float2 (&v)[R]) {
  if constexpr (R == 1) return;
  else if constexpr (R == 2 || R == 4 || R == 8) dft_reg<R, -1, true>(v);
  else if constexpr (pow2_part(R) == R) dft_split<R, 4>(v);
  else if constexpr (is_prime(R)) dft_prime<R>(v);
  else dft_split<R, split_factor(R)>(v);
}

}  // namespace gen
}  // namespace shl
