// FFTs of whole lines held in one thread's registers, for line lengths known at compile time.
//
// A line of N = N1 N2 points sits in v[N].  forward() transforms it in place and leaves frequency
// LinePlan<N>::freq(p) at position p; inverse() takes that order back to v[n] = x(n) (unnormalised).
// Coprime factors use the prime-factor index maps (no twiddles between the two stages), others the
// Cooley-Tukey form with compile-time twiddles.  Every index and every root of unity is a constant of
// the instantiation, so a transform is straight-line arithmetic: no shared memory, no table loads, no
// index instructions.  Short transforms (radix 6 to 16) are built the same way from radix 2, 3, 4, 5
// and 8.
#pragma once

#include <utility>

#include "fft.cuh"
#include "packed.cuh"

namespace pt {
namespace rl {

template <class F, int... I>
__device__ __forceinline__ void sfor_impl(F&& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
// f(integral_constant<0>), ..., f(integral_constant<E - 1>)
template <int E, class F>
__device__ __forceinline__ void sfor(F&& f) {
  sfor_impl(f, std::make_integer_sequence<int, E>{});
}

// sine and cosine of |x| <= pi/4 by their power series (host, at compile time)
constexpr double series_sin(double x) {
  double t = x, s = x;
  for (int k = 1; k < 14; ++k) {
    t *= -x * x / double((2 * k) * (2 * k + 1));
    s += t;
  }
  return s;
}
constexpr double series_cos(double x) {
  double t = 1.0, s = 1.0;
  for (int k = 1; k < 14; ++k) {
    t *= -x * x / double((2 * k - 1) * (2 * k));
    s += t;
  }
  return s;
}

struct Root {
  double re, im;
};
// exp(-2 pi i k / n), reduced to an octant so that symmetric roots have equal components
constexpr Root root(int k, int n) {
  constexpr double half_pi = 1.57079632679489661923;
  k %= n;
  const int q = 4 * k / n, r = 4 * k - q * n;  // angle = (q + r / n) pi/2
  const bool far = 2 * r > n;
  const double a = half_pi * double(far ? n - r : r) / double(n);
  const double c = far ? series_sin(a) : series_cos(a), s = far ? series_cos(a) : series_sin(a);
  return q == 0 ? Root{c, -s} : q == 1 ? Root{-s, -c} : q == 2 ? Root{-c, s} : Root{s, c};
}

// a * exp(-+2 pi i K / N)
template <int K, int N, bool INV, class T>
__device__ __forceinline__ cx<T> twiddle(cx<T> a) {
  constexpr int k = K % N;
  if constexpr (k == 0) {
    return a;
  } else if constexpr (4 * k == N) {
    return rot90<INV>(a);
  } else if constexpr (2 * k == N) {
    return cx<T>{-a.re, -a.im};
  } else if constexpr (4 * k == 3 * N) {
    return rot90<!INV>(a);
  } else if constexpr ((8 * k) % N == 0) {
    constexpr Root w = root(k, N);
    constexpr double r = 0.70710678118654752440;
    // (+-1 +- i)/sqrt 2: the sum or difference of the components, scaled once each
    constexpr bool pr = w.re > 0, pi = (w.im > 0) != INV;
    const T p = a.re + a.im, m = a.re - a.im;
    // (x + i y)(sr + i si): re = sr x - si y, im = si x + sr y
    const T re = pr ? (pi ? m : p) : (pi ? -p : -m);
    const T im = pr ? (pi ? p : -m) : (pi ? m : -p);
    return cx<T>{re * T(r), im * T(r)};
  } else {
    constexpr Root w = root(k, N);
    constexpr T c = T(w.re), s = T(INV ? -w.im : w.im);
    return cx<T>{a.re * c - a.im * s, a.re * s + a.im * c};
  }
}

// p + rot90(q) and p - rot90(q)
template <bool INV, class T>
__device__ __forceinline__ void cross(cx<T> p, cx<T> q, cx<T>& a, cx<T>& b) {
  const cx<T> r = rot90<INV>(q);
  a = p + r;
  b = p - r;
}
// p + rot90(q) h and p - rot90(q) h
template <bool INV, class T>
__device__ __forceinline__ void cross(cx<T> p, cx<T> q, T h, cx<T>& a, cx<T>& b) {
  const T s = INV ? h : -h;
  a = cx<T>{fma(-s, q.im, p.re), fma(s, q.re, p.im)};
  b = cx<T>{fma(s, q.im, p.re), fma(-s, q.re, p.im)};
}
template <bool INV, class T>
__device__ __forceinline__ void pdft4(cx<T>& a0, cx<T>& a1, cx<T>& a2, cx<T>& a3) {
  const cx<T> s0 = padd(a0, a2), s1 = psub(a0, a2), s2 = padd(a1, a3), s3 = psub(a1, a3);
  a0 = padd(s0, s2);
  a2 = psub(s0, s2);
  cross<INV>(s1, s3, a1, a3);
}
// the DFTs of fft.cuh with packed (FP32) and fused operations
template <int R, bool INV, class T>
__device__ __forceinline__ void pdft(cx<T>* a) {
  if constexpr (R == 2) {
    const cx<T> t = psub(a[0], a[1]);
    a[0] = padd(a[0], a[1]);
    a[1] = t;
  } else if constexpr (R == 3) {
    const cx<T> s = padd(a[1], a[2]), d = psub(a[1], a[2]), t = pfma(s, T(-0.5), a[0]);
    a[0] = padd(a[0], s);
    cross<INV>(t, d, T(0.86602540378443864676), a[1], a[2]);
  } else if constexpr (R == 4) {
    pdft4<INV>(a[0], a[1], a[2], a[3]);
  } else if constexpr (R == 5) {
    constexpr T c1 = T(0.30901699437494742410), c2 = T(-0.80901699437494742410);
    constexpr T s1 = T(0.95105651629515357212), s2 = T(0.58778525229247312917);
    const cx<T> t1 = padd(a[1], a[4]), t2 = padd(a[2], a[3]), d1 = psub(a[1], a[4]), d2 = psub(a[2], a[3]);
    const cx<T> b1 = pfma(t2, c2, pfma(t1, c1, a[0])), b2 = pfma(t2, c1, pfma(t1, c2, a[0]));
    const cx<T> e1 = pfma(d2, s2, pmul(d1, s1)), e2 = pfma(d2, -s1, pmul(d1, s2));
    a[0] = padd(padd(a[0], t1), t2);
    cross<INV>(b1, e1, a[1], a[4]);
    cross<INV>(b2, e2, a[2], a[3]);
  } else {
    constexpr T r = T(0.70710678118654752440);
    cx<T> e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6], o0 = a[1], o1 = a[3], o2 = a[5], o3 = a[7];
    pdft4<INV>(e0, e1, e2, e3);
    pdft4<INV>(o0, o1, o2, o3);
    const cx<T> p1 = o1 + rot90<INV>(o1), p3 = rot90<INV>(o3) - o3;
    a[0] = padd(e0, o0);
    a[4] = psub(e0, o0);
    a[1] = pfma(p1, r, e1);
    a[5] = pfma(p1, -r, e1);
    cross<INV>(e2, o2, a[2], a[6]);
    a[3] = pfma(p3, r, e3);
    a[7] = pfma(p3, -r, e3);
  }
}

constexpr int gcd(int a, int b) { return b ? gcd(b, a % b) : a; }
// a^{-1} mod m (1 if m == 1)
constexpr int inv_mod(int a, int m) {
  for (int x = 1; x < m; ++x)
    if ((a * x) % m == 1) return x;
  return 0;
}

// index maps of N = N1 N2: position of input (n1, n2) and output frequency of (k1, k2)
template <int N1, int N2>
struct Pair {
  static constexpr int N = N1 * N2;
  static constexpr bool pfa = gcd(N1, N2) == 1;
  static constexpr int pos(int n1, int n2) { return pfa ? (N2 * n1 + N1 * n2) % N : n1 * N2 + n2; }
  static constexpr int freq(int k1, int k2) {
    return pfa ? (N2 * inv_mod(N2 % N1, N1) * k1 + N1 * inv_mod(N1 % N2, N2) * k2) % N : k1 + N1 * k2;
  }
};

template <int R, bool INV, class T>
__device__ __forceinline__ void short_dft(cx<T>* a);

// DFT of length N1 N2 of a[], input and output in natural order
template <int N1, int N2, bool INV, class T>
__device__ __forceinline__ void pair_dft(cx<T>* a) {
  using P = Pair<N1, N2>;
  cx<T> b[P::N];
  sfor<N2>([&](auto n2) {
    cx<T> t[N1];
    sfor<N1>([&](auto n1) { t[n1] = a[P::pos(n1, n2)]; });
    short_dft<N1, INV>(t);
    sfor<N1>([&](auto k1) {
      constexpr int e = P::pfa ? 0 : int(k1) * int(n2);
      b[k1 * N2 + n2] = twiddle<e, P::N, INV>(t[k1]);
    });
  });
  sfor<N1>([&](auto k1) {
    cx<T> t[N2];
    sfor<N2>([&](auto n2) { t[n2] = b[k1 * N2 + n2]; });
    short_dft<N2, INV>(t);
    sfor<N2>([&](auto k2) { a[P::freq(k1, k2)] = t[k2]; });
  });
}

template <int R, bool INV, class T>
__device__ __forceinline__ void short_dft(cx<T>* a) {
  if constexpr (R == 1) return;
  else if constexpr (R == 6) pair_dft<2, 3, INV>(a);
  else if constexpr (R == 9) pair_dft<3, 3, INV>(a);
  else if constexpr (R == 10) pair_dft<2, 5, INV>(a);
  else if constexpr (R == 12) pair_dft<3, 4, INV>(a);
  else if constexpr (R == 16) pair_dft<4, 4, INV>(a);
  else pdft<R, INV>(a);
}

// the split of a line length: the shorter factor first, coprime where the length allows it
constexpr int first_factor(int n) {
  return n == 18 ? 2 : n == 25 ? 5 : n == 27 ? 3 : n == 45 ? 5 : n == 50 ? 5 : n == 16 ? 4 : n == 20 ? 4 : n == 24 ? 3 : n == 30 ? 5 : n == 32 ? 4 : n == 36 ? 4 : n == 40 ? 5
         : n == 48 ? 3 : n == 54 ? 6 : n == 60 ? 5 : n == 64 ? 8 : 0;
}

template <int N>
struct Line {
  static constexpr int N1 = first_factor(N), N2 = N / N1;
  using P = Pair<N1, N2>;
  // frequency at position p after forward()
  static constexpr int freq(int p) {
    for (int a = 0; a < N1; ++a)
      for (int b = 0; b < N2; ++b)
        if (P::pos(a, b) == p) return P::freq(a, b);
    return 0;
  }
  template <class T>
  static __device__ __forceinline__ void forward(cx<T>* v) {
    sfor<N2>([&](auto n2) {
      cx<T> t[N1];
      sfor<N1>([&](auto n1) { t[n1] = v[P::pos(n1, n2)]; });
      short_dft<N1, false>(t);
      sfor<N1>([&](auto k1) {
        constexpr int e = P::pfa ? 0 : int(k1) * int(n2);
        v[P::pos(k1, n2)] = twiddle<e, N, false>(t[k1]);
      });
    });
    sfor<N1>([&](auto k1) {
      cx<T> t[N2];
      sfor<N2>([&](auto n2) { t[n2] = v[P::pos(k1, n2)]; });
      short_dft<N2, false>(t);
      sfor<N2>([&](auto k2) { v[P::pos(k1, k2)] = t[k2]; });
    });
  }
  // the first stage of inverse(): what is left is one DFT of N1 points per n2 (inverse_group)
  template <class T>
  static __device__ __forceinline__ void inverse_first(cx<T>* v) {
    sfor<N1>([&](auto k1) {
      cx<T> t[N2];
      sfor<N2>([&](auto k2) { t[k2] = v[P::pos(k1, k2)]; });
      short_dft<N2, true>(t);
      sfor<N2>([&](auto n2) {
        constexpr int e = P::pfa ? 0 : int(k1) * int(n2);
        v[P::pos(k1, n2)] = twiddle<e, N, true>(t[n2]);
      });
    });
  }
  // the points P::pos(n1, n2), n1 < N1, of the inverse transform
  template <int n2, class T>
  static __device__ __forceinline__ void inverse_group(const cx<T>* v, cx<T>* t) {
    sfor<N1>([&](auto k1) { t[k1] = v[P::pos(k1, n2)]; });
    short_dft<N1, true>(t);
  }
  template <class T>
  static __device__ __forceinline__ void inverse(cx<T>* v) {
    inverse_first(v);
    sfor<N2>([&](auto n2) {
      cx<T> t[N1];
      inverse_group<int(n2)>(v, t);
      sfor<N1>([&](auto n1) { v[P::pos(n1, n2)] = t[n1]; });
    });
  }
};

}  // namespace rl
}  // namespace pt
