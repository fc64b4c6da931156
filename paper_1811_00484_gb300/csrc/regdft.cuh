// DFTs of 2 to 32 points held in one thread's registers, every index and every
// constant known at compile time.
//
// Composite lengths with coprime factors A, B use the prime-factor map
// (n = B n1 + A n2 mod AB, k by the Chinese remainder theorem: no twiddles,
// the permutations are register names); 9, 16, 25, 27 and 32 use the
// decimation n = B n1 + n2, k = k1 + A k2 with constant twiddles.  dft_half_in
// and dft_half_out prune an even length for the matvec's zero padding (second
// half of the inputs zero) and crop (second half of the outputs unused): two
// half-length DFTs instead of one full-length one.
#pragma once

#include "fft.cuh"

namespace vie {

// cos and sin of 2 pi m / R (0 <= m < R), reduced to [0, pi/4] by exact integer
// symmetries and summed as Taylor series in double at compile time
struct UnitRoot {
  double c, s;
};
__host__ __device__ constexpr UnitRoot unit_root(int m, int R) {
  // work in units of 1/8 turn: angle = (8 m / R) octants
  m = ((m % R) + R) % R;
  const int oct = (8 * m) / R;                       // 0 .. 7
  const int rem = 8 * m - oct * R;                   // angle inside the octant: rem / R octants
  const int num = (oct & 1) ? R - rem : rem;         // distance from the nearest axis, in 1/R octants
  const double x = 0.78539816339744830962 * (double)num / (double)R;
  const double x2 = x * x;
  double c = 1.0, s = 1.0, t = 1.0;
  for (int i = 1; i < 12; ++i) {
    t *= -x2 / (double)((2 * i - 1) * (2 * i));
    c += t;
  }
  t = 1.0;
  for (int i = 1; i < 12; ++i) {
    t *= -x2 / (double)((2 * i) * (2 * i + 1));
    s += t;
  }
  s *= x;
  // axis nearest below (even octant: angle from axis oct/2) or above (odd octant)
  const int ax = ((oct + 1) / 2) & 3;                // nearest axis
  const double sg = (oct & 1) ? -s : s;              // signed offset from it
  if (ax == 0) return UnitRoot{c, sg};
  if (ax == 1) return UnitRoot{-sg, c};
  if (ax == 2) return UnitRoot{-c, -sg};
  return UnitRoot{sg, -c};
}

template <int I> struct Int {
  static constexpr int v = I;
};
template <int I, int N, typename F> __device__ __forceinline__ void unrolled_from(F&& f) {
  if constexpr (I < N) {
    f(Int<I>());
    unrolled_from<I + 1, N>(f);
  }
}
// f(Int<0>) ... f(Int<N-1>)
template <int N, typename F> __device__ __forceinline__ void unrolled(F&& f) { unrolled_from<0, N>(f); }

template <typename C> struct RealPart;
template <> struct RealPart<float2> { using type = float; };
template <> struct RealPart<double2> { using type = double; };

// v exp(-2 pi i M / R) (forward) or its conjugate (INV)
template <int M0, int R, bool INV, typename C> __device__ __forceinline__ C mul_root(C v) {
  using T = typename RealPart<C>::type;
  constexpr int M = ((M0 % R) + R) % R;
  if constexpr (M == 0) {
    return v;
  } else if constexpr (2 * M == R) {
    return mk(-v.x, -v.y);
  } else if constexpr (4 * M == R) {
    return INV ? mul_i(v) : mul_mi(v);
  } else if constexpr (4 * M == 3 * R) {
    return INV ? mul_mi(v) : mul_i(v);
  } else if constexpr (8 * M == R || 8 * M == 3 * R || 8 * M == 5 * R || 8 * M == 7 * R) {
    constexpr UnitRoot u = unit_root(M, R);
    constexpr T r = (T)0.70710678118654752440;
    constexpr bool cp = u.c > 0, sp = (INV ? u.s : -u.s) > 0;      // signs of the factor's parts
    const T p = cp ? v.x : -v.x, q = cp ? v.y : -v.y;
    if constexpr (cp == sp) return mk(r * (p - q), r * (p + q));   // +-(1 + i)
    else return mk(r * (p + q), r * (q - p));                      // +-(1 - i)
  } else {
    constexpr UnitRoot u = unit_root(M, R);
    constexpr T c = (T)u.c, s = (T)(INV ? u.s : -u.s);
    return mk(v.x * c - v.y * s, v.x * s + v.y * c);
  }
}

__host__ __device__ constexpr int inverse_mod(int a, int m) {
  for (int i = 1; i < m; ++i)
    if ((a % m) * i % m == 1) return i;
  return m == 1 ? 0 : 1;
}

template <int R> struct Split;                         // R = A B; kPfa: coprime map
#define VIE_SPLIT(R, X, Y, P) \
  template <> struct Split<R> { static constexpr int A = X, B = Y; static constexpr bool kPfa = P; }
VIE_SPLIT(6, 2, 3, true);
VIE_SPLIT(9, 3, 3, false);
VIE_SPLIT(10, 2, 5, true);
VIE_SPLIT(12, 4, 3, true);
VIE_SPLIT(14, 2, 7, true);
VIE_SPLIT(15, 3, 5, true);
VIE_SPLIT(16, 4, 4, false);
VIE_SPLIT(18, 2, 9, true);
VIE_SPLIT(20, 4, 5, true);
VIE_SPLIT(21, 3, 7, true);
VIE_SPLIT(24, 8, 3, true);
VIE_SPLIT(25, 5, 5, false);
VIE_SPLIT(27, 3, 9, false);
VIE_SPLIT(28, 4, 7, true);
VIE_SPLIT(32, 4, 8, false);
#undef VIE_SPLIT

// in-place DFT of v[0..R), natural order in and out
template <int R, bool INV, typename C> __device__ __forceinline__ void dft_reg(C (&v)[R]) {
  using T = typename RealPart<C>::type;
  if constexpr (R == 1) {
  } else if constexpr (R == 2) {
    dft2(v);
  } else if constexpr (R == 3) {
    dft3<C, T>(v, INV);
  } else if constexpr (R == 4) {
    dft4(v[0], v[1], v[2], v[3], INV);
  } else if constexpr (R == 5) {
    dft5<C, T>(v, INV);
  } else if constexpr (R == 7) {
    // sums and differences of mirrored inputs, real coefficients
    C p[3], m[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      p[j] = v[j + 1] + v[6 - j];
      m[j] = v[j + 1] - v[6 - j];
    }
    const C x0 = v[0];
    v[0] = x0 + (p[0] + p[1] + p[2]);
    unrolled<3>([&](auto ik) {
      constexpr int k = decltype(ik)::v + 1;
      C a = x0, b = mk((T)0, (T)0);
      unrolled<3>([&](auto ij) {
        constexpr int j = decltype(ij)::v;
        constexpr UnitRoot u = unit_root((j + 1) * k, 7);
        constexpr T c = (T)u.c, s = (T)u.s;
        a.x = fma(c, p[j].x, a.x);
        a.y = fma(c, p[j].y, a.y);
        if constexpr (j == 0) {
          b = mk(s * m[0].x, s * m[0].y);
        } else {
          b.x = fma(s, m[j].x, b.x);
          b.y = fma(s, m[j].y, b.y);
        }
      });
      const C ib = INV ? mul_i(b) : mul_mi(b);
      v[k] = a + ib;
      v[7 - k] = a - ib;
    });
  } else if constexpr (R == 8) {
    dft8<C, T>(v, INV);
  } else {
    constexpr int A = Split<R>::A, B = Split<R>::B;
    C w[R];
    unrolled<B>([&](auto in2) {
      constexpr int n2 = decltype(in2)::v;
      C t[A];
      unrolled<A>([&](auto in1) {
        constexpr int n1 = decltype(in1)::v;
        t[n1] = v[Split<R>::kPfa ? (B * n1 + A * n2) % R : B * n1 + n2];
      });
      dft_reg<A, INV>(t);
      unrolled<A>([&](auto ik1) {
        constexpr int k1 = decltype(ik1)::v;
        w[n2 * A + k1] = Split<R>::kPfa ? t[k1] : mul_root<n2 * k1, R, INV>(t[k1]);
      });
    });
    unrolled<A>([&](auto ik1) {
      constexpr int k1 = decltype(ik1)::v;
      C t[B];
      unrolled<B>([&](auto in2) { t[decltype(in2)::v] = w[decltype(in2)::v * A + k1]; });
      dft_reg<B, INV>(t);
      unrolled<B>([&](auto ik2) {
        constexpr int k2 = decltype(ik2)::v;
        constexpr int k = Split<R>::kPfa
                              ? (k1 * B * inverse_mod(B, A) + k2 * A * inverse_mod(A, B)) % R
                              : k1 + A * k2;
        v[k] = t[k2];
      });
    });
  }
}

// DFT of (x[0..R/2), 0, ..., 0), R even: X[2k] from x, X[2k+1] from x_m w_R^m
template <int R, bool INV, typename C>
__device__ __forceinline__ void dft_half_in(const C (&x)[R / 2], C (&X)[R]) {
  constexpr int M = R / 2;
  C e[M], o[M];
  unrolled<M>([&](auto im) {
    constexpr int m = decltype(im)::v;
    e[m] = x[m];
    o[m] = mul_root<m, R, INV>(x[m]);
  });
  dft_reg<M, INV>(e);
  dft_reg<M, INV>(o);
#pragma unroll
  for (int k = 0; k < M; ++k) {
    X[2 * k] = e[k];
    X[2 * k + 1] = o[k];
  }
}

// outputs 0 .. R/2 - 1 of the DFT of X, R even
template <int R, bool INV, typename C>
__device__ __forceinline__ void dft_half_out(const C (&X)[R], C (&x)[R / 2]) {
  constexpr int M = R / 2;
  C e[M], o[M];
#pragma unroll
  for (int k = 0; k < M; ++k) {
    e[k] = X[2 * k];
    o[k] = X[2 * k + 1];
  }
  dft_reg<M, INV>(e);
  dft_reg<M, INV>(o);
  unrolled<M>([&](auto im) {
    constexpr int m = decltype(im)::v;
    x[m] = e[m] + mul_root<m, R, INV>(o[m]);
  });
}

}  // namespace vie
