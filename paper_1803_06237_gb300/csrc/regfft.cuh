// Register-resident FFT of a compile-time length L (one line per thread).
//
// Same decimation-in-frequency Stockham scheme as fft.cuh, but every index is
// a compile-time constant: the L values live in registers, each stage is a
// fixed permutation with butterflies of radix 4, 2, 3 or 5 (greedy, in that
// order), and the twiddles exp(-2 pi i k / L) are compile-time constants (the
// table argument, tw[k] = exp(-2 pi i k / L), is no longer read).  No memory
// traffic, no barriers, no integer division.
#pragma once

#include <type_traits>

#include "fft.cuh"
#include "twiddle.cuh"

namespace vie {

__host__ __device__ constexpr int first_radix(int n) {
  return (n % 4 == 0) ? 4 : (n % 2 == 0) ? 2 : (n % 3 == 0) ? 3 : (n % 5 == 0) ? 5 : 0;
}

__host__ __device__ constexpr bool reg_fft_supported(int n) {
  return n == 1 ? true : (first_radix(n) == 0 ? false : reg_fft_supported(n / first_radix(n)));
}

// The stages multiply by the compile-time constants TwConst, so no twiddle is
// loaded and multiplications by 1 fold.

// compile-time loop: f(std::integral_constant<int, I>) for I in [B, E)
template <int B, int E, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(f);
  }
}

// The R-point DFT whose inputs from the NZ-th on are zero (the padding in a
// transform's first stage), without the sums with them: the compiler has to
// keep x + 0, which turns -0 into 0.
template <typename V, bool INV, int R, int NZ>
__device__ __forceinline__ void dft_lead(V* t) {
  if constexpr (NZ >= R) {
    dft_small<V, INV>(t, R);
  } else if constexpr (NZ <= 1) {
#pragma unroll
    for (int u = 1; u < R; ++u) t[u] = t[0];
  } else if constexpr (R == 3) {          // two inputs
    typedef typename real_of<V>::type T;
    const V x = t[0], y = t[1];
    V m, q;                               // x - y / 2, y sqrt(3) / 2 rotated
    m.x = x.x - T(0.5) * y.x;
    m.y = x.y - T(0.5) * y.y;
    const T s3 = RadixConst<T>::s3;
    q.x = INV ? -s3 * y.y : s3 * y.y;
    q.y = INV ? s3 * y.x : -s3 * y.x;
    t[0] = add(x, y);
    t[1] = add(m, q);
    t[2] = sub(m, q);
  } else if constexpr (R == 4 && NZ == 2) {
    const V x = t[0], y = t[1];
    V iy;
    iy.x = INV ? -y.y : y.y;
    iy.y = INV ? y.x : -y.x;
    t[0] = add(x, y);
    t[1] = add(x, iy);
    t[2] = sub(x, y);
    t[3] = sub(x, iy);
  } else if constexpr (R == 5 && NZ <= 3) {
    typedef typename real_of<V>::type T;
    const T c1 = RadixConst<T>::c51, c2 = RadixConst<T>::c52, s1 = RadixConst<T>::s51, s2 = RadixConst<T>::s52;
    const T g = INV ? T(-1) : T(1);
    const V x = t[0], y = t[1];
    V z;
    if constexpr (NZ == 3) z = t[2];
    else { z.x = 0; z.y = 0; }
    V m1, m2, i1, i2;
    if constexpr (NZ == 3) {
      m1.x = x.x + c1 * y.x + c2 * z.x; m1.y = x.y + c1 * y.y + c2 * z.y;
      m2.x = x.x + c2 * y.x + c1 * z.x; m2.y = x.y + c2 * y.y + c1 * z.y;
      i1.x = g * (s1 * y.y + s2 * z.y); i1.y = -g * (s1 * y.x + s2 * z.x);
      i2.x = g * (s2 * y.y - s1 * z.y); i2.y = -g * (s2 * y.x - s1 * z.x);
      t[0] = add(add(x, y), z);
    } else {
      m1.x = x.x + c1 * y.x; m1.y = x.y + c1 * y.y;
      m2.x = x.x + c2 * y.x; m2.y = x.y + c2 * y.y;
      i1.x = g * s1 * y.y; i1.y = -g * s1 * y.x;
      i2.x = g * s2 * y.y; i2.y = -g * s2 * y.x;
      t[0] = add(x, y);
    }
    t[1] = add(m1, i1);
    t[4] = sub(m1, i1);
    t[2] = add(m2, i2);
    t[3] = sub(m2, i2);
  } else {
    dft_small<V, INV>(t, R);
  }
}

// H: inputs of the transform from a[H] on are zero (they are not read in the
// first stage, the only one that H < L applies to).
template <typename V, bool INV, int L, int N, int S, int H = L>
struct RegStage {
  // N: current sub-length, S: product of the radices already applied
  static __device__ __forceinline__ void run(V (&a)[L], const V* __restrict__ tw) {
    constexpr int R = first_radix(N);
    static_assert(R != 0, "length must be 2^a 3^b 5^c");
    constexpr int M = N / R;
    V b[L];
    static_for<0, M>([&](auto pc) {
      constexpr int p = decltype(pc)::value;
      // inputs of this butterfly below H (first stage: S = 1)
      constexpr int NZ = H >= L ? R : (p >= H ? 0 : (H - 1 - p) / M + 1);
#pragma unroll
      for (int q = 0; q < S; ++q) {
        V t[R];
#pragma unroll
        for (int u = 0; u < R; ++u) t[u] = a[q + S * (p + u * M)];
        dft_lead<V, INV, R, (NZ < R ? NZ : R)>(t);
        b[q + S * (R * p)] = t[0];
        static_for<1, R>([&](auto uc) {
          constexpr int u = decltype(uc)::value;
          if constexpr (p == 0) {
            b[q + S * (R * p + u)] = t[u];
          } else {
            // w_L^(p u S), a compile-time constant
            typedef TwConst<L, p * u * S> W;
            typedef typename real_of<V>::type T;
            b[q + S * (R * p + u)] = mul_cs(t[u], (T)W::c, INV ? -(T)W::s : (T)W::s);
          }
        });
      }
    });
#pragma unroll
    for (int i = 0; i < L; ++i) a[i] = b[i];
    RegStage<V, INV, L, M, S * R>::run(a, tw);
  }
};

template <typename V, bool INV, int L, int S, int H>
struct RegStage<V, INV, L, 1, S, H> {
  static __device__ __forceinline__ void run(V (&)[L], const V* __restrict__) {}
};

// In-place transform of a[0..L): forward (exp(-i)) or inverse (exp(+i), no
// scaling).  H < L: a[H..L) are zero and are not added.
template <typename V, bool INV, int L, int H = L>
__device__ __forceinline__ void reg_fft(V (&a)[L], const V* __restrict__ tw) {
  RegStage<V, INV, L, L, 1, H>::run(a, tw);
}

// a[z] times exp(-/+ 2 pi i z / L), z < L / 2 (the odd frequencies' input, or
// the conjugate on their output)
template <typename V, bool INV, int L>
__device__ __forceinline__ void half_twiddle(V (&a)[L / 2]) {
  typedef typename real_of<V>::type T;
  static_for<1, L / 2>([&](auto zc) {
    constexpr int z = decltype(zc)::value;
    typedef TwConst<L, z> W;
    a[z] = mul_cs(a[z], (T)W::c, INV ? -(T)W::s : (T)W::s);
  });
}

}  // namespace vie
