// Larger radices of the line transforms, built from those of fft_fast.cuh: products of two coprime
// lengths by the prime-factor mapping (Good-Thomas, no twiddles), 9 = 3 x 3 by one Cooley-Tukey
// step.
#pragma once

#include "fft_fast.cuh"

namespace xfft {
namespace fast {

// length A B, A and B coprime: n = (B a + A b) mod A B, k = (B (B^-1 mod A) p + A (A^-1 mod B) q)
// mod A B, a two-dimensional A x B transform
template <typename C, int A, int B, bool INV>
struct DftCoprime {
  static constexpr int inverse(int x, int m) {
    int r = 1;
    while ((x * r) % m != 1 % m) ++r;
    return r;
  }
  __host__ __device__ __forceinline__ static void run(C* v) {
    constexpr int kA = B * inverse(B % A, A), kB = A * inverse(A % B, B);
    C t[A][B];
#pragma unroll
    for (int a = 0; a < A; ++a) {
#pragma unroll
      for (int b = 0; b < B; ++b) t[a][b] = v[(B * a + A * b) % (A * B)];
      Dft<C, B, INV>::run(t[a]);
    }
#pragma unroll
    for (int q = 0; q < B; ++q) {
      C c[A];
#pragma unroll
      for (int a = 0; a < A; ++a) c[a] = t[a][q];
      Dft<C, A, INV>::run(c);
#pragma unroll
      for (int p = 0; p < A; ++p) v[(kA * p + kB * q) % (A * B)] = c[p];
    }
  }
};

// length R R: inputs n = R a + b, outputs k = p + R q; cs, sn: cos and sin of 2 pi k / R^2
template <typename C, int R, bool INV>
struct DftSquare {
  template <typename T>
  __host__ __device__ __forceinline__ static void run(C* v, const T* cs, const T* sn) {
    C t[R][R];
#pragma unroll
    for (int b = 0; b < R; ++b) {
      C c[R];
#pragma unroll
      for (int a = 0; a < R; ++a) c[a] = v[R * a + b];
      Dft<C, R, INV>::run(c);
#pragma unroll
      for (int p = 0; p < R; ++p) {
        if (b > 0 && p > 0) {
          C w;
          w.x = cs[b * p];
          w.y = INV ? sn[b * p] : -sn[b * p];
          t[p][b] = cmul(c[p], w);
        } else {
          t[p][b] = c[p];
        }
      }
    }
#pragma unroll
    for (int p = 0; p < R; ++p) {
      Dft<C, R, INV>::run(t[p]);
#pragma unroll
      for (int q = 0; q < R; ++q) v[p + R * q] = t[p][q];
    }
  }
};

template <typename C, bool INV>
struct Dft<C, 9, INV> {
  __host__ __device__ __forceinline__ static void run(C* v) {
    typedef decltype(v[0].x) T;
    const T cs[5] = {
                     (T)1.0, (T)0.7660444431189780352, (T)0.17364817766693034885,
                     (T)-0.5, (T)-0.93969262078590838405};
    const T sn[5] = {
                     (T)0.0, (T)0.64278760968653932632, (T)0.98480775301220805937,
                     (T)0.86602540378443864676, (T)0.34202014332566873304};
    DftSquare<C, 3, INV>::run(v, cs, sn);
  }
};
template <typename C, bool INV>
struct Dft<C, 10, INV> : DftCoprime<C, 2, 5, INV> {};
template <typename C, bool INV>
struct Dft<C, 12, INV> : DftCoprime<C, 3, 4, INV> {};
template <typename C, bool INV>
struct Dft<C, 15, INV> : DftCoprime<C, 3, 5, INV> {};

}  // namespace fast
}  // namespace xfft
