// X-FFT preconditioner on grids of any supported size: five passes of line transforms with the
// factors of each length given at run time.
//
//   pass 1  z axis, real to complex (rows of n2 reals as n2 / 2 complex values), fused f -= alpha q
//   pass 2  y axis            pass 3  x axis, Green operator, x axis inverse
//   pass 4  y axis inverse    pass 5  z axis complex to real, fused f^T z partial sums
// Spectrum layout per right-hand side: [c][i][j][k2], k2 <= n2 / 2 contiguous, twice the transform.
//
// A length n = R1 RM RL (factors of at most 16, RM = 1 where two are the better choice: line_plan in
// fft.cu) is transformed by decimation
// in time in place: index (n1, m, l) = n1 RM RL + m RL + l; an R1-point DFT over n1 for every
// (m, l), twiddle W_n^(k1 (m RL + l)); an RM-point DFT over m, twiddle W_(RM RL)^(km l); an RL-point
// DFT over l; frequency k = k1 + R1 km + R1 RM kl.  The first DFT reads its inputs from global
// memory and the last one writes to it (lanes run over consecutive columns), so a line crosses
// shared memory once per factor after the first and needs one barrier there, and no reordering.
// In pass 3 a thread applies the Green operator to the outputs of its own last DFTs and runs the
// inverse of the same DFTs on the same places.
//
// What bounds it: FP64, the FP64 pipe (2 FMAs per SM and clock); FP32, memory traffic: fields
// and spectrum of one right-hand side are read and written once per pass.  The Green operator is a
// table of the inverses (9 reals per frequency, built once per grid): its factorisation, about 200
// operations and three square roots per frequency, costs more than the read.  Where a context has no
// room for the table, pass 3 forms the factorisation instead (whole call, with and without the table:
// FP64 256^3 8.3 and 12.0 ms, FP32 0.61 and 0.67 ms).
//
// Per right-hand side inside the solvers (enriched block included), against Stockham passes with
// compile-time plans where a length had one (256, 64) and run-time radix loops elsewhere:
//   FP32  256^3 1.30 -> 0.75 ms, 200 x 160 x 144 1.25 -> 0.27 ms, 90 x 120 x 100 0.276 -> 0.051 ms
//   FP64  64^3 0.139 -> 0.112 ms, 54 x 60 x 50 0.278 -> 0.118 ms
// The square FP32 planes of 32 to 128 nodes stay on the y-z plane path, three passes instead of five
// (128^3: 0.065 ms).
#pragma once

#include "fft_radix.cuh"
#include "xfft_kernels.h"

namespace xfft {

// factors of one axis; the z axis is planned for n2 / 2
struct LinePlan {
  int n, R1, RM, RL;
};

namespace lines {

using fast::cadd;
using fast::cmul;
using fast::cmulc;
using fast::csub;

template <typename T>
struct CplxOf;
template <>
struct CplxOf<double> {
  typedef double2 type;
};
template <>
struct CplxOf<float> {
  typedef float2 type;
};

constexpr int kLineThreads = 256;
// resident blocks per SM asked of the compiler: FP32 64 or 80 registers per thread (128 where a
// thread holds a second set of values in flight, HEAVY), FP64 128 or 255
template <typename T, int MR, bool HEAVY = false>
constexpr int min_blocks() {
  return sizeof(T) == 4 ? (HEAVY ? 2 : MR > 12 ? 3 : 4) : (MR > 12 ? 1 : 2);
}

template <int R>
struct Radix {
  static constexpr int v = R;
};
// f(Radix<R>()) for the run-time radix R <= MR (uniform over the block).  Kernels are instantiated
// for MR = 12 and 16: the largest radix decides their registers and so the warps in flight.
template <int MR, typename F>
__device__ __forceinline__ void with_radix(int R, const F& f) {
  if constexpr (MR > 12) {
    if (R == 15) {
      f(Radix<15>());
      return;
    }
    if (R == 16) {
      f(Radix<16>());
      return;
    }
  }
  switch (R) {
    case 1: f(Radix<1>()); break;
    case 2: f(Radix<2>()); break;
    case 3: f(Radix<3>()); break;
    case 4: f(Radix<4>()); break;
    case 5: f(Radix<5>()); break;
    case 6: f(Radix<6>()); break;
    case 8: f(Radix<8>()); break;
    case 9: f(Radix<9>()); break;
    case 10: f(Radix<10>()); break;
    default: f(Radix<12>()); break;
  }
}

template <bool INV, typename C>
__device__ __forceinline__ C twid(C a, C w) {
  return INV ? cmulc(a, w) : cmul(a, w);
}

// ---------------------------------------------------------------- column tiles (y and x axes)
// B = 2^lb columns of one line each in shared memory, buf[(position << lb) + column]; a thread
// keeps its column col = tid & (B - 1), and its lines' work items start at t0 with step nt.
// First factor: reads ld(n) for the line's elements n, writes the twiddled DFTs.
template <int MR, bool INV, typename C, typename LD>
__device__ __forceinline__ void first_factor(const LinePlan& p, C* buf, int lb, int col, int t0, int nt,
                                             const C* __restrict__ tw, const LD& ld) {
  const int NR = p.RM * p.RL;
  with_radix<MR>(p.R1, [&](auto rc) {
    constexpr int R = decltype(rc)::v;
    for (int j = t0; j < NR; j += nt) {
      C v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = ld(j + r * NR);
      fast::Dft<C, R, INV>::run(v);
#pragma unroll
      for (int r = 0; r < R; ++r) buf[((r * NR + j) << lb) + col] = r ? twid<INV>(v[r], __ldg(tw + r * j)) : v[0];
    }
  });
}
// middle factor, in place (forward order: DFT, then twiddle; the inverse of pass 3 runs the
// mirrored order, with the first factor's twiddle after its DFT)
template <int MR, bool INV, bool MIRROR, typename C>
__device__ __forceinline__ void mid_factor(const LinePlan& p, C* buf, int lb, int col, int t0, int nt,
                                           const C* __restrict__ tw) {
  const int NR = p.RM * p.RL;
  with_radix<MR>(p.RM, [&](auto rc) {
    constexpr int R = decltype(rc)::v;
    for (int w = t0; w < p.R1 * p.RL; w += nt) {
      const int k1 = w / p.RL, l = w - k1 * p.RL;
      C* b = buf + ((k1 * NR + l) << lb) + col;
      C v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = b[(r * p.RL) << lb];
      fast::Dft<C, R, INV>::run(v);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const C t = __ldg(tw + (MIRROR ? k1 * (r * p.RL + l) : r * l * p.R1));
        b[(r * p.RL) << lb] = twid<INV>(v[r], t);
      }
    }
  });
}

// ---------------------------------------------------------------- y axis
template <typename T, int MR, bool INV>
__global__ void __launch_bounds__(kLineThreads, min_blocks<T, MR>())
    k_line_y(typename CplxOf<T>::type* __restrict__ spec, long long sstride, LinePlan p, int K2, int cols, int lb,
             int n_rhs, const int* __restrict__ active, const typename CplxOf<T>::type* __restrict__ tw) {
  typedef typename CplxOf<T>::type C;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int tile = blockIdx.x / n_rhs, rhs = blockIdx.x - tile * n_rhs;
  if (active && !active[rhs]) return;
  C* buf = reinterpret_cast<C*>(smraw);
  const int col = threadIdx.x & ((1 << lb) - 1), t0 = threadIdx.x >> lb, nt = blockDim.x >> lb;
  const int q = (tile << lb) + col;
  const bool ok = q < cols;
  const int ci = q / K2;
  C* line = spec + rhs * sstride + (long long)ci * p.n * K2 + (q - ci * K2);
  C zero;
  zero.x = zero.y = T(0);
  first_factor<MR, INV>(p, buf, lb, col, t0, nt, tw, [&](int j) { return ok ? line[(long long)j * K2] : zero; });
  __syncthreads();
  if (p.RM > 1) {
    mid_factor<MR, INV, false>(p, buf, lb, col, t0, nt, tw);
    __syncthreads();
  }
  if (!ok) return;
  with_radix<MR>(p.RL, [&](auto rc) {
    constexpr int R = decltype(rc)::v;
    for (int w = t0; w < p.R1 * p.RM; w += nt) {  // w = k1 RM + km
      const int k1 = w / p.RM, km = w - k1 * p.RM;
      const int k0 = k1 + p.R1 * km;
      C v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = buf[((w * R + r) << lb) + col];
      fast::Dft<C, R, INV>::run(v);
#pragma unroll
      for (int r = 0; r < R; ++r) line[(long long)(k0 + r * p.R1 * p.RM) * K2] = v[r];
    }
  });
}

// ---------------------------------------------------------------- x axis, Green operator, x inverse
// What the symbol of a frequency is formed from (green_factor): e_a and e_a - 1 per axis, 1 / h_a, |T| / 2
template <typename T>
struct SymbolArgs {
  const typename CplxOf<T>::type* ge[3];
  const typename CplxOf<T>::type* gs[3];
  T ih[3], halfvol;
  int K2;
};

// columns q = j K2 + k2 of the n1 K2 lines of one component; TABLE: the inverses come from the table,
// otherwise every frequency's symbol is factorised here
template <typename T, int MR, bool TABLE>
__global__ void __launch_bounds__(kLineThreads, min_blocks<T, MR, true>())
    k_line_x(typename CplxOf<T>::type* __restrict__ spec, long long sstride, LinePlan p, int cols, int lb, int n_rhs,
             const int* __restrict__ active, const typename CplxOf<T>::type* __restrict__ tw,
             const T* __restrict__ table, const SymbolArgs<T> sy) {
  typedef typename CplxOf<T>::type C;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int tile = blockIdx.x / n_rhs, rhs = blockIdx.x - tile * n_rhs;
  if (active && !active[rhs]) return;
  C* buf = reinterpret_cast<C*>(smraw);
  const int col = threadIdx.x & ((1 << lb) - 1), t0 = threadIdx.x >> lb, nt = blockDim.x >> lb;
  const int q = (tile << lb) + col;
  const bool ok = q < cols;
  const int n = p.n, NR = p.RM * p.RL;
  const long long cs = (long long)n * cols;  // component stride; a line's elements are cols apart
  C* line = spec + rhs * sstride + q;
  const int bc = n << lb;  // buffer of one component
  C zero;
  zero.x = zero.y = T(0);
  // first factor of the three components; FP32: the next component's loads are in flight while one
  // is transformed (FP64 has no registers for it, and its pipe is the limit)
  constexpr int kPipe = sizeof(T) == 4 ? 2 : 1;
  with_radix<MR>(p.R1, [&](auto rc) {
    constexpr int R = decltype(rc)::v;
    for (int j = t0; j < NR; j += nt) {
      C v[kPipe][R];
      const C* e = line + (long long)j * cols;
      const long long st = (long long)NR * cols;
      if (kPipe == 2) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[0][r] = ok ? e[r * st] : zero;
      }
#pragma unroll(kPipe == 2 ? 3 : 1)
      for (int c = 0; c < 3; ++c) {
        const int cl = kPipe == 2 ? c + 1 : c;  // the component to load now
        if (cl < 3) {
#pragma unroll
          for (int r = 0; r < R; ++r) v[cl % kPipe][r] = ok ? e[cl * cs + r * st] : zero;
        }
        C* u = v[c % kPipe];
        fast::Dft<C, R, false>::run(u);
#pragma unroll
        for (int r = 0; r < R; ++r)
          buf[c * bc + ((r * NR + j) << lb) + col] = r ? cmul(u[r], __ldg(tw + r * j)) : u[0];
      }
    }
  });
  __syncthreads();
  if (p.RM > 1) {
    for (int c = 0; c < 3; ++c) mid_factor<MR, false, false>(p, buf + c * bc, lb, col, t0, nt, tw);
    __syncthreads();
  }
  if (ok)
    with_radix<MR>(p.RL, [&](auto rc) {
      constexpr int R = decltype(rc)::v;
      for (int w = t0; w < p.R1 * p.RM; w += nt) {  // w = k1 RM + km
        const int k1 = w / p.RM, km = w - k1 * p.RM;
        const int k0 = k1 + p.R1 * km, kstep = p.R1 * p.RM;
        C* b = buf + ((w * R) << lb) + col;
        T g[9], h[9];  // the inverse at this frequency and (FP32) in flight the one at the next
        const T* t = table + (long long)k0 * cols + q;
        if (TABLE && kPipe == 2) {
#pragma unroll
          for (int i = 0; i < 9; ++i) g[i] = __ldg(t + i * cs);
        }
#pragma unroll 1
        for (int c = 0; c < 3; ++c) {
          C v[R];
#pragma unroll
          for (int r = 0; r < R; ++r) v[r] = b[c * bc + (r << lb)];
          fast::Dft<C, R, false>::run(v);
#pragma unroll
          for (int r = 0; r < R; ++r) b[c * bc + (r << lb)] = v[r];
        }
        if constexpr (!TABLE) {
          const int j = q / sy.K2, k2 = q - j * sy.K2;
#pragma unroll 1
          for (int r = 0; r < R; ++r) {
            const int kx = k0 + r * kstep;
            C* f = b + (r << lb);
            C F0 = f[0], F1 = f[bc], F2 = f[2 * bc];
            fast::GreenFactor<C, T> gf;
            if (fast::green_factor<C, T>(gf, sy.ge[0][kx], sy.ge[1][j], sy.ge[2][k2], sy.gs[0][kx], sy.gs[1][j],
                                         sy.gs[2][k2], sy.ih[0], sy.ih[1], sy.ih[2], sy.halfvol))
              fast::green_solve<C, T>(gf, F0, F1, F2);
            else
              F0 = F1 = F2 = zero;
            f[0] = F0;
            f[bc] = F1;
            f[2 * bc] = F2;
          }
        }
        for (int r = 0; TABLE && r < R; ++r) {
          if (kPipe == 1) {
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = __ldg(t + i * cs);
          }
          if (r + 1 < R) {
            t += (long long)kstep * cols;
            if (kPipe == 2) {
#pragma unroll
              for (int i = 0; i < 9; ++i) h[i] = __ldg(t + i * cs);
            }
          }
          const T i00 = g[0], i11 = g[1], i22 = g[2];
          C i10, i20, i21;
          i10.x = g[3];
          i10.y = g[4];
          i20.x = g[5];
          i20.y = g[6];
          i21.x = g[7];
          i21.y = g[8];
          C* f = b + (r << lb);
          const C F0 = f[0], F1 = f[bc], F2 = f[2 * bc];
          C z0, z1, z2;
          z0.x = i00 * F0.x + (i10.x * F1.x + i10.y * F1.y) + (i20.x * F2.x + i20.y * F2.y);
          z0.y = i00 * F0.y + (i10.x * F1.y - i10.y * F1.x) + (i20.x * F2.y - i20.y * F2.x);
          z1.x = i11 * F1.x + (i10.x * F0.x - i10.y * F0.y) + (i21.x * F2.x + i21.y * F2.y);
          z1.y = i11 * F1.y + (i10.x * F0.y + i10.y * F0.x) + (i21.x * F2.y - i21.y * F2.x);
          z2.x = i22 * F2.x + (i20.x * F0.x - i20.y * F0.y) + (i21.x * F1.x - i21.y * F1.y);
          z2.y = i22 * F2.y + (i20.x * F0.y + i20.y * F0.x) + (i21.x * F1.y + i21.y * F1.x);
          f[0] = z0;
          f[bc] = z1;
          f[2 * bc] = z2;
          if (kPipe == 2) {
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = h[i];
          }
        }
#pragma unroll 1
        for (int c = 0; c < 3; ++c) {
          C v[R];
#pragma unroll
          for (int r = 0; r < R; ++r) v[r] = b[c * bc + (r << lb)];
          fast::Dft<C, R, true>::run(v);
          // l = r: the twiddle of the factor that the forward transform ran before this one
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int e = p.RM > 1 ? km * r * p.R1 : k1 * r;
            b[c * bc + (r << lb)] = cmulc(v[r], __ldg(tw + e));
          }
        }
      }
    });
  __syncthreads();
  if (p.RM > 1) {
    for (int c = 0; c < 3; ++c) mid_factor<MR, true, true>(p, buf + c * bc, lb, col, t0, nt, tw);
    __syncthreads();
  }
  if (!ok) return;
  with_radix<MR>(p.R1, [&](auto rc) {
    constexpr int R = decltype(rc)::v;
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
      C* lc = line + c * cs;
      for (int j = t0; j < NR; j += nt) {
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = buf[c * bc + ((r * NR + j) << lb) + col];
        fast::Dft<C, R, true>::run(v);
#pragma unroll
        for (int r = 0; r < R; ++r) lc[(long long)(j + r * NR) * cols] = v[r];
      }
    }
  });
}

// ---------------------------------------------------------------- z axis
// Rows of n2 = 2 M reals, B rows per block.  Shared memory: the padded factor layout
// [row][k1 P1 + m P3 + l] (odd pitches: lanes over k1 or m hit different banks), then rows of M in
// natural order.
// Division of an item index i by a launch constant d through m = ceil(2^32 / d) (0: d = 1), exact
// while i d < 2^32: one multiplication instead of about twenty instructions per work item, which the
// z passes feel (FP32, bound by issue as much as by memory).
struct Divisor {
  int d;
  unsigned m;
  __device__ __forceinline__ int of(int i) const { return m ? (int)__umulhi((unsigned)i, m) : i; }
};
struct RowPlan {
  int B, P1, P3, LS;  // rows per block, pitches of k1 and m, row pitch
  // work items of a row: RM RL (first factor), R1 RL (middle), R1 RM (last), pairs; RL and R1
  Divisor nr, mid, last, half, rl, r1;
};

// middle factor over a block's rows, in place
template <int MR, bool INV, typename C>
__device__ __forceinline__ void row_mid(const LinePlan& p, const RowPlan& w, C* buf, const C* __restrict__ tw) {
  with_radix<MR>(p.RM, [&](auto rc) {
    constexpr int R = decltype(rc)::v;
    const int per = w.mid.d;
    for (int i = threadIdx.x; i < w.B * per; i += blockDim.x) {
      const int row = w.mid.of(i), j = i - row * per;
      const int k1 = w.rl.of(j), l = j - k1 * p.RL;
      C* b = buf + row * w.LS + k1 * w.P1 + l;
      C v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = b[r * w.P3];
      fast::Dft<C, R, INV>::run(v);
#pragma unroll
      for (int r = 0; r < R; ++r) b[r * w.P3] = twid<INV>(v[r], __ldg(tw + 2 * r * l * p.R1));
    }
  });
}
// last factor of a work item's outputs t = k0 + r step: pre(row, k0, step, g) may load what
// out(row, k0, step, v, g) combines with the values v, while the DFT runs
template <int MR, bool INV, typename C, typename PRE, typename OUT>
__device__ __forceinline__ void row_last(const LinePlan& p, const RowPlan& w, const C* buf, int nrows, const PRE& pre,
                                         const OUT& out) {
  with_radix<MR>(p.RL, [&](auto rc) {
    constexpr int R = decltype(rc)::v;
    const int per = w.last.d;
    for (int i = threadIdx.x; i < nrows * per; i += blockDim.x) {
      const int row = w.last.of(i), k0 = i - row * per;  // k0 = k1 + R1 km
      const int km = w.r1.of(k0), k1 = k0 - km * p.R1;
      const C* b = buf + row * w.LS + k1 * w.P1 + km * w.P3;
      C v[R], g[R];
      pre(row, k0, per, g);
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = b[r];
      fast::Dft<C, R, INV>::run(v);
      out(row, k0, per, v, g);
    }
  });
}

template <typename T, int MR>
__global__ void __launch_bounds__(kLineThreads, min_blocks<T, MR>())
    k_line_z_fwd(T* __restrict__ f, typename CplxOf<T>::type* __restrict__ spec, long long stride, long long sstride,
                 LinePlan p, RowPlan w, long long rows, const int* __restrict__ active,
                 const typename CplxOf<T>::type* __restrict__ tw, unsigned long long* __restrict__ units,
                 const T* __restrict__ qv, const RhsState* __restrict__ st) {
  typedef typename CplxOf<T>::type C;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int rhs = blockIdx.y;
  if (active && !active[rhs]) return;
  if (units && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(units, 1ULL);
  C* buf = reinterpret_cast<C*>(smraw);
  C* nat = buf + w.B * w.LS;
  const int M = p.n, NR = p.RM * p.RL;
  const long long row0 = (long long)blockIdx.x * w.B;
  const int nrows = (int)min((long long)w.B, rows - row0);
  T* fr = f + rhs * stride + row0 * 2 * M;
  const T* qr = qv ? qv + rhs * stride + row0 * 2 * M : nullptr;
  const T alpha = qv ? (T)st[rhs].alpha : T(0);
  // pairs of reals as one access where every right-hand side is aligned to them (an odd stride
  // puts every other one on half a pair)
  const bool pairs = (stride & 1) == 0;
  auto get = [&](const T* a, long long m) {
    C v;
    if (pairs) {
      v = *reinterpret_cast<const C*>(a + 2 * m);
    } else {
      v.x = a[2 * m];
      v.y = a[2 * m + 1];
    }
    return v;
  };
  with_radix<MR>(p.R1, [&](auto rc) {
    constexpr int R = decltype(rc)::v;
    for (int i = threadIdx.x; i < nrows * NR; i += blockDim.x) {
      const int row = w.nr.of(i), j = i - row * NR;
      const int m = w.rl.of(j), l = j - m * p.RL;
      const long long o = (long long)row * M + j;
      C v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = get(fr, o + r * NR);
      if (qv) {  // fused CG update f -= alpha A d
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const C a = get(qr, o + r * NR);
          v[r].x -= alpha * a.x;
          v[r].y -= alpha * a.y;
          if (pairs) {
            *reinterpret_cast<C*>(fr + 2 * (o + r * NR)) = v[r];
          } else {
            fr[2 * (o + r * NR)] = v[r].x;
            fr[2 * (o + r * NR) + 1] = v[r].y;
          }
        }
      }
      fast::Dft<C, R, false>::run(v);
      C* b = buf + row * w.LS + m * w.P3 + l;
#pragma unroll
      for (int r = 0; r < R; ++r) b[r * w.P1] = r ? cmul(v[r], __ldg(tw + 2 * r * j)) : v[0];
    }
  });
  __syncthreads();
  if (p.RM > 1) {
    row_mid<MR, false>(p, w, buf, tw);
    __syncthreads();
  }
  row_last<MR, false>(p, w, buf, nrows, [](int, int, int, auto&) {}, [&](int row, int k0, int step, auto& v, auto&) {
    constexpr int R = sizeof(v) / sizeof(C);
#pragma unroll
    for (int r = 0; r < R; ++r) nat[row * M + k0 + r * step] = v[r];
  });
  __syncthreads();
  // twice the real transform: X_k = E + w^k O, X_(M-k) = conj(E - w^k O) with E = Z_k + conj Z_(M-k),
  // O = -i (Z_k - conj Z_(M-k)), w = exp(-2 pi i / n2)
  const int half = M / 2 + 1, K2 = M + 1;
  C* sp = spec + rhs * sstride + row0 * K2;
  for (int i = threadIdx.x; i < nrows * half; i += blockDim.x) {
    const int row = w.half.of(i), k = i - row * half;
    const C a = nat[row * M + k], b = nat[row * M + (k ? M - k : 0)];
    C E, O;
    E.x = a.x + b.x;
    E.y = a.y - b.y;
    O.x = a.y + b.y;
    O.y = b.x - a.x;
    O = cmul(O, __ldg(tw + k));
    C* s = sp + (long long)row * K2;
    s[k] = cadd(E, O);
    if (2 * k != M) {
      C X = csub(E, O);
      X.y = -X.y;
      s[M - k] = X;
    }
  }
}

template <typename T, int MR>
__global__ void __launch_bounds__(kLineThreads, min_blocks<T, MR>())
    k_line_z_inv(const typename CplxOf<T>::type* __restrict__ spec, const T* __restrict__ f, T* __restrict__ z,
                 long long stride, long long sstride, LinePlan p, RowPlan w, long long rows, T scale,
                 const int* __restrict__ active, const typename CplxOf<T>::type* __restrict__ tw,
                 double* __restrict__ partials, int nparts) {
  typedef typename CplxOf<T>::type C;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ T red[kLineThreads];
  const int rhs = blockIdx.y;
  if (active && !active[rhs]) return;
  C* buf = reinterpret_cast<C*>(smraw);
  C* nat = buf + w.B * w.LS;
  const int M = p.n, NR = p.RM * p.RL;
  const long long row0 = (long long)blockIdx.x * w.B;
  const int nrows = (int)min((long long)w.B, rows - row0);
  // Z_k = E + i O, Z_(M-k) = conj E + i conj O with E = Y_k + conj Y_(M-k), O = conj(w^k) (Y_k -
  // conj Y_(M-k)); the imaginary parts at k = 0 and M do not enter a real row
  const int half = M / 2 + 1, K2 = M + 1;
  const C* sp = spec + rhs * sstride + row0 * K2;
  constexpr int U = sizeof(T) == 4 ? 4 : 2;  // pairs whose loads a thread has in flight
  for (int i0 = threadIdx.x; i0 < nrows * half; i0 += U * blockDim.x) {
    C a[U], b[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * blockDim.x;
      if (i < nrows * half) {
        const int row = w.half.of(i), k = i - row * half;
        const C* s = sp + (long long)row * K2;
        a[u] = s[k];
        b[u] = s[M - k];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * blockDim.x;
      if (i >= nrows * half) break;
      const int row = w.half.of(i), k = i - row * half;
      if (k == 0) a[u].y = b[u].y = T(0);
      C E, O;
      E.x = a[u].x + b[u].x;
      E.y = a[u].y - b[u].y;
      O.x = a[u].x - b[u].x;
      O.y = a[u].y + b[u].y;
      O = cmulc(O, __ldg(tw + k));
      C Z;
      Z.x = E.x - O.y;
      Z.y = E.y + O.x;
      nat[row * M + k] = Z;
      if (k && 2 * k != M) {
        Z.x = E.x + O.y;
        Z.y = O.x - E.y;
        nat[row * M + M - k] = Z;
      }
    }
  }
  __syncthreads();
  with_radix<MR>(p.R1, [&](auto rc) {
    constexpr int R = decltype(rc)::v;
    for (int i = threadIdx.x; i < nrows * NR; i += blockDim.x) {
      const int row = w.nr.of(i), j = i - row * NR;
      const int m = w.rl.of(j), l = j - m * p.RL;
      C v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = nat[row * M + j + r * NR];
      fast::Dft<C, R, true>::run(v);
      C* b = buf + row * w.LS + m * w.P3 + l;
#pragma unroll
      for (int r = 0; r < R; ++r) b[r * w.P1] = r ? cmulc(v[r], __ldg(tw + 2 * r * j)) : v[0];
    }
  });
  __syncthreads();
  if (p.RM > 1) {
    row_mid<MR, true>(p, w, buf, tw);
    __syncthreads();
  }
  const T* fr = f + rhs * stride + row0 * 2 * M;
  T* zr = z + rhs * stride + row0 * 2 * M;
  const bool pairs = (stride & 1) == 0;
  T acc = T(0);
  const auto load_f = [&](int row, int t0, int step, auto& g) {
    constexpr int R = sizeof(g) / sizeof(C);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const long long o = 2 * ((long long)row * M + t0 + r * step);
      if (pairs) {
        g[r] = *reinterpret_cast<const C*>(fr + o);
      } else {
        g[r].x = fr[o];
        g[r].y = fr[o + 1];
      }
    }
  };
  row_last<MR, true>(p, w, buf, nrows, load_f, [&](int row, int t0, int step, auto& v, auto& g) {
    constexpr int R = sizeof(v) / sizeof(C);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const long long o = 2 * ((long long)row * M + t0 + r * step);
      C a;
      a.x = v[r].x * scale;
      a.y = v[r].y * scale;
      if (pairs) {
        *reinterpret_cast<C*>(zr + o) = a;
      } else {
        zr[o] = a.x;
        zr[o + 1] = a.y;
      }
      acc += a.x * g[r].x;
      acc += a.y * g[r].y;
    }
  });
  const double tot = block_sum1<T>(acc, red);
  if (threadIdx.x == 0) partials[(long long)rhs * nparts + blockIdx.x] = tot;
}

// ---------------------------------------------------------------- Green table
// Inverse of M(xi) per frequency: (00, 11, 22, Re 10, Im 10, Re 20, Im 20, Re 21, Im 21), each
// [kx][j][k2]; zeros at xi = 0.  Formed from the Cholesky factor in the table's own precision.
template <typename T>
__global__ void k_line_green(T* __restrict__ table, int n0, int n1, const SymbolArgs<T> sy) {
  typedef typename CplxOf<T>::type C;
  const int K2 = sy.K2;
  const long long n = (long long)n0 * n1 * K2;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int k2 = (int)(i % K2), j = (int)((i / K2) % n1), kx = (int)(i / ((long long)K2 * n1));
    fast::GreenFactor<C, T> gf;
    T v[9] = {};
    if (fast::green_factor<C, T>(gf, sy.ge[0][kx], sy.ge[1][j], sy.ge[2][k2], sy.gs[0][kx], sy.gs[1][j], sy.gs[2][k2],
                                 sy.ih[0], sy.ih[1], sy.ih[2], sy.halfvol)) {
      C c[3];
#pragma unroll
      for (int col = 0; col < 3; ++col) {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          c[r].x = T(r == col);
          c[r].y = T(0);
        }
        fast::green_solve<C, T>(gf, c[0], c[1], c[2]);
        v[col] = c[col].x;
        if (col == 0) {
          v[3] = c[1].x;
          v[4] = c[1].y;
          v[5] = c[2].x;
          v[6] = c[2].y;
        } else if (col == 1) {
          v[7] = c[2].x;
          v[8] = c[2].y;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) table[k * n + i] = v[k];
  }
}

}  // namespace lines

// A grid's plans and launch shapes.
struct LineGrid {
  int n0, n1, n2, K2;
  LinePlan ax[3];  // ax[2]: the plan of n2 / 2
  lines::RowPlan rp;
  int zblocks;
};
bool line_grid(LineGrid& g, int n0, int n1, int n2, bool dbl);  // false for an unsupported length (fft.cu)

// launchers of one precision (instantiated in fft_lines_f32.cu and fft_lines_f64.cu; table: nullptr where
// the context has none); lines_opt_in for the current device before the first launch
template <typename T>
cudaError_t lines_opt_in();
template <typename T>
cudaError_t lines_precondition(const LineGrid& g, T* f, T* z, void* spec, long long stride, long long sstride,
                               const int* active, const void* const* tw, const T* table,
                               const lines::SymbolArgs<T>& sy, unsigned long long* units, const T* q,
                               const RhsState* st, double* partials, int nparts, int n_rhs, cudaStream_t s);
template <typename T>
cudaError_t lines_green_table(T* table, const LineGrid& g, const lines::SymbolArgs<T>& sy, cudaStream_t s);

}  // namespace xfft
