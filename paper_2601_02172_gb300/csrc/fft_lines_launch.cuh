// Launchers of the line passes (fft_lines.cuh) for one precision.
#pragma once

#include <algorithm>

#include "fft_lines.cuh"

namespace xfft {
namespace lines {

// The most dynamic shared memory that a launch below asks for (column_bits; the z passes stay at 64 KB).
constexpr size_t kLineShared = 200 * 1024;

// Columns per block (2^lb) of the y and x passes: 128 bytes of every plane crossed, fewer where a
// block's lines would pass 100 KB of shared memory (two blocks per SM) or the launch would not give
// every SM two blocks; never below 4 (32-byte sectors) unless shared memory asks for it.
inline int column_bits(size_t line_bytes, size_t csize, long long cols, int n_rhs) {
  int lb = csize == 8 ? 4 : 3;
  while (lb > 2 && ((line_bytes << lb) > 100 * 1024 || ((cols >> lb) + 1) * n_rhs < 2 * 152)) --lb;
  while (lb > 0 && (line_bytes << lb) > kLineShared) --lb;
  return lb;
}
inline int column_threads(const LinePlan& p, int lb) {
  const int items = (p.n / std::min(p.R1, p.RL)) << lb;
  return std::min(kLineThreads, std::max(32, (items + 31) / 32 * 32));
}
inline int max_radix(const LinePlan& p) { return std::max(p.R1, std::max(p.RM, p.RL)); }

}  // namespace lines

// All lengths share the kernels of a precision and radix class, and the opt-in to more than 48 KB of
// shared memory belongs to the kernel, not to a launch: it is given once, at its largest, so that
// no launch of another grid (another context in another thread, another node of a graph) finds it lowered.
template <typename T>
cudaError_t lines_opt_in() {
  using namespace lines;
  const void* const kernels[] = {
      (const void*)k_line_z_fwd<T, 12>,    (const void*)k_line_z_fwd<T, 16>,    (const void*)k_line_z_inv<T, 12>,
      (const void*)k_line_z_inv<T, 16>,    (const void*)k_line_y<T, 12, false>, (const void*)k_line_y<T, 16, false>,
      (const void*)k_line_y<T, 12, true>,  (const void*)k_line_y<T, 16, true>,  (const void*)k_line_x<T, 12, true>,
      (const void*)k_line_x<T, 16, true>,  (const void*)k_line_x<T, 12, false>, (const void*)k_line_x<T, 16, false>};
  for (const void* k : kernels) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLineShared);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t lines_precondition(const LineGrid& g, T* f, T* z, void* spec_v, long long stride, long long sstride,
                               const int* active, const void* const* tw, const T* table,
                               const lines::SymbolArgs<T>& sy, unsigned long long* units, const T* q,
                               const RhsState* st, double* partials, int nparts, int n_rhs, cudaStream_t s) {
  using namespace lines;
  typedef typename CplxOf<T>::type C;
  C* spec = static_cast<C*>(spec_v);
  const C* tw0 = static_cast<const C*>(tw[0]);
  const C* tw1 = static_cast<const C*>(tw[1]);
  const C* tw2 = static_cast<const C*>(tw[2]);
  const long long rows = 3LL * g.n0 * g.n1;
  const LinePlan& pz = g.ax[2];
  const size_t smz = sizeof(C) * (size_t)g.rp.B * (g.rp.LS + pz.n);
  const int nz = g.rp.B * (pz.n / std::min(pz.R1, pz.RL));
  const int tz = std::min(kLineThreads, std::max(32, (nz + 31) / 32 * 32));
  const auto fz = max_radix(pz) > 12 ? k_line_z_fwd<T, 16> : k_line_z_fwd<T, 12>;
  const auto iz = max_radix(pz) > 12 ? k_line_z_inv<T, 16> : k_line_z_inv<T, 12>;
  fz<<<dim3(g.zblocks, n_rhs), tz, smz, s>>>(f, spec, stride, sstride, pz, g.rp, rows, active, tw2, units,
                                                          q, st);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;

  const int ycols = 3 * g.n0 * g.K2;
  const size_t ly = sizeof(C) * g.n1;
  const int by = column_bits(ly, sizeof(C), ycols, n_rhs);
  const int gy = (ycols + (1 << by) - 1) >> by, ty = column_threads(g.ax[1], by);
  const bool big_y = max_radix(g.ax[1]) > 12;
  const auto fy = big_y ? k_line_y<T, 16, false> : k_line_y<T, 12, false>;
  const auto iy = big_y ? k_line_y<T, 16, true> : k_line_y<T, 12, true>;
  fy<<<gy * n_rhs, ty, ly << by, s>>>(spec, sstride, g.ax[1], g.K2, ycols, by, n_rhs, active, tw1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;

  const int xcols = g.n1 * g.K2;
  const size_t lx = 3 * sizeof(C) * g.n0;
  const int bx = column_bits(lx, sizeof(C), xcols, n_rhs);
  const int gx = (xcols + (1 << bx) - 1) >> bx, tx = column_threads(g.ax[0], bx);
  const bool big_x = max_radix(g.ax[0]) > 12;
  const auto kx = table ? (big_x ? k_line_x<T, 16, true> : k_line_x<T, 12, true>)
                        : (big_x ? k_line_x<T, 16, false> : k_line_x<T, 12, false>);
  kx<<<gx * n_rhs, tx, lx << bx, s>>>(spec, sstride, g.ax[0], xcols, bx, n_rhs, active, tw0, table, sy);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;

  iy<<<gy * n_rhs, ty, ly << by, s>>>(spec, sstride, g.ax[1], g.K2, ycols, by, n_rhs, active, tw1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const double scale = 0.5 / ((double)g.n0 * g.n1 * g.n2);  // the spectrum holds twice the transform
  iz<<<dim3(g.zblocks, n_rhs), tz, smz, s>>>(spec, f, z, stride, sstride, pz, g.rp, rows, (T)scale, active,
                                                          tw2, partials, nparts);
  return cudaGetLastError();
}

template <typename T>
cudaError_t lines_green_table(T* table, const LineGrid& g, const lines::SymbolArgs<T>& sy, cudaStream_t s) {
  const long long n = (long long)g.n0 * g.n1 * g.K2;
  const int blocks = (int)std::min<long long>((n + 127) / 128, 152 * 64);
  lines::k_line_green<T><<<blocks, 128, 0, s>>>(table, g.n0, g.n1, sy);
  return cudaGetLastError();
}

#define XFFT_LINES_INST(T)                                                                                         \
  template cudaError_t lines_opt_in<T>();                                                                          \
  template cudaError_t lines_precondition<T>(const LineGrid&, T*, T*, void*, long long, long long, const int*,      \
                                             const void* const*, const T*, const lines::SymbolArgs<T>&,            \
                                             unsigned long long*, const T*, const RhsState*, double*, int, int,    \
                                             cudaStream_t);                                                        \
  template cudaError_t lines_green_table<T>(T*, const LineGrid&, const lines::SymbolArgs<T>&, cudaStream_t);

}  // namespace xfft
