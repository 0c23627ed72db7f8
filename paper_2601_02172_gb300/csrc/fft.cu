// X-FFT preconditioner P^{-1} = diag(A0_11^{-1}, I) (eqs. scaledPreconditioner,
// constantCoefficientPreconditioner, GreenHermitian).
//
// The constant-coefficient operator A0_11 = int grad^s N_FE : grad^s N_FE is a periodic
// convolution, diagonalised by the 3D DFT into 3x3 Hermitian blocks
//   M(xi) = Z(xi)^H A0_11,v Z(xi),   Z = c(xi) (x) I_3,   c_j = exp(i theta . Y_j),
// theta_a = 2 pi xi_a / n_a.  Summing the six Kuhn tets in closed form gives
//   M(xi) = (|T| / 2) sum_tets ( |G|^2 I + G G^H ),   G = sum_a c_a grad N_a,
// and for the tet (p,q,r): G_p = s_p/h_p, G_q = e_p s_q/h_q, G_r = e_p e_q s_r/h_r with
// e_a = exp(i theta_a), s_a = e_a - 1.  xi = 0 maps to 0 (mean-free standard part).
//
// The 3D transforms are hand written: the y-z plane path (three passes) for FP32 on square planes of
// 32 to 128 nodes (fft_slab.cuh), five passes of line transforms otherwise (fft_lines.cuh).  This
// file holds the plans, the enriched block (the identity on the scaled enriched DOFs, or inverse
// 3x3 blocks, with its f^T z sum) and the dispatch.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>
#include <type_traits>
#include <vector>

#include "fft_lines.cuh"
#include "xfft_kernels.h"

namespace xfft {

struct FftPlan {
  GridDev g;
  LineGrid lf, ld;  // line passes in FP32 and FP64
  double2* twd[3];
  float2* twf[3];
  double2* ged[3];  // e_a(xi)
  double2* gsd[3];  // e_a(xi) - 1
  float2* gef[3];
  float2* gsf[3];
  bool slab;               // the FP32 passes take the y-z plane path (fft_slab.cu)
  float* gtab = nullptr;   // its Green factor table
  float* tabf = nullptr;   // Green tables of the line passes, the caller's memory (fft_table_fill)
  double* tabd = nullptr;
  void* pool = nullptr;
};

// slab path (fft_slab.cu)
bool slab_supported(int n0, int n1, int n2);
size_t slab_table_floats(int n0, int n1);
int slab_z_blocks(int n0);
cudaError_t slab_green_table(float* table, int n0, int n1, const void* const* ge, const void* const* gs,
                             const double* ih, double halfvol, cudaStream_t s);
cudaError_t slab_precondition(int n0, int n1, float* f, float* z, void* spec, long long stride, long long sstride,
                              const int* active, const void* tw0, const void* tw1, const void* tw2,
                              const float* table, const void* const* ge, const void* const* gs,
                              const double* ih, double halfvol, unsigned long long* units, const float* q,
                              const RhsState* st, double* partials, int nparts, int n_rhs, cudaStream_t s);

// ---------------------------------------------------------------- enriched block
// z_X = f_X (identity on the scaled enriched DOFs, eq. scaledPreconditioner) or, with eblk
// (6 x nX: inverse of each node's 3x3 block, entries 00, 11, 22, 01, 02, 12), z_X = B^-1 f_X per
// enriched node.  Enriched DOFs are component-major: f[off + c nX + j].
template <typename T>
__global__ void k_enr_precond(T* __restrict__ f, T* __restrict__ z, long long stride,
                              long long off, int nX, const int* __restrict__ active,
                              double* __restrict__ partials, int nparts, int slot0,
                              const T* __restrict__ q, const RhsState* __restrict__ st,
                              const T* __restrict__ eblk) {
  __shared__ T red[256];
  const int rhs = blockIdx.y;
  if (active && !active[rhs]) return;
  T* fr = f + rhs * stride + off;
  T* zr = z + rhs * stride + off;
  const T* qr = q ? q + rhs * stride + off : nullptr;
  const T alpha = q ? (T)st[rhs].alpha : T(0);
  T acc = T(0);
  if (!eblk) {
    const long long count = 3LL * nX;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
      T v = fr[i];
      if (q) {
        v -= alpha * qr[i];  // fused CG update f -= alpha A d
        fr[i] = v;
      }
      zr[i] = v;
      acc += v * v;
    }
  } else {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nX; j += gridDim.x * blockDim.x) {
      T v[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        v[c] = fr[(long long)c * nX + j];
        if (q) {
          v[c] -= alpha * qr[(long long)c * nX + j];
          fr[(long long)c * nX + j] = v[c];
        }
      }
      const T b00 = eblk[j], b11 = eblk[nX + j], b22 = eblk[2 * (long long)nX + j];
      const T b01 = eblk[3 * (long long)nX + j], b02 = eblk[4 * (long long)nX + j];
      const T b12 = eblk[5 * (long long)nX + j];
      const T z0 = b00 * v[0] + b01 * v[1] + b02 * v[2];
      const T z1 = b01 * v[0] + b11 * v[1] + b12 * v[2];
      const T z2 = b02 * v[0] + b12 * v[1] + b22 * v[2];
      zr[j] = z0;
      zr[nX + j] = z1;
      zr[2 * (long long)nX + j] = z2;
      acc += v[0] * z0 + v[1] * z1 + v[2] * z2;
    }
  }
  const double tot = block_sum1<T>(acc, red);
  if (threadIdx.x == 0) partials[(long long)rhs * nparts + slot0 + blockIdx.x] = tot;
}

// ---------------------------------------------------------------- plan
// Factors of a line of n values: two of at most 16 where possible, else three.  The estimate per
// value: operations of the DFTs (c(R) / R), six per twiddle step, six per crossing of shared memory,
// and the largest radix (FP64: 1.5 times), which costs registers and leaves few work items per line.
// So FP32 takes 256 = 16 x 16 (three factors: twice the instructions, and the pass is bound by their
// issue as much as by memory), FP64 8 x 4 x 8 (16-point DFTs leave one block of 250 registers per SM
// and the FP64 pipe at 60 % instead of 80 %).
static bool line_plan(LinePlan& p, int n, bool dbl) {
  static const int radix[] = {1, 2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16};
  static const double cost[] = {0, 2, 4, 4, 8, 6, 8, 10, 10, 8, 12, 10.5};
  constexpr int nr = sizeof(radix) / sizeof(radix[0]);
  double best = 1e30;
  for (int a = 1; a < nr; ++a)
    for (int m = 0; m < nr; ++m)
      for (int b = 0; b < nr; ++b) {
        if (radix[a] * radix[m] * radix[b] != n || (b == 0 && m > 0) || b > a) continue;
        const double c = cost[a] + cost[m] + cost[b] + 12.0 * ((m > 0) + (b > 0)) + (dbl ? 1.5 : 1.0) * std::max(radix[a], radix[m]);
        if (c < best) {
          best = c;
          p.n = n;
          p.R1 = radix[a];
          p.RM = radix[m];
          p.RL = radix[b];
        }
      }
  return best < 1e30;
}

bool line_grid(LineGrid& lg, int n0, int n1, int n2, bool dbl) {
  lg.n0 = n0;
  lg.n1 = n1;
  lg.n2 = n2;
  lg.K2 = n2 / 2 + 1;
  if ((n2 & 1) || !line_plan(lg.ax[0], n0, dbl) || !line_plan(lg.ax[1], n1, dbl) || !line_plan(lg.ax[2], n2 / 2, dbl))
    return false;
  const LinePlan& p = lg.ax[2];
  lines::RowPlan& r = lg.rp;
  r.P3 = p.RL | 1;
  r.P1 = p.RM > 1 ? (p.RM * r.P3) | 1 : r.P3;
  r.LS = p.R1 * r.P1;
  const auto divisor = [](int d) {
    lines::Divisor v;
    v.d = d;
    v.m = d > 1 ? (unsigned)(((1ULL << 32) + d - 1) / d) : 0u;
    return v;
  };
  r.nr = divisor(p.RM * p.RL);
  r.mid = divisor(p.R1 * p.RL);
  r.last = divisor(p.R1 * p.RM);
  r.half = divisor(p.n / 2 + 1);
  r.rl = divisor(p.RL);
  r.r1 = divisor(p.R1);
  // rows per block: about 256 work items of the larger factor, 64 KB of FP64 shared memory, and at
  // least two blocks per SM
  const long long rows = 3LL * n0 * n1;
  r.B = 32;
  while (r.B > 1 && (r.B * (p.n / std::max(p.R1, p.RL)) > 2 * lines::kLineThreads ||
                     (size_t)r.B * (r.LS + p.n) * 16 > 64 * 1024 || (r.B > 2 && rows / r.B < 2 * 152)))
    r.B /= 2;
  lg.zblocks = (int)((rows + r.B - 1) / r.B);
  return true;
}

static const void* const* as_void(const float2* const* p) { return reinterpret_cast<const void* const*>(p); }

template <typename T>
static lines::SymbolArgs<T> symbol_args(const FftPlan* p) {
  lines::SymbolArgs<T> sy;
  for (int a = 0; a < 3; ++a) {
    if constexpr (std::is_same<T, double>::value) {
      sy.ge[a] = p->ged[a];
      sy.gs[a] = p->gsd[a];
    } else {
      sy.ge[a] = p->gef[a];
      sy.gs[a] = p->gsf[a];
    }
    sy.ih[a] = (T)(1.0 / p->g.h[a]);
  }
  sy.halfvol = (T)(0.5 * p->g.vol_tet);
  sy.K2 = p->lf.K2;
  return sy;
}

size_t fft_table_bytes(const FftPlan* p, bool dbl) {
  if (!dbl && p->slab) return 0;
  return 9 * (size_t)p->g.n0 * p->g.n1 * p->lf.K2 * (dbl ? sizeof(double) : sizeof(float));
}

cudaError_t fft_table_fill(FftPlan* p, bool dbl, void* mem, cudaStream_t s) {
  const cudaError_t e = dbl ? lines_green_table<double>((double*)mem, p->ld, symbol_args<double>(p), s)
                            : lines_green_table<float>((float*)mem, p->lf, symbol_args<float>(p), s);
  if (e != cudaSuccess) return e;
  if (dbl) p->tabd = (double*)mem;
  else p->tabf = (float*)mem;
  return cudaSuccess;
}

void fft_table_drop(FftPlan* p) {
  p->tabf = nullptr;
  p->tabd = nullptr;
}

cudaError_t fft_plane_table(FftPlan* p) {
  if (!p->slab || p->gtab) return cudaSuccess;
  const GridDev& g = p->g;
  const double ih[3] = {1.0 / g.h[0], 1.0 / g.h[1], 1.0 / g.h[2]};
  float* t = nullptr;
  cudaError_t e = cudaMalloc(&t, slab_table_floats(g.n0, g.n1) * sizeof(float));
  if (e != cudaSuccess) return e;
  e = slab_green_table(t, g.n0, g.n1, as_void(p->gef), as_void(p->gsf), ih, 0.5 * g.vol_tet, 0);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    cudaFree(t);
    return e;
  }
  p->gtab = t;
  return cudaSuccess;
}

// the line kernels' shared-memory opt-in, once per device (20 calls of 10-20 us)
static cudaError_t opt_in_device() {
  static std::mutex mu;
  static std::vector<int> done;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  if (std::find(done.begin(), done.end(), dev) != done.end()) return cudaSuccess;
  if ((e = lines_opt_in<float>()) == cudaSuccess) e = lines_opt_in<double>();
  if (e == cudaSuccess) done.push_back(dev);
  return e;
}

FftPlan* fft_plan_create(const GridDev& g, bool f32, cudaError_t* err) {
  *err = cudaSuccess;
  FftPlan* p = new FftPlan();
  p->g = g;
  p->slab = slab_supported(g.n0, g.n1, g.n2);
  if (!line_grid(p->lf, g.n0, g.n1, g.n2, false) || !line_grid(p->ld, g.n0, g.n1, g.n2, true)) {
    *err = cudaErrorInvalidValue;
    delete p;
    return nullptr;
  }
  if ((*err = opt_in_device()) != cudaSuccess) {
    delete p;
    return nullptr;
  }
  // tables: twiddles exp(-2 pi i k / n) and Green phases per axis
  const int n[3] = {g.n0, g.n1, g.n2};
  size_t tot2d = 0;
  for (int a = 0; a < 3; ++a) tot2d += 3 * (size_t)n[a];
  *err = cudaMalloc(&p->pool, tot2d * (sizeof(double2) + sizeof(float2)));
  if (*err != cudaSuccess) {
    delete p;
    return nullptr;
  }
  std::vector<double2> hd(tot2d);
  std::vector<float2> hf(tot2d);
  size_t off = 0;
  double2* dbase = reinterpret_cast<double2*>(p->pool);
  float2* fbase = reinterpret_cast<float2*>(dbase + tot2d);
  for (int a = 0; a < 3; ++a) {
    const int m = n[a];
    p->twd[a] = dbase + off;
    p->twf[a] = fbase + off;
    p->ged[a] = dbase + off + m;
    p->gef[a] = fbase + off + m;
    p->gsd[a] = dbase + off + 2 * m;
    p->gsf[a] = fbase + off + 2 * m;
    for (int k = 0; k < m; ++k) {
      const double th = 2.0 * M_PI * (double)k / (double)m;
      const double c = cos(th), s = sin(th), sh = sin(0.5 * th);
      hd[off + k] = make_double2(c, -s);
      hd[off + m + k] = make_double2(c, s);
      hd[off + 2 * m + k] = make_double2(-2.0 * sh * sh, s);
    }
    off += 3 * m;
  }
  for (size_t i = 0; i < tot2d; ++i) hf[i] = make_float2((float)hd[i].x, (float)hd[i].y);
  *err = cudaMemcpy(dbase, hd.data(), tot2d * sizeof(double2), cudaMemcpyHostToDevice);
  if (*err == cudaSuccess) *err = cudaMemcpy(fbase, hf.data(), tot2d * sizeof(float2), cudaMemcpyHostToDevice);
  if (*err == cudaSuccess && f32) *err = fft_plane_table(p);
  if (*err != cudaSuccess) {
    fft_plan_destroy(p);
    return nullptr;
  }
  return p;
}

void fft_plan_destroy(FftPlan* p) {
  if (!p) return;
  if (p->pool) cudaFree(p->pool);
  if (p->gtab) cudaFree(p->gtab);
  delete p;
}

size_t fft_spectrum_elems(const FftPlan* p) { return 3ULL * p->g.n0 * p->g.n1 * p->lf.K2; }

static int zpass_blocks(const FftPlan* p, bool dbl) {
  return dbl ? p->ld.zblocks : p->slab ? slab_z_blocks(p->g.n0) : p->lf.zblocks;
}

static int enr_blocks(int nX) {
  if (nX <= 0) return 1;
  const long long n = 3LL * nX;
  long long nb = (n + 255) / 256;
  if (nb > 256) nb = 256;
  return (int)nb;
}

int precondition_blocks(const FftPlan* p, int nX, bool dbl) { return zpass_blocks(p, dbl) + enr_blocks(nX); }

// the FFT passes (standard part) of n_rhs right-hand sides
static cudaError_t standard_part(const FftPlan* p, float* f, float* z, void* spec, long long stride, const int* active,
                                 double* partials, int nparts, int n_rhs, cudaStream_t s, unsigned long long* units,
                                 const float* q, const RhsState* st) {
  const long long sstride = (long long)fft_spectrum_elems(p);
  if (p->slab) {
    const double ih[3] = {1.0 / p->g.h[0], 1.0 / p->g.h[1], 1.0 / p->g.h[2]};
    if (!p->gtab) return cudaErrorInvalidValue;
    return slab_precondition(p->g.n0, p->g.n1, f, z, spec, stride, sstride, active, p->twf[0], p->twf[1], p->twf[2],
                             p->gtab, as_void(p->gef), as_void(p->gsf), ih, 0.5 * p->g.vol_tet, units, q, st, partials,
                             nparts, n_rhs, s);
  }
  return lines_precondition<float>(p->lf, f, z, spec, stride, sstride, active, as_void(p->twf), p->tabf,
                                   symbol_args<float>(p), units, q, st, partials, nparts, n_rhs, s);
}
static cudaError_t standard_part(const FftPlan* p, double* f, double* z, void* spec, long long stride,
                                 const int* active, double* partials, int nparts, int n_rhs, cudaStream_t s,
                                 unsigned long long* units, const double* q, const RhsState* st) {
  return lines_precondition<double>(p->ld, f, z, spec, stride, (long long)fft_spectrum_elems(p), active,
                                    reinterpret_cast<const void* const*>(p->twd), p->tabd, symbol_args<double>(p),
                                    units, q, st, partials, nparts, n_rhs, s);
}

template <typename T>
cudaError_t launch_precondition(const FftPlan* p, T* f, T* z, void* spec, long long stride, int nX, const int* active,
                                double* partials, int nparts, int n_rhs, cudaStream_t s, unsigned long long* units,
                                const T* q, const RhsState* st, const T* eblk, int group) {
  // the FFT passes for `group` right-hand sides at a time: the spectrum of a group can stay in L2
  // between the passes; the enriched block afterwards for all of them
  const int step = group > 0 && group < n_rhs ? group : n_rhs;
  for (int r0 = 0; r0 < n_rhs; r0 += step) {
    const int nr = std::min(step, n_rhs - r0);
    const cudaError_t e = standard_part(p, f + r0 * stride, z + r0 * stride, spec, stride, active ? active + r0 : nullptr,
                                        partials + (long long)r0 * nparts, nparts, nr, s, units,
                                        q ? q + r0 * stride : nullptr, st ? st + r0 : nullptr);
    if (e != cudaSuccess) return e;
  }
  k_enr_precond<T><<<dim3(enr_blocks(nX), n_rhs), 256, 0, s>>>(f, z, stride, 3 * p->g.N, nX, active, partials, nparts,
                                                               zpass_blocks(p, sizeof(T) == 8), q, st, eblk);
  return cudaGetLastError();
}

template cudaError_t launch_precondition<float>(const FftPlan*, float*, float*, void*, long long, int,
                                                const int*, double*, int, int, cudaStream_t,
                                                unsigned long long*, const float*, const RhsState*,
                                                const float*, int);
template cudaError_t launch_precondition<double>(const FftPlan*, double*, double*, void*, long long, int,
                                                 const int*, double*, int, int, cudaStream_t,
                                                 unsigned long long*, const double*, const RhsState*,
                                                 const double*, int);

}  // namespace xfft
