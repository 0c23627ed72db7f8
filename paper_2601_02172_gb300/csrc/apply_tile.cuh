// Uncut-tet stencil of the FP64 and double-word applies.
//
// What bounds it: arithmetic.  GB300 issues two FP64 FMAs per SM and clock (a warp instruction
// holds the pipe 16 clocks), and a double-word operation is about ten FP32 ones, so loads,
// shared-memory traffic, selects and barriers are nearly free and the count of T operations per
// voxel is the time.  Hence, against the marching kernel of apply_kernels.cuh (FP32):
//  * every voxel is evaluated once: no recomputed halo along y, z or x.  A block takes a tile of
//    ty x tz voxel columns for cx planes; node forces inside the tile are combined in shared
//    memory and stored, those on the tile's faces (shared with neighbour tiles) are added with
//    atomics to q, which the launcher clears.
//  * the twelve cube edges of a voxel carry all node differences the six Kuhn tets use; the
//    differences of the four edges in plane x + 1 are kept for the next step (24 new differences
//    per voxel instead of 54), and tensions are summed per edge before the corner forces.
//  * cut tets take zero moduli (no branch), stresses sums come from the edge tensions (24
//    additions instead of 36 multiply-adds) and <d, q> from the node forces.  The forces sum to zero, so
//    a caller's d may be taken relative to its first node there (REL): the plain sum's
//    error grows with the mean of d (10^6 times its variation: 4e-11 of the result on 48^3), that of the
//    tets' energies does not, and the relative sum matches those at 3 subtractions per node instead of 36
//    multiply-adds per voxel.  The CG directions (FUSED) have no mean.
// About 240 operations per voxel (uniform voxels: 210 for the voxel, 22 for each of its about 1.3 node
// visits; counted by ncu at 64^3: 246 with the caller's sums) instead of about 470, and no padding of the
// plane to 15 x 15 node tiles: the tile's shape is a launch parameter (pick_tile).
#pragma once

#include "apply_kernels.cuh"

namespace xfft {

constexpr int kTileThreads = 128;     // largest block
constexpr int kTileMaxBlocks = 1216;  // blocks per right-hand side (they loop over the items)

struct TileShape {
  int threads;   // block size, a multiple of 32
  int ty, tz;    // voxel columns per tile
  int nty, ntz;  // tiles per plane
  int cx, ncx;   // planes per item, items along x
  int items;     // nty ntz ncx
  int blocks;    // min(items, kTileMaxBlocks)
};
TileShape pick_tile(const GridDev& g, int n_rhs);  // apply.cu

template <typename T, bool TOTAL, bool SIG, bool UNIFORM, bool FUSED, int NPH>
__global__ void __launch_bounds__(kTileThreads, 3)
    k_apply_tile(const typename Store<T>::type* __restrict__ d, typename Store<T>::type* __restrict__ q,
                 const ApplyArgs a, const TileShape ts) {
  typedef typename Store<T>::type S;
  constexpr int kNodes = 2 * kTileThreads;  // pick_tile keeps (ty + 1)(tz + 1) <= 2 threads
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int rhs = blockIdx.y;
  if (a.active && !a.active[rhs]) return;
  if (a.units_uncut && tid == 0 && blockIdx.x == 0) atomicAdd(a.units_uncut, 1ULL);
  const GridDev& g = a.g;
  const int n0 = g.n0, n1 = g.n1, n2 = g.n2;
  const long long N = g.N;
  const long long plane = (long long)n1 * n2;
  const int ty = ts.ty, tz = ts.tz, row = tz + 1, nodes = (ty + 1) * row;
  const S* dr = d + rhs * a.stride;
  S* qr = q + rhs * a.stride;

  __shared__ T P[3][kNodes][3];           // node planes (3 in turn)
  __shared__ T C[12][kTileThreads];       // corner forces [2 dy + dz][component] of the plane
  __shared__ double red[7 * 32];

  const int iy = tid / tz, iz = tid - iy * tz;
  T ih[3], wk[3], l0[NPH], m0[NPH], Eb[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    ih[k] = (T)(1.0 / g.h[k]);
    wk[k] = (T)(g.vol_tet / g.h[k]);
  }
  edge_moduli<T, UNIFORM, NPH>(g, a.ph, l0, m0);
  if (TOTAL) edge_strain<T, UNIFORM>(g, a.eps + 6 * rhs, Eb);
  // fused CG update: d_new = z + beta d_old, u += alpha d_old at the nodes the item owns
  const S* zr = FUSED ? static_cast<const S*>(a.fz) + rhs * a.stride : nullptr;
  S* dnr = FUSED ? static_cast<S*>(a.fdnew) + rhs * a.stride : nullptr;
  S* ur = FUSED ? static_cast<S*>(a.fu) + rhs * a.stride : nullptr;
  const T fa = FUSED ? (T)a.st[rhs].alpha : T(0);
  const T fb = FUSED ? (T)a.st[rhs].beta : T(0);

  constexpr bool REL = SIG && !TOTAL && !FUSED && std::is_same<T, double>::value;
  T ref[3] = {T(0), T(0), T(0)};
  if (REL) {
#pragma unroll
    for (int i = 0; i < 3; ++i) ref[i] = from_store<T>(dr[i * N]);
  }
  T en = T(0);
  T sg[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
  for (int item = blockIdx.x; item < ts.items; item += gridDim.x) {
    const int tile = item % (ts.nty * ts.ntz), xc = item / (ts.nty * ts.ntz);
    const int y0 = (tile / ts.ntz) * ty, z0 = (tile % ts.ntz) * tz;
    const int vy = min(ty, n1 - y0), vz = min(tz, n2 - z0);  // voxels of this tile
    const int x0 = xc * ts.cx, x1 = min(x0 + ts.cx, n0);
    const bool valid = iy < vy && iz < vz;
    const long long yz = (long long)(y0 + iy) * n2 + z0 + iz;

    // node plane x (wrapped) into P[buf]; own: the item updates the plane's own nodes
    auto load = [&](int x, int buf, bool own) {
      for (int nl = tid; nl < nodes; nl += nthr) {
        const int ay = nl / row, az = nl - ay * row;
        if (ay > vy || az > vz) continue;
        const int yy = y0 + ay == n1 ? 0 : y0 + ay, zz = z0 + az == n2 ? 0 : z0 + az;
        const long long nd = (long long)x * plane + (long long)yy * n2 + zz;
        const bool mine = FUSED && own && ay < vy && az < vz;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          T v = from_store<T>(dr[i * N + nd]);
          if (FUSED) {
            const T dn = from_store<T>(zr[i * N + nd]) + fb * v;
            if (mine) {
              dnr[i * N + nd] = to_store(dn);
              ur[i * N + nd] = to_store(from_store<T>(ur[i * N + nd]) + fa * v);
            }
            v = dn;
          }
          P[buf][nl][i] = v;
        }
      }
    };
    // q at the tile's nodes of plane x from the corner forces in C; nodes on a face of the item
    // are shared with other items (or, on a periodic axis of one tile, with itself)
    auto emit = [&](int x, int buf, bool face) {
      for (int nl = tid; nl < nodes; nl += nthr) {
        const int ay = nl / row, az = nl - ay * row;
        if (ay > vy || az > vz) continue;
        const int yy = y0 + ay == n1 ? 0 : y0 + ay, zz = z0 + az == n2 ? 0 : z0 + az;
        const long long nd = (long long)x * plane + (long long)yy * n2 + zz;
        const bool lo_y = ay > 0, hi_y = ay < vy, lo_z = az > 0, hi_z = az < vz;
        const int v00 = ay * tz + az;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          T f = T(0);
          if (hi_y && hi_z) f = C[i][v00];
          if (hi_y && lo_z) f += C[3 + i][v00 - 1];
          if (lo_y && hi_z) f += C[6 + i][v00 - tz];
          if (lo_y && lo_z) f += C[9 + i][v00 - tz - 1];
          en += f * (REL ? P[buf][nl][i] - ref[i] : P[buf][nl][i]);
          if (face || !lo_y || !hi_y || !lo_z || !hi_z)
            atomicAdd(&qr[i * N + nd], to_store(f));
          else
            qr[i * N + nd] = to_store(f);
        }
      }
    };

    __syncthreads();  // the previous item's P and C are no longer read
    load(x0, 0, true);
    T D[12][3];    // edge differences (times 1/h_k unless UNIFORM), plus eps_bar when TOTAL
    T pend[4][3];  // corner forces on plane x + 1: [2 dy + dz][component]
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int i = 0; i < 3; ++i) pend[c][i] = T(0);
    int buf = 0;
    for (int x = x0; x < x1; ++x) {
      const int bn = buf == 2 ? 0 : buf + 1;
      unsigned code = 0xaaau;  // every tet cut: zero moduli (threads without a voxel)
      float svf = 1.0f;
      if (valid) {
        code = a.code[(long long)x * plane + yz];
        if (a.scale) svf = a.scale[(long long)x * plane + yz];
      }
      load(x + 1 == n0 ? 0 : x + 1, bn, x + 1 < x1);
      __syncthreads();
      T F1[4][3];
      if (valid) {
        const int b0 = iy * row + iz;
        auto diff = [&](int e, int k, const T (&hi)[3], const T (&lo)[3]) {
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            T v = hi[i] - lo[i];
            if (!UNIFORM) v *= ih[k];
            if (TOTAL) v += Eb[i][k];
            D[e][i] = v;
          }
        };
        // corner c = dx + 2 dy + 4 dz; edges along y and z in plane x + 1 become those of plane x
        const T(&u0)[3] = P[buf][b0];
        const T(&u2)[3] = P[buf][b0 + row];
        const T(&u4)[3] = P[buf][b0 + 1];
        const T(&u6)[3] = P[buf][b0 + row + 1];
        const T(&u1)[3] = P[bn][b0];
        const T(&u3)[3] = P[bn][b0 + row];
        const T(&u5)[3] = P[bn][b0 + 1];
        const T(&u7)[3] = P[bn][b0 + row + 1];
        if (x == x0) {
          diff(cube_edge(0, 1), 1, u2, u0);
          diff(cube_edge(4, 1), 1, u6, u4);
          diff(cube_edge(0, 2), 2, u4, u0);
          diff(cube_edge(2, 2), 2, u6, u2);
        } else {
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            D[cube_edge(0, 1)][i] = D[cube_edge(1, 1)][i];
            D[cube_edge(4, 1)][i] = D[cube_edge(5, 1)][i];
            D[cube_edge(0, 2)][i] = D[cube_edge(1, 2)][i];
            D[cube_edge(2, 2)][i] = D[cube_edge(3, 2)][i];
          }
        }
        diff(cube_edge(0, 0), 0, u1, u0);
        diff(cube_edge(2, 0), 0, u3, u2);
        diff(cube_edge(4, 0), 0, u5, u4);
        diff(cube_edge(6, 0), 0, u7, u6);
        diff(cube_edge(1, 1), 1, u3, u1);
        diff(cube_edge(5, 1), 1, u7, u5);
        diff(cube_edge(1, 2), 2, u5, u1);
        diff(cube_edge(3, 2), 2, u7, u3);
        const T sv = from_store<T>(svf);
        T lp[NPH], mp[NPH];
#pragma unroll
        for (int ph = 0; ph < NPH; ++ph) {
          lp[ph] = a.scale ? l0[ph] * sv : l0[ph];
          mp[ph] = a.scale ? m0[ph] * sv : m0[ph];
        }
        T Te[12][3];
        voxel_tets<T, NPH>(D, Te, code, lp, mp);
        if (SIG) voxel_stress_sums(Te, sg);
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            const T f = corner_force<UNIFORM>(Te, wk, c, i);
            const int cc = (c & 2) + (c >> 2);  // 2 dy + dz
            if (c & 1) F1[cc][i] = f;
            else C[3 * cc + i][tid] = pend[cc][i] + f;
          }
#pragma unroll
        for (int cc = 0; cc < 4; ++cc)
#pragma unroll
          for (int i = 0; i < 3; ++i) pend[cc][i] = F1[cc][i];
      }
      __syncthreads();
      emit(x, buf, x == x0);
      buf = bn;
    }
    __syncthreads();
    if (valid) {
#pragma unroll
      for (int cc = 0; cc < 4; ++cc)
#pragma unroll
        for (int i = 0; i < 3; ++i) C[3 * cc + i][tid] = pend[cc][i];
    }
    __syncthreads();
    emit(x1 == n0 ? 0 : x1, buf, true);
  }
  const double r2 = 1.41421356237309504880;
  const double ws = UNIFORM ? g.h[0] : g.vol_tet;
  double v[7] = {to_double(en), to_double(sg[0]) * ws, to_double(sg[1]) * ws, to_double(sg[2]) * ws,
                 to_double(sg[3]) * ws * r2, to_double(sg[4]) * ws * r2, to_double(sg[5]) * ws * r2};
  double tot[7];
  __syncthreads();
  block_sum<7>(v, red, tot);
  if (tid == 0) {
#pragma unroll
    for (int k = 0; k < 7; ++k) a.partials[((long long)rhs * 7 + k) * a.nparts + blockIdx.x] = tot[k];
  }
}

// Stencil launches of one phase count NPH (2: one interface; 3: two interfaces).  The phase
// counts are instantiated in separate translation units (apply.cu, apply_multi.cu).  FP32: the
// marching kernel, plain stores; FP64 and double-word: the tile kernel on a cleared q.
template <typename T, int NPH>
cudaError_t launch_uncut_nph(const typename Store<T>::type* d, typename Store<T>::type* q,
                             const ApplyArgs& a, int n_rhs, cudaStream_t s) {
  const GridDev& g = a.g;
  const bool uni = g.h[0] == g.h[1] && g.h[1] == g.h[2];
  const bool sig = a.want_sig || a.eps;
  if constexpr (std::is_same<T, float>::value) {
    const int gz = (g.n2 + kTZ - 2) / (kTZ - 1);
    const int gy = (g.n1 + kTY - 2) / (kTY - 1);
    const int gx = (g.n0 + kCX - 1) / kCX;
    dim3 block(kTZ, kTY, 1);
    dim3 grid(gz, gy, gx * n_rhs);
#define XFFT_LAUNCH(TOT, SG, FU)                                                             \
  do {                                                                                       \
    if (uni) k_apply_uncut<TOT, SG, true, FU, NPH><<<grid, block, 0, s>>>(d, q, a, gx);    \
    else k_apply_uncut<TOT, SG, false, FU, NPH><<<grid, block, 0, s>>>(d, q, a, gx);       \
  } while (0)
    if (a.fz) {
      if (sig) XFFT_LAUNCH(false, true, true);
      else XFFT_LAUNCH(false, false, true);
    } else if (a.eps) XFFT_LAUNCH(true, true, false);
    else if (sig) XFFT_LAUNCH(false, true, false);
    else XFFT_LAUNCH(false, false, false);
#undef XFFT_LAUNCH
  } else {
    const TileShape ts = pick_tile(g, n_rhs);
    const dim3 grid(ts.blocks, n_rhs);
    cudaError_t e = cudaMemsetAsync(q, 0, sizeof(*q) * (size_t)n_rhs * a.stride, s);
    if (e != cudaSuccess) return e;
#define XFFT_LAUNCH(TOT, SG, FU)                                                             \
  do {                                                                                       \
    if (uni) k_apply_tile<T, TOT, SG, true, FU, NPH><<<grid, ts.threads, 0, s>>>(d, q, a, ts); \
    else k_apply_tile<T, TOT, SG, false, FU, NPH><<<grid, ts.threads, 0, s>>>(d, q, a, ts);    \
  } while (0)
    if (a.fz) {
      // the fused CG update serves the FP64 solver (not the double-word residuals)
      if constexpr (std::is_same<T, double>::value) {
        if (sig) XFFT_LAUNCH(false, true, true);
        else XFFT_LAUNCH(false, false, true);
      } else {
        return cudaErrorInvalidValue;
      }
    } else if (a.eps) XFFT_LAUNCH(true, true, false);
    else if (sig) XFFT_LAUNCH(false, true, false);
    else XFFT_LAUNCH(false, false, false);
#undef XFFT_LAUNCH
  }
  return cudaGetLastError();
}

#define XFFT_APPLY_INST_NPH(EXT, T, NPH)                                                         \
  EXT template cudaError_t launch_uncut_nph<T, NPH>(const Store<T>::type*, Store<T>::type*,      \
                                                    const ApplyArgs&, int, cudaStream_t);

}  // namespace xfft
