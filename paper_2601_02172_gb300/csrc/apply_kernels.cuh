// Matrix-free stiffness apply of the scaled X-FEM system (eqs. Kapp, b, resVector):
//   q = sum_e Lambda_e^T int_e B~^T C (eps_bar + B~ d_e)        (eps_bar only in TOTAL mode)
// with fused reductions <d, A d> = sum_e int eps(d) : C : eps(d) and int_Y C (eps_bar + grad^s d).
//
// Uncut tets (constant strain, one phase): the FP32 kernel here marches along x in 2.5 D, the FP64
// and double-word one is apply_tile.cuh; both evaluate a voxel's six Kuhn tets by its edges (cube_edge,
// voxel_tet below).
//
// Cut tets: apply_cut.cuh (one thread per cut tet, atomics after the uncut kernel).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "xfft_kernels.h"

namespace xfft {

constexpr int kTZ = 16;  // threads along z (half a warp; a warp covers two y rows)
constexpr int kTY = 16;  // threads along y
#ifndef XFFT_UNCUT_CX
#define XFFT_UNCUT_CX 32
#endif
constexpr int kCX = XFFT_UNCUT_CX;  // output planes per block along x
#ifndef XFFT_UNCUT_MINB
#define XFFT_UNCUT_MINB 2  // resident blocks per SM asked of the FP32 uncut kernel
#endif

// symmetric tensor stored as (00, 11, 22, 12, 02, 01)
template <typename T>
__device__ __forceinline__ T sym_at(const T (&s)[6], int i, int j) {
  if (i == j) return s[i];
  const int k = i + j;  // 1 -> (0,1), 2 -> (0,2), 3 -> (1,2)
  return k == 1 ? s[5] : (k == 2 ? s[4] : s[3]);
}

template <typename T>
__device__ __forceinline__ void mandel_to_tensor(const double* e, T (&E)[6]) {
  const double r = 0.70710678118654752440;
  E[0] = (T)e[0];
  E[1] = (T)e[1];
  E[2] = (T)e[2];
  E[3] = (T)(e[3] * r);
  E[4] = (T)(e[4] * r);
  E[5] = (T)(e[5] * r);
}

template <typename T>
__device__ __forceinline__ void iso_stress(const T (&e)[6], T lam, T mu, T (&s)[6]) {
  const T tr = e[0] + e[1] + e[2];
  const T m2 = mu + mu;
  s[0] = lam * tr + m2 * e[0];
  s[1] = lam * tr + m2 * e[1];
  s[2] = lam * tr + m2 * e[2];
  s[3] = m2 * e[3];
  s[4] = m2 * e[4];
  s[5] = m2 * e[5];
}

template <typename T>
__device__ __forceinline__ T ddot(const T (&s)[6], const T (&e)[6]) {
  return s[0] * e[0] + s[1] * e[1] + s[2] * e[2] + T(2) * (s[3] * e[3] + s[4] * e[4] + s[5] * e[5]);
}

// ---------------------------------------------------------------- uncut stencil
// edge of the cube along axis k starting at corner c (bit k of c is 0): 4 k + the other two bits
__host__ __device__ constexpr int cube_edge(int c, int k) {
  return 4 * k + (k == 0 ? c >> 1 : k == 1 ? (c & 1) | ((c >> 2) << 1) : c & 3);
}

// One Kuhn tet: the displacement-gradient columns of the tet are the node differences D along its
// path 0 -> e_p -> e_p+e_q -> (1,1,1); its tensions sigma e_k are added to (or, as the edge's first
// contribution, stored in) the voxel's edge sums Te.  l, m: lambda, mu of the tet (zero for a cut
// tet) times the voxel scale.
template <typename T, int t>
__device__ __forceinline__ void voxel_tet(const T (&D)[12][3], T (&Te)[12][3], T l, T m) {
  constexpr int p = perm_p(t), q = perm_q(t), r = perm_r(t);
  constexpr int E[3] = {p == 0 ? cube_edge(0, 0) : q == 0 ? cube_edge(1 << p, 0) : cube_edge(6, 0),
                        p == 1 ? cube_edge(0, 1) : q == 1 ? cube_edge(1 << p, 1) : cube_edge(5, 1),
                        p == 2 ? cube_edge(0, 2) : q == 2 ? cube_edge(1 << p, 2) : cube_edge(3, 2)};
  // the first tet that reaches a shared edge stores; p edges are shared by tets 2p and 2p + 1
  constexpr bool first_r = t == 0 || t == 1 || t == 3;
  const T tr = D[E[0]][0] + D[E[1]][1] + D[E[2]][2];
  const T s01 = D[E[0]][1] + D[E[1]][0], s02 = D[E[0]][2] + D[E[2]][0], s12 = D[E[1]][2] + D[E[2]][1];
  const T m2 = m + m;
  const T lt = l * tr;
  const T t01 = m * s01, t02 = m * s02, t12 = m * s12;
  // sigma of the tet (times the common factor of l and m): column k is its tension on the edge
  // along k, up to the weight w_k that the corner forces apply
  const T S[3][3] = {{lt + m2 * D[E[0]][0], t01, t02}, {t01, lt + m2 * D[E[1]][1], t12}, {t02, t12, lt + m2 * D[E[2]][2]}};
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const bool st = k == p ? (t & 1) == 0 : k == q ? true : first_r;
      Te[E[k]][i] = st ? S[k][i] : Te[E[k]][i] + S[k][i];
    }
}

// The six tets of a voxel with codes `code`; lp, mp: phase moduli times the voxel scale
template <typename T, int NPH>
__device__ __forceinline__ void voxel_tets(const T (&D)[12][3], T (&Te)[12][3], unsigned code, const T (&lp)[NPH],
                                           const T (&mp)[NPH]) {
  const auto modulus = [&](int t, const T (&v)[NPH]) {
    const unsigned cd = (code >> (2 * t)) & 3u;
    T r = cd == 0u ? v[0] : T(0);
    if (cd == 1u) r = v[1];
    if (NPH > 2 && cd == 3u) r = v[NPH - 1];
    return r;
  };
  voxel_tet<T, 0>(D, Te, modulus(0, lp), modulus(0, mp));
  voxel_tet<T, 1>(D, Te, modulus(1, lp), modulus(1, mp));
  voxel_tet<T, 2>(D, Te, modulus(2, lp), modulus(2, mp));
  voxel_tet<T, 3>(D, Te, modulus(3, lp), modulus(3, mp));
  voxel_tet<T, 4>(D, Te, modulus(4, lp), modulus(4, mp));
  voxel_tet<T, 5>(D, Te, modulus(5, lp), modulus(5, mp));
}

// Stress sums of a voxel from its edge sums: int sigma_ik is component i summed over the edges
// along k, up to the weight applied after the block sums.
template <typename T>
__device__ __forceinline__ void voxel_stress_sums(const T (&Te)[12][3], T (&sg)[6]) {
  const auto sum4 = [&](int k, int i) {
    return (Te[4 * k][i] + Te[4 * k + 1][i]) + (Te[4 * k + 2][i] + Te[4 * k + 3][i]);
  };
  sg[0] += sum4(0, 0);
  sg[1] += sum4(1, 1);
  sg[2] += sum4(2, 2);
  sg[3] += sum4(1, 2);
  sg[4] += sum4(0, 2);
  sg[5] += sum4(0, 1);
}

// Force component i on corner c (bits x = 1, y = 2, z = 4): an edge pulls its end corner and pushes
// its start corner.
template <bool UNIFORM, typename T>
__device__ __forceinline__ T corner_force(const T (&Te)[12][3], const T (&wk)[3], int c, int i) {
  const T ex = Te[cube_edge(c & 6, 0)][i], ey = Te[cube_edge(c & 5, 1)][i], ez = Te[cube_edge(c & 3, 2)][i];
  T f;
  if (UNIFORM) {
    f = (c & 1) ? ex : -ex;
    f = (c & 2) ? f + ey : f - ey;
    f = (c & 4) ? f + ez : f - ez;
  } else {
    f = (c & 1) ? ex * wk[0] : ex * -wk[0];
    f = f + ey * ((c & 2) ? wk[1] : -wk[1]);
    f = f + ez * ((c & 4) ? wk[2] : -wk[2]);
  }
  return f;
}

// Moduli factors of the edge form: uniform voxels use raw differences with |T| / h^2 in the moduli;
// otherwise differences carry 1/h_k and corner forces the weights |T| / h_k.
template <typename T, bool UNIFORM, int NPH>
__device__ __forceinline__ void edge_moduli(const GridDev& g, const PhaseDev& ph, T (&l0)[NPH], T (&m0)[NPH]) {
  const double w = UNIFORM ? g.vol_tet / (g.h[0] * g.h[0]) : 1.0;
#pragma unroll
  for (int p = 0; p < NPH; ++p) {
    l0[p] = (T)(ph.lam[p] * w);
    m0[p] = (T)(ph.mu[p] * w);
  }
}
// eps_bar as it adds to the differences (raw differences carry a factor h)
template <typename T, bool UNIFORM>
__device__ __forceinline__ void edge_strain(const GridDev& g, const double* e, T (&Eb)[3][3]) {
  const double rs = 0.70710678118654752440;
  const double sc = UNIFORM ? g.h[0] : 1.0;
  Eb[0][0] = (T)(e[0] * sc);
  Eb[1][1] = (T)(e[1] * sc);
  Eb[2][2] = (T)(e[2] * sc);
  Eb[1][2] = Eb[2][1] = (T)(e[3] * rs * sc);
  Eb[0][2] = Eb[2][0] = (T)(e[4] * rs * sc);
  Eb[0][1] = Eb[1][0] = (T)(e[5] * rs * sc);
}

// The FP32 stencil.  A block of kTZ x kTY (16 x 16) threads owns one voxel column each (y, z), with a
// halo row and column on the low side, and walks along x; node planes of d are staged in shared
// memory one step ahead, forces on the plane's nodes are combined in shared memory and forces on
// the next plane stay in registers, so every node force is written once with a plain store.
//
// What bounds it: instruction issue, then memory (78 bytes per voxel and right-hand side with the
// fused update).  The voxel's twelve edges carry all its differences (those of the next plane are
// kept: 24 subtractions per voxel) and its tension sums; cut tets take zero moduli by selects instead
// of six branches with their own re-convergence; corner forces cross threads as 16-byte vectors
// (three stores and three loads per voxel instead of twelve shuffles and twelve accesses).
template <bool TOTAL, bool SIG, bool UNIFORM, bool FUSED, int NPH>
__global__ void __launch_bounds__(kTZ* kTY, XFFT_UNCUT_MINB)
    k_apply_uncut(const float* __restrict__ d, float* __restrict__ q, const ApplyArgs a, int nxchunks) {
  const int tz = threadIdx.x, ty = threadIdx.y;
  const int tid = tz + kTZ * ty;
  const int rhs = blockIdx.z / nxchunks;
  const int xc = blockIdx.z - rhs * nxchunks;
  if (a.active && !a.active[rhs]) return;
  if (a.units_uncut && tid == 0 && blockIdx.x == 0 && blockIdx.y == 0 && xc == 0)
    atomicAdd(a.units_uncut, 1ULL);
  const GridDev& g = a.g;
  const int n0 = g.n0, n1 = g.n1, n2 = g.n2;
  // element indices inside a right-hand side fit 32 bits (3 N <= 3 2^28)
  const unsigned N = (unsigned)g.N, plane = (unsigned)(n1 * n2);
  const int z0 = blockIdx.x * (kTZ - 1), y0 = blockIdx.y * (kTY - 1), x0 = xc * kCX;
  const int x1 = min(x0 + kCX, n0);
  const float* dr = d + rhs * a.stride;
  float* qr = q + rhs * a.stride;

  __shared__ float4 P[2][kTY + 1][kTZ + 1];  // node planes
  __shared__ float4 C[3][kTY][kTZ];          // forces on the corners (dy, dz) = (0, 1), (1, 0), (1, 1)

  constexpr int kPlaneNodes = (kTY + 1) * (kTZ + 1);
  int ld_slot[2];
  unsigned ld_off[2];
  bool slot_own[2];  // the block updates the plane nodes with 1 <= iy < kTY, 1 <= iz < kTZ
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int lin = tid + k * kTZ * kTY;
    ld_slot[k] = lin < kPlaneNodes ? lin : -1;
    const int iy = lin / (kTZ + 1), iz = lin - iy * (kTZ + 1);
    const int yy = ((y0 - 1 + iy) % n1 + n1) % n1;
    const int zz = ((z0 - 1 + iz) % n2 + n2) % n2;
    ld_off[k] = yy * n2 + zz;
    slot_own[k] = FUSED && ld_slot[k] >= 0 && iy >= 1 && iy <= kTY - 1 && iz >= 1 && iz <= kTZ - 1 &&
                  y0 - 1 + iy < n1 && z0 - 1 + iz < n2;
  }
  const int yg = y0 - 1 + ty, zg = z0 - 1 + tz;
  const int yv = (yg % n1 + n1) % n1, zv = (zg % n2 + n2) % n2;
  const bool own = ty >= 1 && tz >= 1 && yg < n1 && zg < n2;

  float ih[3], wk[3], l0[NPH], m0[NPH], Eb[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    ih[k] = (float)(1.0 / g.h[k]);
    wk[k] = (float)(g.vol_tet / g.h[k]);
  }
  edge_moduli<float, UNIFORM, NPH>(g, a.ph, l0, m0);
  if (TOTAL) edge_strain<float, UNIFORM>(g, a.eps + 6 * rhs, Eb);

  // fused CG update: d_new = z + beta d_old, u += alpha d_old
  const float* zr = FUSED ? static_cast<const float*>(a.fz) + rhs * a.stride : nullptr;
  float* dnr = FUSED ? static_cast<float*>(a.fdnew) + rhs * a.stride : nullptr;
  float* ur = FUSED ? static_cast<float*>(a.fu) + rhs * a.stride : nullptr;
  const float fa = FUSED ? (float)a.st[rhs].alpha : 0.0f;
  const float fb = FUSED ? (float)a.st[rhs].beta : 0.0f;

  // Two-stage plane pipeline: fetch() issues the global loads of a node plane into registers,
  // commit() (one step later, after the arithmetic of the current step was issued) forms the
  // fused update, stores the block's own nodes and fills the shared-memory plane.
  float pf[2][9];  // per load slot: z (or d) 0..2, d_old 3..5, u 6..8
  unsigned pf_nd[2] = {0, 0};
  bool pf_own[2] = {false, false};
  auto fetch = [&](int xp, bool own_plane) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      pf_own[k] = false;
      if (ld_slot[k] >= 0) {
        const unsigned nd = xp * plane + ld_off[k];
        pf_nd[k] = nd;
        if (FUSED) {
          pf[k][0] = zr[nd];
          pf[k][1] = zr[N + nd];
          pf[k][2] = zr[2 * N + nd];
          pf[k][3] = dr[nd];
          pf[k][4] = dr[N + nd];
          pf[k][5] = dr[2 * N + nd];
          pf_own[k] = own_plane && slot_own[k];
          if (pf_own[k]) {
            pf[k][6] = ur[nd];
            pf[k][7] = ur[N + nd];
            pf[k][8] = ur[2 * N + nd];
          }
        } else {
          pf[k][0] = dr[nd];
          pf[k][1] = dr[N + nd];
          pf[k][2] = dr[2 * N + nd];
        }
      }
    }
  };
  auto commit = [&](int buf) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (ld_slot[k] >= 0) {
        float4 v;
        if (FUSED) {
          v.x = pf[k][0] + fb * pf[k][3];
          v.y = pf[k][1] + fb * pf[k][4];
          v.z = pf[k][2] + fb * pf[k][5];
          if (pf_own[k]) {
            const unsigned nd = pf_nd[k];
            dnr[nd] = v.x;
            dnr[N + nd] = v.y;
            dnr[2 * N + nd] = v.z;
            ur[nd] = pf[k][6] + fa * pf[k][3];
            ur[N + nd] = pf[k][7] + fa * pf[k][4];
            ur[2 * N + nd] = pf[k][8] + fa * pf[k][5];
          }
        } else {
          v.x = pf[k][0];
          v.y = pf[k][1];
          v.z = pf[k][2];
        }
        v.w = 0.0f;
        (&P[buf][0][0])[ld_slot[k]] = v;
      }
    }
  };

  float D[12][3];    // edge differences (times 1/h_k unless UNIFORM), plus eps_bar when TOTAL
  float pend[4][3];  // corner forces on plane x + 1: [2 dy + dz][component]
  float uo[4][3];    // plane x at the corners [2 dy + dz]
  auto corners = [&](int buf, float (&u)[4][3]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float4 v = P[buf][ty + (c >> 1)][tz + (c & 1)];
      u[c][0] = v.x;
      u[c][1] = v.y;
      u[c][2] = v.z;
    }
  };
  auto diff = [&](int e, int k, const float (&hi)[3], const float (&lo)[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      float v = hi[i] - lo[i];
      if (!UNIFORM) v *= ih[k];
      if (TOTAL) v += Eb[i][k];
      D[e][i] = v;
    }
  };

  float en = 0.0f;
  float sg[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  const int xfirst = ((x0 - 1) % n0 + n0) % n0;
  fetch(xfirst, false);
  commit(0);
  fetch(xfirst + 1 == n0 ? 0 : xfirst + 1, x0 < x1);
  // the voxel's phase code and modulus scale are loaded one x step ahead as well
  const unsigned yz = yv * n2 + zv;
  unsigned nx_code = a.code[xfirst * plane + yz];
  float nx_scale = a.scale ? a.scale[xfirst * plane + yz] : 1.0f;
  __syncthreads();
  corners(0, uo);
  diff(cube_edge(0, 1), 1, uo[2], uo[0]);
  diff(cube_edge(4, 1), 1, uo[3], uo[1]);
  diff(cube_edge(0, 2), 2, uo[1], uo[0]);
  diff(cube_edge(2, 2), 2, uo[3], uo[2]);
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int i = 0; i < 3; ++i) pend[c][i] = 0.0f;
  int xw = xfirst;  // the wrapped voxel index x0 - 1 + s, advanced without a division per step
  for (int s = 0; s <= x1 - x0; ++s, xw = xw + 1 >= n0 ? xw + 1 - n0 : xw + 1) {
    const unsigned code = nx_code;
    const float sv = nx_scale;
    commit((s + 1) & 1);  // plane x0 + s
    if (s + 1 <= x1 - x0) {
      const int x1w = xw + 1 >= n0 ? xw + 1 - n0 : xw + 1;  // voxel of the next step
      const int xn = xw + 2 >= n0 ? xw + 2 - n0 : xw + 2;  // plane x0 + s + 1
      fetch(xn, x0 + s + 1 < x1);
      nx_code = a.code[x1w * plane + yz];
      if (a.scale) nx_scale = a.scale[x1w * plane + yz];
    }
    __syncthreads();
    float un[4][3];
    corners((s + 1) & 1, un);
    diff(cube_edge(0, 0), 0, un[0], uo[0]);
    diff(cube_edge(2, 0), 0, un[2], uo[2]);
    diff(cube_edge(4, 0), 0, un[1], uo[1]);
    diff(cube_edge(6, 0), 0, un[3], uo[3]);
    diff(cube_edge(1, 1), 1, un[2], un[0]);
    diff(cube_edge(5, 1), 1, un[3], un[1]);
    diff(cube_edge(1, 2), 2, un[1], un[0]);
    diff(cube_edge(3, 2), 2, un[3], un[2]);
    float Te[12][3];
    {
      float lp[NPH], mp[NPH];
#pragma unroll
      for (int ph = 0; ph < NPH; ++ph) {
        lp[ph] = l0[ph] * sv;
        mp[ph] = m0[ph] * sv;
      }
      // warps whose voxels each lie in one phase (most of them) need no selects
      const bool one = code == 0u || code == 0x555u || (NPH > 2 && code == 0xfffu);
      if (__all_sync(0xffffffffu, one)) {
        const float l = code == 0u ? lp[0] : NPH > 2 && code == 0xfffu ? lp[NPH - 1] : lp[1];
        const float m = code == 0u ? mp[0] : NPH > 2 && code == 0xfffu ? mp[NPH - 1] : mp[1];
        voxel_tet<float, 0>(D, Te, l, m);
        voxel_tet<float, 1>(D, Te, l, m);
        voxel_tet<float, 2>(D, Te, l, m);
        voxel_tet<float, 3>(D, Te, l, m);
        voxel_tet<float, 4>(D, Te, l, m);
        voxel_tet<float, 5>(D, Te, l, m);
      } else {
        voxel_tets<float, NPH>(D, Te, code, lp, mp);
      }
    }
    if (SIG && own && s >= 1) voxel_stress_sums(Te, sg);
    float f0[3];  // force on the thread's own node (dy, dz) = (0, 0)
#pragma unroll
    for (int cc = 0; cc < 4; ++cc) {
      const int c = (cc & 2) + 4 * (cc & 1);  // corner on plane x
      float f[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        f[i] = pend[cc][i] + corner_force<UNIFORM>(Te, wk, c, i);
        pend[cc][i] = corner_force<UNIFORM>(Te, wk, c + 1, i);
      }
      if (cc == 0) {
        f0[0] = f[0];
        f0[1] = f[1];
        f0[2] = f[2];
      } else {
        C[cc - 1][ty][tz] = make_float4(f[0], f[1], f[2], 0.0f);
      }
    }
    __syncthreads();
    if (own && s >= 1) {
      const float4 fz = C[0][ty][tz - 1], fy = C[1][ty - 1][tz], fyz = C[2][ty - 1][tz - 1];
      const unsigned nd = xw * plane + yz;
      const float q0 = (f0[0] + fz.x) + (fy.x + fyz.x);
      const float q1 = (f0[1] + fz.y) + (fy.y + fyz.y);
      const float q2 = (f0[2] + fz.z) + (fy.z + fyz.z);
      qr[nd] = q0;
      qr[N + nd] = q1;
      qr[2 * N + nd] = q2;
      en += q0 * uo[0][0] + q1 * uo[0][1] + q2 * uo[0][2];  // <d, q> of this node
    }
    // plane x + 1 becomes plane x
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      D[cube_edge(0, 1)][i] = D[cube_edge(1, 1)][i];
      D[cube_edge(4, 1)][i] = D[cube_edge(5, 1)][i];
      D[cube_edge(0, 2)][i] = D[cube_edge(1, 2)][i];
      D[cube_edge(2, 2)][i] = D[cube_edge(3, 2)][i];
#pragma unroll
      for (int c = 0; c < 4; ++c) uo[c][i] = un[c][i];
    }
  }
  double tot[7] = {};
  if (SIG) {
    __shared__ double red[7 * 32];
    const double ws = UNIFORM ? g.h[0] : g.vol_tet, r2 = 1.41421356237309504880;
    const double v[7] = {(double)en, sg[0] * ws, sg[1] * ws, sg[2] * ws, sg[3] * ws * r2, sg[4] * ws * r2, sg[5] * ws * r2};
    block_sum<7>(v, red, tot);
  } else {
    __shared__ float red1[kTZ * kTY];
    tot[0] = block_sum1<float>(en, red1);
  }
  if (tid == 0) {
    const int bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * xc);
#pragma unroll
    for (int k = 0; k < 7; ++k) a.partials[((long long)rhs * 7 + k) * a.nparts + bid] = tot[k];
  }
}

}  // namespace xfft
