// FP64 cut-tet apply from reduced element records (FP64 solvers).
//
// What bounds it: the FP64 pipe (2 FMAs per SM and clock), so the record is chosen for the fewest
// operations per tet and right-hand side.  With es the (constant) strain of the standard part and w
// the enriched vertex values, the element's energy is a quadratic form in (es, w); summed over the two
// sides s (apply_cut.cuh's notation, v_sb = (m.c)_s g_b + m_sb gamma_s):
//   stress      sigma = lam tr(es) I + 2 mu es + (sum_b w_b . l_b) I + sym(sum_b w_b (x) p_b),
//               lam, mu = sum_s V_s (lambda_s, mu_s), l_b = sum_s lambda_s v_sb, p_b = sum_s 2 mu_s v_sb
//   std forces  q_a  = sigma g_a
//   enr forces  q~_b = tr(es) l_b + es p_b + sum_a K_ba w_a, K the 12 x 12 enriched block
// with D0^-1/2 of every enriched DOF folded into l, p and K.  About 320 operations instead of the 790
// of the moment form (both sides' tensors, five stresses): 12 x 12 K as a symmetric product 144,
// l and p 96, strains, forces and sums the rest.  The record is 128 reals against 68, stored
// [group of 32 tets][real][tet] so that a warp's loads are whole lines; right-hand sides of one
// group run next to each other and read it from L2.
//
// Six right-hand sides at 64^3 with 115,022 cut tets (ncu): 1.21 -> 0.44 ms, the FP64 pipe 92 %
// active (360 FP64 instructions per tet, conversions and addresses included); in the solver with the
// fused stencil 0.201 -> 0.074 ms per right-hand side.  16^3, one right-hand side (2,094 tets): 58 ->
// 19 us, one warp per block over 66 SMs instead of 17 blocks of 128.
#pragma once

#include "apply_kernels.cuh"

namespace xfft {

// record: 0, 1: lam, mu; 2 + 3 b + x: l_b; 14 + 9 b + 3 x + y: p_b[y] / 2 times D0^-1/2 of (b, x);
// 50 + k: upper triangle of K, row by row, DOFs 3 b + x
constexpr int kEl = 128;
constexpr int kElL = 2, kElP = 14, kElK = 50;

// one warp per block, blocks loop over the groups of 32 tets
constexpr int kElBlocksMax = 2432;

template <bool TOTAL, bool SIG>
__global__ void __launch_bounds__(32, 14)
    k_apply_cut_el(const double* __restrict__ d, double* __restrict__ q, const CutData cd, const ApplyArgs a,
                   int n_rhs) {
  const int rhs = blockIdx.x % n_rhs, blk = blockIdx.x / n_rhs, nblk = gridDim.x / n_rhs;
  if (a.active && !a.active[rhs]) return;
  const int lane = threadIdx.x;
  if (a.units_cut && lane == 0 && blk == 0) atomicAdd(a.units_cut, 1ULL);
  const long long N = a.g.N;
  const int nX = a.nX, ncut = cd.ncut;
  const double* dr = d + rhs * a.stride;
  double* qr = q + rhs * a.stride;
  const double ih[3] = {1.0 / a.g.h[0], 1.0 / a.g.h[1], 1.0 / a.g.h[2]};
  double E[6];
  if (TOTAL) mandel_to_tensor(a.eps + 6 * rhs, E);
  double en = 0.0, sg[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int grp = blk; 32 * grp < ncut; grp += nblk) {
    const int e = 32 * grp + lane;
    if (e >= ncut) break;
    const int t = __ldg(cd.ip + 9 * ncut + e);
    const int4 n4 = __ldg(cd.n4 + e), e4 = __ldg(cd.e4 + e);
    const double* R = cd.el + ((long long)grp * kEl) * 32 + lane;
    const int nd[4] = {n4.x, n4.y, n4.z, n4.w}, ej[4] = {e4.x, e4.y, e4.z, e4.w};
    double w[12];
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int x = 0; x < 3; ++x) w[3 * b + x] = dr[3 * N + (long long)x * nX + ej[b]];
    // path differences along the axes p, q, r of the Kuhn tet, put in axis order with selects
    const int p = perm_p(t), q1 = perm_q(t);
    double H[3][3];  // H[k][i] = d u_i / d x_k
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double u0 = dr[i * N + nd[0]], u1 = dr[i * N + nd[1]], u2 = dr[i * N + nd[2]], u3 = dr[i * N + nd[3]];
      const double dp = u1 - u0, dq = u2 - u1, dz = u3 - u2;
#pragma unroll
      for (int k = 0; k < 3; ++k) H[k][i] = (k == p ? dp : k == q1 ? dq : dz) * ih[k];
    }
    // twice the standard strain of d (00, 11, 22, 12, 02, 01); es adds eps_bar in TOTAL mode
    const double d2[6] = {H[0][0] + H[0][0], H[1][1] + H[1][1], H[2][2] + H[2][2],
                          H[1][2] + H[2][1], H[0][2] + H[2][0], H[0][1] + H[1][0]};
    double e2[6], tr = H[0][0] + H[1][1] + H[2][2];
#pragma unroll
    for (int k = 0; k < 6; ++k) e2[k] = TOTAL ? d2[k] + (E[k] + E[k]) : d2[k];
    if (TOTAL) tr += E[0] + E[1] + E[2];
    const double lam = __ldg(R), mu = __ldg(R + 32);
    double qe[12], twl = lam * tr, M[3][3];
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        const double l = __ldg(R + 32 * (kElL + 3 * b + x));
        twl += w[3 * b + x] * l;
        double f = tr * l;
#pragma unroll
        for (int y = 0; y < 3; ++y) {
          const double pv = __ldg(R + 32 * (kElP + 9 * b + 3 * x + y));
          const int s = x == y ? x : 6 - x - y;  // (1,2) 3, (0,2) 4, (0,1) 5
          f += e2[s] * pv;
          M[x][y] = b == 0 ? w[x] * pv : M[x][y] + w[3 * b + x] * pv;
        }
        qe[3 * b + x] = f;
      }
    double S[6];
#pragma unroll
    for (int k = 0; k < 3; ++k) S[k] = twl + mu * e2[k] + (M[k][k] + M[k][k]);
    S[3] = mu * e2[3] + (M[1][2] + M[2][1]);
    S[4] = mu * e2[4] + (M[0][2] + M[2][0]);
    S[5] = mu * e2[5] + (M[0][1] + M[1][0]);
    // enriched block
    {
      const double* K = R + 32 * kElK;
#pragma unroll
      for (int i = 0; i < 12; ++i)
#pragma unroll
        for (int j = i; j < 12; ++j) {
          const double k = __ldg(K + 32 * (12 * i - (i * (i - 1)) / 2 + (j - i)));
          qe[i] += k * w[j];
          if (j != i) qe[j] += k * w[i];
        }
    }
    // <d, q>: sigma : eps(d) + sum_b w_b . q~_b
    double s = 0.5 * (S[0] * d2[0] + S[1] * d2[1] + S[2] * d2[2]) + S[3] * d2[3] + S[4] * d2[4] + S[5] * d2[5];
#pragma unroll
    for (int i = 0; i < 12; ++i) s += w[i] * qe[i];
    en += s;
    if (SIG) {
#pragma unroll
      for (int k = 0; k < 6; ++k) sg[k] += S[k];
    }
    // standard forces: tension sigma e_k / h_k on the path edges
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double c[3] = {(i == 0 ? S[0] : i == 1 ? S[5] : S[4]) * ih[0], (i == 0 ? S[5] : i == 1 ? S[1] : S[3]) * ih[1],
                           (i == 0 ? S[4] : i == 1 ? S[3] : S[2]) * ih[2]};
      const double tp = p == 0 ? c[0] : p == 1 ? c[1] : c[2];
      const double tq = q1 == 0 ? c[0] : q1 == 1 ? c[1] : c[2];
      const int r1 = 3 - p - q1;
      const double tz = r1 == 0 ? c[0] : r1 == 1 ? c[1] : c[2];
      atomicAdd(&qr[i * N + nd[0]], -tp);
      atomicAdd(&qr[i * N + nd[1]], tp - tq);
      atomicAdd(&qr[i * N + nd[2]], tq - tz);
      atomicAdd(&qr[i * N + nd[3]], tz);
    }
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int x = 0; x < 3; ++x) atomicAdd(&qr[3 * N + (long long)x * nX + ej[b]], qe[3 * b + x]);
  }
  const double r2 = 1.41421356237309504880;
  double v[7] = {en, sg[0], sg[1], sg[2], sg[3] * r2, sg[4] * r2, sg[5] * r2};
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    const double s = SIG || k == 0 ? warp_sum(v[k]) : 0.0;
    if (lane == 0) a.partials[((long long)rhs * 7 + k) * a.nparts + a.part_offset_cut + blk] = s;
  }
}

}  // namespace xfft
