// Per-tet geometry of the X-FEM setup, shared by the setup kernels and a host-compiled check
// (the functions are __host__ __device__): classification of a tet against K level sets, the
// exact moments of the two sides of a cut tet, and the cut tet's scaled element matrix formed
// from them (the optional cache of the FP32 iterations).
#pragma once

#include <math.h>

#include "xfft_kernels.h"

#define XFFT_HD __host__ __device__

namespace xfft {

// Classification of tet (a, b, c, d vertex values per level set): returns the 2-bit code and,
// for a cut tet, the minus / plus phases; *two is set if a second interface cuts the tet.
XFFT_HD inline unsigned classify_tet(const double* const* Lv, int nL, int* pm, int* pp,
                                        bool* two) {
  int first = nL;
  bool cut = false;
  for (int l = 0; l < nL; ++l) {
    const double* x = Lv[l];
    const double mn = fmin(fmin(x[0], x[1]), fmin(x[2], x[3]));
    const double mx = fmax(fmax(x[0], x[1]), fmax(x[2], x[3]));
    if (first == nL) {
      if (mn < 0.0) {  // minus phase if any vertex is negative
        first = l;
        cut = mx > 0.0;
        *pp = nL;
      }
    } else if (cut && mn < 0.0) {
      if (mx > 0.0) *two = true;
      if (*pp == nL) *pp = l;
    }
  }
  *pm = first;
  return cut ? kCodeCut : phase_code(first);
}

// ---------------------------------------------------------------- side moments
struct Moments {
  double m[4];
  double M[10];
};

// Add the moments of a sub-tetrahedron of volume v: int N_b = v/4 S_b and int N_b N_c =
// v/20 (pp_bc + S_b S_c), where S_b = sum_v beta_vb and pp_bc = sum_v beta_vb beta_vc over its
// vertices' parent barycentric coordinates beta_v.  Arguments: S, then the packed pp.
XFFT_HD inline void add_subtet(Moments& acc, double v, double s0, double s1, double s2, double s3, double p00,
                               double p01, double p02, double p03, double p11, double p12, double p13, double p22,
                               double p23, double p33) {
  const double v4 = 0.25 * v, v20 = 0.05 * v;
  acc.m[0] += v4 * s0;
  acc.m[1] += v4 * s1;
  acc.m[2] += v4 * s2;
  acc.m[3] += v4 * s3;
  acc.M[0] += v20 * (p00 + s0 * s0);
  acc.M[1] += v20 * (p01 + s0 * s1);
  acc.M[2] += v20 * (p02 + s0 * s2);
  acc.M[3] += v20 * (p03 + s0 * s3);
  acc.M[4] += v20 * (p11 + s1 * s1);
  acc.M[5] += v20 * (p12 + s1 * s2);
  acc.M[6] += v20 * (p13 + s1 * s3);
  acc.M[7] += v20 * (p22 + s2 * s2);
  acc.M[8] += v20 * (p23 + s2 * s3);
  acc.M[9] += v20 * (p33 + s3 * s3);
}

XFFT_HD inline double pick4(const double L[4], int i) { return i < 2 ? (i ? L[1] : L[0]) : (i == 3 ? L[3] : L[2]); }

// Moments of side s (+1: s L_h >= 0) of a cut tet with nodal values L, its vertices in the order
// perm (vertex perm[k] of the tet is vertex k here), which brings every cut to one of three forms:
//   one strictly positive vertex (first):  tet of it and the edge points to the others
//   one strictly negative vertex (first):  prism (other three) -> (their edge points to it)
//   two and two (positive ones first):     prism (a1, x11, x12) -> (a2, x21, x22)
// An edge point is (1 - t) v + t w with L = 0 there (a vertex with L = 0 is its own edge point).  The
// prisms split into the three tets of consecutive points; the volumes |det beta| are products of the
// edge coordinates.  Nothing is indexed by data, so on the GPU all of it stays in registers.
XFFT_HD inline void side_moments_ordered(const double L[4], int s, double vol, Moments& out, int perm[4]) {
  for (int c = 0; c < 4; ++c) out.m[c] = 0.0;
  for (int c = 0; c < 10; ++c) out.M[c] = 0.0;
  const double x0 = s * L[0], x1 = s * L[1], x2 = s * L[2], x3 = s * L[3];
  const int np = (x0 > 0.0) + (x1 > 0.0) + (x2 > 0.0) + (x3 > 0.0);
  const int nq = (x0 < 0.0) + (x1 < 0.0) + (x2 < 0.0) + (x3 < 0.0);
  if (np == 1 || nq == 1) {
    const double g = np == 1 ? 1.0 : -1.0;  // the lone vertex is the one with g x > 0
    const int a = g * x0 > 0.0 ? 0 : g * x1 > 0.0 ? 1 : g * x2 > 0.0 ? 2 : 3;
    perm[0] = a;
    perm[1] = a == 0 ? 1 : 0;
    perm[2] = a <= 1 ? 2 : 1;
    perm[3] = a <= 2 ? 3 : 2;
    const double la = pick4(L, a), l0 = pick4(L, perm[1]), l1 = pick4(L, perm[2]), l2 = pick4(L, perm[3]);
    if (np == 1) {
      const double t0 = la / (la - l0), t1 = la / (la - l1), t2 = la / (la - l2);
      const double u0 = 1.0 - t0, u1 = 1.0 - t1, u2 = 1.0 - t2;
      add_subtet(out, t0 * t1 * t2 * vol, 1.0 + u0 + u1 + u2, t0, t1, t2, 1.0 + u0 * u0 + u1 * u1 + u2 * u2, u0 * t0,
                 u1 * t1, u2 * t2, t0 * t0, 0.0, 0.0, t1 * t1, 0.0, t2 * t2);
    } else {
      const double t0 = l0 / (l0 - la), t1 = l1 / (l1 - la), t2 = l2 / (l2 - la);
      const double u0 = 1.0 - t0, u1 = 1.0 - t1, u2 = 1.0 - t2;
      const double c0 = u0 * t0, c1 = u1 * t1, c2 = u2 * t2;
      add_subtet(out, t0 * vol, t0, 1.0 + u0, 1.0, 1.0, t0 * t0, c0, 0.0, 0.0, 1.0 + u0 * u0, 0.0, 0.0, 1.0, 0.0, 1.0);
      add_subtet(out, u0 * t1 * vol, t0 + t1, u0, 1.0 + u1, 1.0, t0 * t0 + t1 * t1, c0, c1, 0.0, u0 * u0, 0.0, 0.0,
                 1.0 + u1 * u1, 0.0, 1.0);
      add_subtet(out, u0 * u1 * t2 * vol, t0 + t1 + t2, u0, u1, 1.0 + u2, t0 * t0 + t1 * t1 + t2 * t2, c0, c1, c2,
                 u0 * u0, 0.0, 0.0, u1 * u1, 0.0, 1.0 + u2 * u2);
    }
  } else {
    perm[0] = x0 > 0.0 ? 0 : x1 > 0.0 ? 1 : 2;
    perm[1] = x3 > 0.0 ? 3 : x2 > 0.0 ? 2 : 1;
    perm[2] = x0 < 0.0 ? 0 : x1 < 0.0 ? 1 : 2;
    perm[3] = x3 < 0.0 ? 3 : x2 < 0.0 ? 2 : 1;
    const double a1 = pick4(L, perm[0]), a2 = pick4(L, perm[1]), b1 = pick4(L, perm[2]), b2 = pick4(L, perm[3]);
    const double t11 = a1 / (a1 - b1), t12 = a1 / (a1 - b2), t21 = a2 / (a2 - b1), t22 = a2 / (a2 - b2);
    const double u11 = 1.0 - t11, u12 = 1.0 - t12, u21 = 1.0 - t21, u22 = 1.0 - t22;
    const double c11 = u11 * t11, c12 = u12 * t12, c21 = u21 * t21, c22 = u22 * t22;
    add_subtet(out, t11 * t12 * vol, 1.0 + u11 + u12, 1.0, t11, t12, 1.0 + u11 * u11 + u12 * u12, 0.0, c11, c12, 1.0,
               0.0, 0.0, t11 * t11, 0.0, t12 * t12);
    add_subtet(out, u11 * t12 * t21 * vol, u11 + u12, 1.0 + u21, t11 + t21, t12, u11 * u11 + u12 * u12, 0.0, c11, c12,
               1.0 + u21 * u21, c21, 0.0, t11 * t11 + t21 * t21, 0.0, t12 * t12);
    add_subtet(out, u12 * t21 * t22 * vol, u12, 1.0 + u21 + u22, t21, t12 + t22, u12 * u12, 0.0, 0.0, c12,
               1.0 + u21 * u21 + u22 * u22, c21, c22, t21 * t21, 0.0, t12 * t12 + t22 * t22);
  }
}

// the same in the tet's own vertex order
XFFT_HD inline void side_moments(const double L[4], int s, double vol, Moments& out) {
  Moments o;
  int perm[4];
  side_moments_ordered(L, s, vol, o, perm);
  for (int b = 0; b < 4; ++b) {
    out.m[perm[b]] = o.m[b];
    for (int c = b; c < 4; ++c) out.M[midx(perm[b], perm[c])] = o.M[midx(b, c)];
  }
}

// ---------------------------------------------------------------- cached element matrices
// The paper's caching strategy (Sec. 2.3, next to Algorithm 1): the scaled element matrix of
// every cut tet is formed once per microstructure instead of once per iteration.  On side s
// the strain at the parent P1 function N_b is E_b = es + c_b ew + sym(w_b (x) gamma) (see the
// apply kernels), so with the side moments M_bc = int N_b N_c every entry is a sum of
//   beta(x, u; y, v) = sym(e_x (x) u) : C : sym(e_y (x) v)
//                    = lambda u_x v_y + mu (delta_xy u.v + u_y v_x)
// over u, v in {grad N_a, gamma} with the weights (per side)
//   std (a,x)  - std (b,y):  V beta(x, g_a; y, g_b),  V = sum_bc M_bc
//   std (a,x)  - enr (b,y):  d_by [P beta(x, g_a; y, g_b) + m_b beta(x, g_a; y, gamma)]
//   enr (a,x)  - enr (b,y):  d_ax d_by [Q beta(x, g_a; y, g_b) + R_b beta(x, g_a; y, gamma)
//                                        + R_a beta(x, gamma; y, g_b) + M_ab beta(x, gamma; y, gamma)]
// with m_b = sum_c M_bc, R_a = sum_c M_ac c_c, P = sum_b m_b c_b, Q = sum_bc c_b M_bc c_c and
// d = D0^-1/2 of the enriched DOF.  Computed in FP64, stored as FP32: the upper triangle of the
// 24 x 24 matrix (local DOFs std 3a + x, then enr 12 + 3a + x) row by row, kCutPacked values
// per cut tet, structure of arrays kc[k * ncut + e].
XFFT_HD inline double beta_iso(int x, const double* u, int y, const double* v, double lam,
                                           double mu) {
  const double uv = x == y ? u[0] * v[0] + u[1] * v[1] + u[2] * v[2] : 0.0;
  return lam * u[x] * v[y] + mu * (uv + u[y] * v[x]);
}

struct SideW {
  double lam, mu, V, P, Q, m[4], R[4], M[4][4], gam[3];
};

// Per-side weights of a cut tet: the side's Lame constants, gamma = sum_b c_b grad N_b with
// c_b = |L_b| - s L_b, the moments M_bc (packed as cut_f_M) and their sums V, m_b, R_b, P, Q.
XFFT_HD inline void side_weights(const double L[4], double sgn, const double gr[4][3], const double Mp[10],
                                 double lam, double mu, SideW& W) {
  W.lam = lam;
  W.mu = mu;
  double c[4];
  for (int b = 0; b < 4; ++b) c[b] = fabs(L[b]) - sgn * L[b];
  for (int x = 0; x < 3; ++x) W.gam[x] = c[0] * gr[0][x] + c[1] * gr[1][x] + c[2] * gr[2][x] + c[3] * gr[3][x];
  for (int b = 0; b < 4; ++b)
    for (int cc = 0; cc < 4; ++cc) W.M[b][cc] = Mp[midx(b, cc)];
  W.V = W.P = W.Q = 0.0;
  for (int b = 0; b < 4; ++b) {
    W.m[b] = W.M[b][0] + W.M[b][1] + W.M[b][2] + W.M[b][3];
    W.R[b] = W.M[b][0] * c[0] + W.M[b][1] * c[1] + W.M[b][2] * c[2] + W.M[b][3] * c[3];
    W.V += W.m[b];
    W.P += W.m[b] * c[b];
    W.Q += W.R[b] * c[b];
  }
}

// Entry (i, j) of the scaled 24 x 24 element matrix (local DOFs std 3a + x, enr 12 + 3a + x),
// summed over the two sides; dsc = D0^-1/2 of the tet's enriched DOFs.
XFFT_HD inline double cut_element_entry(int i, int j, const SideW w[2], const double gr[4][3],
                                        const double dsc[4][3]) {
  if (j < i) {
    const int tmp = i;
    i = j;
    j = tmp;
  }
  const bool ie = i >= 12, je = j >= 12;
  const int a = (ie ? i - 12 : i) / 3, x = (ie ? i - 12 : i) % 3;
  const int b = (je ? j - 12 : j) / 3, y = (je ? j - 12 : j) % 3;
  double v = 0.0;
  for (int si = 0; si < 2; ++si) {
    const SideW& W = w[si];
    const double bgg = beta_iso(x, gr[a], y, gr[b], W.lam, W.mu);
    if (!je) {
      v += W.V * bgg;
    } else if (!ie) {
      v += dsc[b][y] * (W.P * bgg + W.m[b] * beta_iso(x, gr[a], y, W.gam, W.lam, W.mu));
    } else {
      v += dsc[a][x] * dsc[b][y] *
           (W.Q * bgg + W.R[b] * beta_iso(x, gr[a], y, W.gam, W.lam, W.mu) +
            W.R[a] * beta_iso(x, W.gam, y, gr[b], W.lam, W.mu) + W.M[a][b] * beta_iso(x, W.gam, y, W.gam, W.lam, W.mu));
    }
  }
  return v;
}

// Contributions of one cut tet to the enriched scaling (eq. XFFT_diagonal, per DOF) and, if
// want_off, to the off-diagonal entries of the per-node 3 x 3 Gram blocks.  On side s,
// grad N_X^a = sum_b N_b V_ab with V_ab = c_b g_a + delta_ab gamma, so
//   D_{a,k} = 1/2 sum_bc M_bc (V_ab . V_ac + V_ab[k] V_ac[k])
// and the (k, l) block entry is 1/2 sum_bc M_bc V_ab[k] V_ac[l] for k != l.  Mp[0] / Mp[1]: the
// packed moments of the plus / minus side; off[a] = entries (0,1), (0,2), (1,2).
XFFT_HD inline void cut_scaling_terms(const double L[4], const double gr[4][3], const double Mp[2][10],
                                      double acc[4][3], double off[4][3], bool want_off) {
  for (int a = 0; a < 4; ++a)
    for (int x = 0; x < 3; ++x) acc[a][x] = off[a][x] = 0.0;
  for (int si = 0; si < 2; ++si) {
    const double s = si == 0 ? 1.0 : -1.0;
    double c[4], gam[3] = {0.0, 0.0, 0.0};
    for (int b = 0; b < 4; ++b) {
      c[b] = fabs(L[b]) - s * L[b];
      for (int x = 0; x < 3; ++x) gam[x] += c[b] * gr[b][x];
    }
    // sum_bc M_bc V_ab[x] V_ac[y] = Q g_x g_y + R_a (g_x gamma_y + gamma_x g_y) + M_aa gamma_x gamma_y with
    // R_a = sum_c M_ac c_c and Q = sum_b c_b R_b: a tenth of the operations of the double sum
    const double* M = Mp[si];
    double R[4], Q = 0.0;
    for (int a = 0; a < 4; ++a) {
      R[a] = M[midx(a, 0)] * c[0] + M[midx(a, 1)] * c[1] + M[midx(a, 2)] * c[2] + M[midx(a, 3)] * c[3];
      Q += c[a] * R[a];
    }
    for (int a = 0; a < 4; ++a) {
      double h[3], k[3];  // Q g + R_a gamma and R_a g + M_aa gamma
      for (int x = 0; x < 3; ++x) {
        h[x] = Q * gr[a][x] + R[a] * gam[x];
        k[x] = R[a] * gr[a][x] + M[midx(a, a)] * gam[x];
      }
      double T[3];
      for (int x = 0; x < 3; ++x) T[x] = gr[a][x] * h[x] + gam[x] * k[x];
      const double tr = T[0] + T[1] + T[2];
      for (int x = 0; x < 3; ++x) acc[a][x] += 0.5 * (tr + T[x]);
      if (want_off) {
        off[a][0] += 0.5 * (gr[a][0] * h[1] + gam[0] * k[1]);
        off[a][1] += 0.5 * (gr[a][0] * h[2] + gam[0] * k[2]);
        off[a][2] += 0.5 * (gr[a][1] * h[2] + gam[1] * k[2]);
      }
    }
  }
}

// Inverse of the symmetric positive definite 3 x 3 matrix (a00, a11, a22; a10, a20, a21) by its
// Cholesky factor: v = (inv00, inv11, inv22, inv10, inv20, inv21); false (and v = identity) on a
// non-positive pivot.
XFFT_HD inline bool block_inverse3(double a00, double a11, double a22, double a10, double a20, double a21,
                                   double v[6]) {
  v[0] = v[1] = v[2] = 1.0;
  v[3] = v[4] = v[5] = 0.0;
  if (!(a00 > 0.0)) return false;
  const double l00 = sqrt(a00);
  const double l10 = a10 / l00, l20 = a20 / l00;
  const double p11 = a11 - l10 * l10;
  if (!(p11 > 0.0)) return false;
  const double l11 = sqrt(p11);
  const double l21 = (a21 - l20 * l10) / l11;
  const double p22 = a22 - l20 * l20 - l21 * l21;
  if (!(p22 > 0.0)) return false;
  const double l22 = sqrt(p22);
  const double m00 = 1.0 / l00, m11 = 1.0 / l11, m22 = 1.0 / l22;
  const double m10 = -l10 * m00 * m11;
  const double m21 = -l21 * m11 * m22;
  const double m20 = -(l20 * m00 + l21 * m10) * m22;
  v[0] = m00 * m00 + m10 * m10 + m20 * m20;
  v[1] = m11 * m11 + m21 * m21;
  v[2] = m22 * m22;
  v[3] = m10 * m11 + m20 * m21;
  v[4] = m20 * m22;
  v[5] = m21 * m22;
  return true;
}

}  // namespace xfft
