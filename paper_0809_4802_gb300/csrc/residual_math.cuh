// FP64 element residual of the two-level VMS weak form (Section 4.1: Eqs. SC_Coarse_Resid_Vec,
// SC_Coarse_Resid_Vec_2, SC_Fine_Resid_Vec and the backward-Euler Remark).
//
// Trilinear fields are evaluated in the monomial basis {1, xi, eta, zeta, xi eta, xi zeta,
// eta zeta, xi eta zeta}: nodal values map to coefficients by a butterfly (modal8), after which a
// value costs 7 FMA and a reference gradient 9 FMA. Test functions are accumulated in the same
// basis and mapped back to nodes once per element (nodal8).
//
// With omega = w_q det J, cof = det(J) J^-T, G[i][al] = dv_i/dxi_al and H = G cof^T (H[i][j] =
// det J dv_i/dx_j, the physical velocity gradient L times det J):
//   omega conv_i = w_q (H v)_i
//   P[i][al] = omega sum_j sigma_ij (J^-1)[al][j],  sigma = nut L - p I
//            = w_q sum_j ( (nut/det) H[i][j] - p delta_ij ) cof[j][al]
//   Tp = -omega tr L = -w_q tr H
// so R_c[a][i] = sum_q N_a src_i + dN_a/dxi_al P[i][al], R_p[a] = sum_q N_a Tp,
// R_f[i] = sum_q b src_i + db/dxi_al P[i][al], src_i = omega (conv_i - f_i + tau dvbar_i).
// One reciprocal (1/det J) per quadrature point.
#pragma once

#include "element_math.cuh"

namespace vms {

// Store slots: x-gradient coefficients (3 x 7), v (3 x 8), p (8), vbar - vbar_n (3 x 8), then the
// monomial sums of the momentum (3 x 8) and continuity (8) test functions.
constexpr int RC_X = 0, RC_V = 21, RC_P = 45, RC_DV = 53, RC_RM = 77, RC_RP = 101, RC_N = 109;

template <class Store>
VMS_HD void residual_load(const Store& C, const double X[8][3], const double U[8][4],
                          const double Uprev[8][3], bool transient) {
  double f[8], c[8];
  VMS_UNROLL
  for (int i = 0; i < 3; ++i) {
    VMS_UNROLL
    for (int a = 0; a < 8; ++a) f[a] = X[a][i];
    modal8(f, c);
    VMS_UNROLL
    for (int m = 1; m < 8; ++m) C.set(RC_X + 7 * i + m - 1, 0.125 * c[m]);
  }
  VMS_UNROLL
  for (int i = 0; i < 3; ++i) {
    VMS_UNROLL
    for (int a = 0; a < 8; ++a) f[a] = U[a][i];
    modal8(f, c);
    VMS_UNROLL
    for (int m = 0; m < 8; ++m) C.set(RC_V + 8 * i + m, 0.125 * c[m]);
  }
  VMS_UNROLL
  for (int a = 0; a < 8; ++a) f[a] = U[a][3];
  modal8(f, c);
  VMS_UNROLL
  for (int m = 0; m < 8; ++m) C.set(RC_P + m, 0.125 * c[m]);
  if (transient) {
    VMS_UNROLL
    for (int i = 0; i < 3; ++i) {
      VMS_UNROLL
      for (int a = 0; a < 8; ++a) f[a] = U[a][i] - Uprev[a][i];
      modal8(f, c);
      VMS_UNROLL
      for (int m = 0; m < 8; ++m) C.set(RC_DV + 8 * i + m, 0.125 * c[m]);
    }
  }
}

// The fields along one line of the Gauss rule (eta and zeta fixed): every one is an intercept plus xi
// times a slope. J[.][1] = j1a + xi j1b, J[.][2] = j2a + xi j2b and J[.][0] = J0; the reference velocity
// gradient's columns vb, g1a + xi g1b, g2a + xi g2b; v = va + xi vb; p = pa + xi pb; vbar - vbar_n = dva + xi dvb.
struct ResLine {
  double J0[3], j1a[3], j1b[3], j2a[3], j2b[3], g1a[3], g1b[3], g2a[3], g2b[3], va[3], vb[3], dva[3], dvb[3], pa, pb;
};
// Its sums: src, xi src, P0, P1, xi P1, P2, xi P2 (per component), Tp, xi Tp.
struct ResSums {
  double s0[3], s1[3], b0[3], c0[3], c1[3], d0[3], d1[3], t0, t1;
};

// The sums of the line whose first point is q0 (and R_f, added to); false if det J <= 0 at a point.
template <bool TRANSIENT, bool FORCE, int N1, class Table>
VMS_HD bool residual_line(const Table& tab, int q0, const ResLine& ln, const double bet[3], double nut, double tau,
                          const double f[3], ResSums& o_, double Rf[3]) {
  constexpr int n1 = N1;
  bool ok = true;
  // One point of the line from its fields: y_i = src_i / w_q, the fluxes P_al,i paired with the
  // reference-gradient components of the test functions, and tr H = -Tp / w_q.
  struct Pt {
    double y[3], P0[3], P1[3], P2[3], tr;
  };
  auto point = [&](const double J[3][3], const double v[3], const double G[3][3], double p, const double dv[3],
                   double wnut, double wq, Pt& o) {
    double cof[3][3];
    double det = cofactor3(J, cof);
    if (!det_ok(det)) { ok = false; det = 1.0; }

    // H = G cof^T: det J times the physical velocity gradient (H[i][j] = det dv_i/dx_j)
    double H[3][3];
    VMS_UNROLL
    for (int i = 0; i < 3; ++i)
      VMS_UNROLL
      for (int j = 0; j < 3; ++j)
        H[i][j] = G[i][0] * cof[j][0] + G[i][1] * cof[j][1] + G[i][2] * cof[j][2];
    // y_i = (H v - det f + tau det (vbar - vbar_n))_i
    VMS_UNROLL
    for (int i = 0; i < 3; ++i) o.y[i] = H[i][0] * v[0] + H[i][1] * v[1] + H[i][2] * v[2];
    if (FORCE) {
      VMS_UNROLL
      for (int i = 0; i < 3; ++i) o.y[i] -= det * f[i];
    }
    if (TRANSIENT) {
      const double td = tau * det;
      VMS_UNROLL
      for (int i = 0; i < 3; ++i) o.y[i] += td * dv[i];
    }
    o.tr = H[0][0] + H[1][1] + H[2][2];
    // P = (s H - w_q p I) cof with s = w_q nut / det: w_q (nut L - p I) times det J^-T
    const double s = wnut * recip_normal(det);
    const double nwp = -wq * p;
    VMS_UNROLL
    for (int i = 0; i < 3; ++i)
      VMS_UNROLL
      for (int j = 0; j < 3; ++j) H[i][j] = i == j ? s * H[i][j] + nwp : s * H[i][j];
    VMS_UNROLL
    for (int i = 0; i < 3; ++i) {
      o.P0[i] = H[i][0] * cof[0][0] + H[i][1] * cof[1][0] + H[i][2] * cof[2][0];
      o.P1[i] = H[i][0] * cof[0][1] + H[i][1] * cof[1][1] + H[i][2] * cof[2][1];
      o.P2[i] = H[i][0] * cof[0][2] + H[i][1] * cof[1][2] + H[i][2] * cof[2][2];
    }
  };
  // The points are taken in symmetric pairs (-x, x): the Gauss points are symmetric about 0 (the middle
  // one of an odd rule is 0), w, b, db1, db2 are even in xi and db0 is odd. The bubble's parts of v and of
  // G's last two columns are therefore formed once for both, and with
  // u = y(x) + y(-x) and d = y(x) - y(-x) a pair adds u to a sum, x d to a xi-moment, and
  // b(x) u_src + db0(x) d_P0 + db1(x) u_P1 + db2(x) u_P2 to R_f; src and Tp are weighted after the sums.
  // The middle point's fields are the intercepts. Every FP64 instruction counts (19 cycles of the SM):
  // these three savings take 5 % of a line's.
  VMS_UNROLL
  for (int pp = 0; pp < n1 / 2; ++pp) {
    const int qh = q0 + n1 - 1 - pp;
    const double x = tab.xi(qh), bh = tab.b(qh), wq = tab.w(qh), wnut = wq * nut;
    const double e0 = tab.db(qh, 0), e1 = tab.db(qh, 1), e2 = tab.db(qh, 2);
    double vt[3], g1t[3], g2t[3];
    VMS_UNROLL
    for (int i = 0; i < 3; ++i) {
      vt[i] = ln.va[i] + bh * bet[i];
      g1t[i] = ln.g1a[i] + e1 * bet[i];
      g2t[i] = ln.g2a[i] + e2 * bet[i];
    }
    Pt lo, hi;
    VMS_UNROLL
    for (int side = 0; side < 2; ++side) {
      const double xi = side ? x : -x, db0 = side ? e0 : -e0;
      double J[3][3], G[3][3], v[3], dv[3];
      VMS_UNROLL
      for (int i = 0; i < 3; ++i) {
        J[i][0] = ln.J0[i];
        J[i][1] = ln.j1a[i] + xi * ln.j1b[i];
        J[i][2] = ln.j2a[i] + xi * ln.j2b[i];
        v[i] = vt[i] + xi * ln.vb[i];
        G[i][0] = ln.vb[i] + db0 * bet[i];
        G[i][1] = g1t[i] + xi * ln.g1b[i];
        G[i][2] = g2t[i] + xi * ln.g2b[i];
        dv[i] = TRANSIENT ? ln.dva[i] + xi * ln.dvb[i] : 0.0;
      }
      point(J, v, G, ln.pa + xi * ln.pb, dv, wnut, wq, side ? hi : lo);
    }
    const double xw = x * wq;
    VMS_UNROLL
    for (int i = 0; i < 3; ++i) {
      const double us = wq * (hi.y[i] + lo.y[i]), ws = hi.y[i] - lo.y[i];
      const double u0 = hi.P0[i] + lo.P0[i], w0 = hi.P0[i] - lo.P0[i];
      const double u1 = hi.P1[i] + lo.P1[i], w1 = hi.P1[i] - lo.P1[i];
      const double u2 = hi.P2[i] + lo.P2[i], w2 = hi.P2[i] - lo.P2[i];
      Rf[i] = Rf[i] + bh * us + e0 * w0 + e1 * u1 + e2 * u2;
      if (pp == 0) {
        o_.s0[i] = us; o_.s1[i] = xw * ws; o_.b0[i] = u0; o_.c0[i] = u1; o_.c1[i] = x * w1; o_.d0[i] = u2;
        o_.d1[i] = x * w2;
      } else {
        o_.s0[i] += us; o_.s1[i] += xw * ws; o_.b0[i] += u0; o_.c0[i] += u1; o_.c1[i] += x * w1; o_.d0[i] += u2;
        o_.d1[i] += x * w2;
      }
    }
    const double ut = hi.tr + lo.tr, wt = hi.tr - lo.tr;
    if (pp == 0) { o_.t0 = -wq * ut; o_.t1 = -xw * wt; }
    else { o_.t0 -= wq * ut; o_.t1 -= xw * wt; }
  }
  if (n1 & 1) {
    // the middle point, xi = 0: no xi-moment, db0 = 0
    const int qm = q0 + n1 / 2;
    const double bm = tab.b(qm), e1 = tab.db(qm, 1), e2 = tab.db(qm, 2), wq = tab.w(qm);
    double J[3][3], G[3][3], v[3];
    VMS_UNROLL
    for (int i = 0; i < 3; ++i) {
      J[i][0] = ln.J0[i]; J[i][1] = ln.j1a[i]; J[i][2] = ln.j2a[i];
      v[i] = ln.va[i] + bm * bet[i];
      G[i][0] = ln.vb[i]; G[i][1] = ln.g1a[i] + e1 * bet[i]; G[i][2] = ln.g2a[i] + e2 * bet[i];
    }
    Pt m;
    point(J, v, G, ln.pa, ln.dva, wq * nut, wq, m);
    VMS_UNROLL
    for (int i = 0; i < 3; ++i) {
      const double ms = wq * m.y[i];
      Rf[i] = Rf[i] + bm * ms + e1 * m.P1[i] + e2 * m.P2[i];
      o_.s0[i] += ms; o_.b0[i] += m.P0[i]; o_.c0[i] += m.P1[i]; o_.d0[i] += m.P2[i];
    }
    o_.t0 -= wq * m.tr;
  }
  return ok;
}

// Quadrature loop. Rcp[32] (node-major 4a+c) and Rf[3] receive the element residual; returns
// false if det J <= 0 at some point (the offending point then uses det J = 1).
//
// The tensor Gauss rule is walked line by line (xi fastest; the table's point order). Along a
// line eta and zeta are fixed, so every trilinear field is a + xi b with a, b formed once per line:
// the three columns of J (J[.][0] constant along the line), the polynomial part of G (its first
// column is also the xi-slope b of v), v's a, p's a and b, and (transient) those of vbar - vbar_n. The test-function sums are factored the same way: a
// monomial xi^a eta^b zeta^c (or its derivative) is xi^a times a line constant, so each line keeps
// seven sums per component (src, xi src, P0, P1, xi P1, P2, xi P2) and two for the continuity term,
// and adds them into the eight monomial sums, which live in the store, once per line.
template <bool TRANSIENT, bool FORCE, int N1, class Store, class Table>
VMS_HD bool residual_qp_loop_n(const Store& C, const Table& tab, const double bet[3], double nut,
                               double tau, const double f[3], double Rcp[32], double Rf[3]) {
  constexpr int n1 = N1;
  VMS_UNROLL
  for (int m = 0; m < 32; ++m) C.set(RC_RM + m, 0.0);
  Rf[0] = Rf[1] = Rf[2] = 0.0;
  bool ok = true;
  for (int k = 0; k < n1; ++k) {
    // plane constants (zeta fixed): the parts of the line constants that do not depend on eta
    const double zeta = tab.zeta(k * n1 * n1);
    double aj0[3], j1a[3], j1b[3], g1a[3], g1b[3], ava[3], avb[3], ada[3], bda[3], adb[3], bdb[3];
    VMS_UNROLL
    for (int i = 0; i < 3; ++i) {
      aj0[i] = C.get(RC_X + 7 * i + 0) + C.get(RC_X + 7 * i + 4) * zeta;
      j1a[i] = C.get(RC_X + 7 * i + 1) + C.get(RC_X + 7 * i + 5) * zeta;
      j1b[i] = C.get(RC_X + 7 * i + 3) + C.get(RC_X + 7 * i + 6) * zeta;
      g1a[i] = C.get(RC_V + 8 * i + 2) + C.get(RC_V + 8 * i + 6) * zeta;
      g1b[i] = C.get(RC_V + 8 * i + 4) + C.get(RC_V + 8 * i + 7) * zeta;
      ava[i] = C.get(RC_V + 8 * i + 0) + C.get(RC_V + 8 * i + 3) * zeta;
      avb[i] = C.get(RC_V + 8 * i + 1) + C.get(RC_V + 8 * i + 5) * zeta;
      if (TRANSIENT) {
        ada[i] = C.get(RC_DV + 8 * i + 0) + C.get(RC_DV + 8 * i + 3) * zeta;
        bda[i] = C.get(RC_DV + 8 * i + 2) + C.get(RC_DV + 8 * i + 6) * zeta;
        adb[i] = C.get(RC_DV + 8 * i + 1) + C.get(RC_DV + 8 * i + 5) * zeta;
        bdb[i] = C.get(RC_DV + 8 * i + 4) + C.get(RC_DV + 8 * i + 7) * zeta;
      }
    }
    const double apa = C.get(RC_P + 0) + C.get(RC_P + 3) * zeta, bpa = C.get(RC_P + 2) + C.get(RC_P + 6) * zeta;
    const double apb = C.get(RC_P + 1) + C.get(RC_P + 5) * zeta, bpb = C.get(RC_P + 4) + C.get(RC_P + 7) * zeta;
    for (int j = 0; j < n1; ++j) {
      const int q0 = (k * n1 + j) * n1;
      const double eta = tab.eta(q0), ez = tab.ez(q0);
      // line constants: along the line J[i][1] = j1a + xi j1b, J[i][2] = j2a + xi j2b, and the
      // same for the reference velocity gradient (g1a, g1b, g2a, g2b); every trilinear field is
      // its plane part plus eta times its eta-slope
      double J0[3], vb[3], va[3], dva[3], dvb[3], j2a[3], j2b[3], g2a[3], g2b[3];
      VMS_UNROLL
      for (int i = 0; i < 3; ++i) {
        J0[i] = aj0[i] + j1b[i] * eta;
        j2a[i] = C.get(RC_X + 7 * i + 2) + C.get(RC_X + 7 * i + 5) * eta;
        j2b[i] = C.get(RC_X + 7 * i + 4) + C.get(RC_X + 7 * i + 6) * eta;
        g2a[i] = C.get(RC_V + 8 * i + 3) + C.get(RC_V + 8 * i + 6) * eta;
        g2b[i] = C.get(RC_V + 8 * i + 5) + C.get(RC_V + 8 * i + 7) * eta;
        vb[i] = avb[i] + g1b[i] * eta;
        va[i] = ava[i] + g1a[i] * eta;
        if (TRANSIENT) {
          dva[i] = ada[i] + bda[i] * eta;
          dvb[i] = adb[i] + bdb[i] * eta;
        }
      }
      const double pa = apa + bpa * eta, pb = apb + bpb * eta;
      ResLine ln;
      VMS_UNROLL
      for (int i = 0; i < 3; ++i) {
        ln.J0[i] = J0[i]; ln.j1a[i] = j1a[i]; ln.j1b[i] = j1b[i]; ln.j2a[i] = j2a[i]; ln.j2b[i] = j2b[i];
        ln.g1a[i] = g1a[i]; ln.g1b[i] = g1b[i]; ln.g2a[i] = g2a[i]; ln.g2b[i] = g2b[i];
        ln.va[i] = va[i]; ln.vb[i] = vb[i];
        if (TRANSIENT) { ln.dva[i] = dva[i]; ln.dvb[i] = dvb[i]; }
      }
      ln.pa = pa; ln.pb = pb;
      ResSums sm;
      if (!residual_line<TRANSIENT, FORCE, N1>(tab, q0, ln, bet, nut, tau, f, sm, Rf)) ok = false;
      const double *s0 = sm.s0, *s1 = sm.s1, *b0 = sm.b0, *c0 = sm.c0, *c1 = sm.c1, *d0 = sm.d0, *d1 = sm.d1;
      const double t0 = sm.t0, t1 = sm.t1;
      // the line's contributions to the monomial sums: xi^a eta^b zeta^c src_i and the
      // derivatives d/dxi (P0), d/deta (P1), d/dzeta (P2) of the same monomials
      VMS_UNROLL
      for (int i = 0; i < 3; ++i) {
        const double sb = s1[i] + b0[i];
        const int r = RC_RM + 8 * i;
        C.set(r + 0, C.get(r + 0) + s0[i]);
        C.set(r + 1, C.get(r + 1) + sb);
        C.set(r + 2, C.get(r + 2) + (eta * s0[i] + c0[i]));
        C.set(r + 3, C.get(r + 3) + (zeta * s0[i] + d0[i]));
        C.set(r + 4, C.get(r + 4) + (eta * sb + c1[i]));
        C.set(r + 5, C.get(r + 5) + (zeta * sb + d1[i]));
        C.set(r + 6, C.get(r + 6) + ez * s0[i] + zeta * c0[i] + eta * d0[i]);
        C.set(r + 7, C.get(r + 7) + ez * sb + zeta * c1[i] + eta * d1[i]);
      }
      C.set(RC_RP + 0, C.get(RC_RP + 0) + t0);
      C.set(RC_RP + 1, C.get(RC_RP + 1) + t1);
      C.set(RC_RP + 2, C.get(RC_RP + 2) + eta * t0);
      C.set(RC_RP + 3, C.get(RC_RP + 3) + zeta * t0);
      C.set(RC_RP + 4, C.get(RC_RP + 4) + eta * t1);
      C.set(RC_RP + 5, C.get(RC_RP + 5) + zeta * t1);
      C.set(RC_RP + 6, C.get(RC_RP + 6) + ez * t0);
      C.set(RC_RP + 7, C.get(RC_RP + 7) + ez * t1);
    }
  }
  double r[8], mm[8];
  VMS_UNROLL
  for (int i = 0; i < 3; ++i) {
    VMS_UNROLL
    for (int m = 0; m < 8; ++m) mm[m] = C.get(RC_RM + 8 * i + m);
    nodal8(mm, r);
    VMS_UNROLL
    for (int a = 0; a < 8; ++a) Rcp[4 * a + i] = 0.125 * r[a];
  }
  VMS_UNROLL
  for (int m = 0; m < 8; ++m) mm[m] = C.get(RC_RP + m);
  nodal8(mm, r);
  VMS_UNROLL
  for (int a = 0; a < 8; ++a) Rcp[4 * a + 3] = 0.125 * r[a];
  return ok;
}

// The quadrature loop for the Gauss rule of nq = 8, 27 or 64 points (the line loop unrolled).
template <bool TRANSIENT, bool FORCE, class Store, class Table>
VMS_HD bool residual_qp_loop(const Store& C, const Table& tab, int nq, const double bet[3],
                             double nut, double tau, const double f[3], double Rcp[32],
                             double Rf[3]) {
  if (nq == 27) return residual_qp_loop_n<TRANSIENT, FORCE, 3>(C, tab, bet, nut, tau, f, Rcp, Rf);
  if (nq == 8) return residual_qp_loop_n<TRANSIENT, FORCE, 2>(C, tab, bet, nut, tau, f, Rcp, Rf);
  return residual_qp_loop_n<TRANSIENT, FORCE, 4>(C, tab, bet, nut, tau, f, Rcp, Rf);
}

#if defined(__CUDACC__)
// One element's residual on one thread: gather the 8 nodes (and the previous step's velocities),
// map them to monomial coefficients in `C`, run the quadrature loop. Returns the element's error
// bits: 1 if det J <= 0 at some point, 4 if a residual entry is not finite (the values of
// FLAG_NEG_JACOBIAN and FLAG_NAN). P provides nut, visc_factor, nu_e, nq, tau and f.
template <bool TRANSIENT, bool FORCE, class Store, class Table, class P>
__device__ __forceinline__ unsigned residual_element(
    int64_t e, const Store& C, const Table& tab, const P& kp,
    const double4_32a* __restrict__ xyz, const double4_32a* __restrict__ u,
    const double4_32a* __restrict__ uprev, const int32_t* __restrict__ conn,
    const double* __restrict__ beta, int nd[8], double Rcp[32], double Rf[3]) {
  {
    const int4* cp = reinterpret_cast<const int4*>(conn + 8 * e);
    const int4 c0 = cp[0], c1 = cp[1];
    nd[0] = c0.x; nd[1] = c0.y; nd[2] = c0.z; nd[3] = c0.w;
    nd[4] = c1.x; nd[5] = c1.y; nd[6] = c1.z; nd[7] = c1.w;
  }
  {
    // one record type at a time, each mapped to its monomial coefficients before the next is
    // loaded (fewer values live at once than gathering all node data first)
    double f[8], c[8], U[8][3];
    {
      double X[8][3];
      VMS_UNROLL
      for (int a = 0; a < 8; ++a) {
        const double4_32a x = xyz[nd[a]];
        X[a][0] = x.x; X[a][1] = x.y; X[a][2] = x.z;
      }
      VMS_UNROLL
      for (int i = 0; i < 3; ++i) {
        VMS_UNROLL
        for (int a = 0; a < 8; ++a) f[a] = X[a][i];
        modal8(f, c);
        VMS_UNROLL
        for (int m = 1; m < 8; ++m) C.set(RC_X + 7 * i + m - 1, 0.125 * c[m]);
      }
    }
    {
      double pn[8];
      VMS_UNROLL
      for (int a = 0; a < 8; ++a) {
        const double4_32a w = u[nd[a]];
        U[a][0] = w.x; U[a][1] = w.y; U[a][2] = w.z; pn[a] = w.w;
      }
      modal8(pn, c);
      VMS_UNROLL
      for (int m = 0; m < 8; ++m) C.set(RC_P + m, 0.125 * c[m]);
    }
    VMS_UNROLL
    for (int i = 0; i < 3; ++i) {
      VMS_UNROLL
      for (int a = 0; a < 8; ++a) f[a] = U[a][i];
      modal8(f, c);
      VMS_UNROLL
      for (int m = 0; m < 8; ++m) C.set(RC_V + 8 * i + m, 0.125 * c[m]);
    }
    if (TRANSIENT) {
      VMS_UNROLL
      for (int a = 0; a < 8; ++a) {
        const double4_32a o = uprev[nd[a]];
        U[a][0] -= o.x; U[a][1] -= o.y; U[a][2] -= o.z;
      }
      VMS_UNROLL
      for (int i = 0; i < 3; ++i) {
        VMS_UNROLL
        for (int a = 0; a < 8; ++a) f[a] = U[a][i];
        modal8(f, c);
        VMS_UNROLL
        for (int m = 0; m < 8; ++m) C.set(RC_DV + 8 * i + m, 0.125 * c[m]);
      }
    }
  }
  const double bet[3] = {beta[3 * e + 0], beta[3 * e + 1], beta[3 * e + 2]};
  const double nut = kp.nu_e ? kp.visc_factor * __ldg(kp.nu_e + e) : kp.nut;
  const bool ok = residual_qp_loop<TRANSIENT, FORCE>(C, tab, kp.nq, bet, nut, kp.tau, kp.f, Rcp, Rf);
  bool finite = isfinite(Rf[0]) && isfinite(Rf[1]) && isfinite(Rf[2]);
  VMS_UNROLL
  for (int k = 0; k < 32; ++k) finite = finite && isfinite(Rcp[k]);
  return (ok ? 0u : 1u) | (finite ? 0u : 4u);
}

// The same residual with the N1^2 lines of the Gauss rule on as many lanes, 32 / N1^2 elements per
// warp (an FP64 instruction takes 64 cycles of a warp, however many lanes are active, so a thread
// per element takes about 170 us alone; a line takes a ninth of the points). The element's fields are
// mapped to their monomial coefficients one per lane; every lane walks its line and forms its shares
// of the 32 monomial sums and of R_f; the lanes then sum one output each and map a component each
// back to the nodes. `sm`: the element's RL_DOUBLES in shared memory; `ln`: the lane's line; lanes
// without an element (`valid` false) only take part in the warp's barriers. `put(a, c, value)`
// receives R_cp, putf(i, value) R_f. Returns error bits as residual_element.
template <int N1> constexpr int rl_doubles() { return RC_RM + 35 * N1 * N1 + 35; }
template <bool TRANSIENT, bool FORCE, int N1, class Table, class P, class Put, class PutF>
__device__ __forceinline__ unsigned residual_lines(
    bool valid, int64_t e, int ln, double* sm, const Table& tab, const P& kp,
    const double4_32a* __restrict__ xyz, const double4_32a* __restrict__ u,
    const double4_32a* __restrict__ uprev, const int32_t* __restrict__ conn,
    const double* __restrict__ beta, const Put& put, const PutF& putf) {
  constexpr int S = N1 * N1;
  double* share = sm + RC_RM;          // [35][S]
  double* total = sm + RC_RM + 35 * S;  // [35]
  unsigned bad = 0;
  if (valid)
    for (int fi = ln; fi < (TRANSIENT ? 10 : 7); fi += S) {  // x (3), v and p (4), v - v_prev (3)
      const int comp = fi < 3 ? fi : (fi < 7 ? fi - 3 : fi - 7);
      const double4_32a* rec = fi < 3 ? xyz : u;
      double fv[8], c[8];
      VMS_UNROLL
      for (int a = 0; a < 8; ++a) {
        const int64_t nd = conn[8 * e + a];
        fv[a] = reinterpret_cast<const double*>(rec + nd)[comp];
        if (TRANSIENT && fi >= 7) fv[a] -= reinterpret_cast<const double*>(uprev + nd)[comp];
      }
      modal8(fv, c);
      double* dst = sm + (fi < 3 ? RC_X + 7 * fi - 1 : (fi < 7 ? RC_V + 8 * comp : RC_DV + 8 * comp));
      if (fi >= 3) dst[0] = 0.125 * c[0];
      VMS_UNROLL
      for (int m = 1; m < 8; ++m) dst[m] = 0.125 * c[m];
    }
  __syncwarp();
  if (valid) {
    const int q0 = ln * N1;
    const double eta = tab.eta(q0), zeta = tab.zeta(q0), ez = tab.ez(q0);
    ResLine L;
    VMS_UNROLL
    for (int i = 0; i < 3; ++i) {
      const double *X = sm + RC_X + 7 * i - 1, *V = sm + RC_V + 8 * i, *D = sm + RC_DV + 8 * i;
      L.j1a[i] = X[2] + X[6] * zeta;
      L.j1b[i] = X[4] + X[7] * zeta;
      L.J0[i] = X[1] + X[5] * zeta + L.j1b[i] * eta;
      L.j2a[i] = X[3] + X[6] * eta;
      L.j2b[i] = X[5] + X[7] * eta;
      L.g1a[i] = V[2] + V[6] * zeta;
      L.g1b[i] = V[4] + V[7] * zeta;
      L.g2a[i] = V[3] + V[6] * eta;
      L.g2b[i] = V[5] + V[7] * eta;
      L.va[i] = V[0] + V[3] * zeta + L.g1a[i] * eta;
      L.vb[i] = V[1] + V[5] * zeta + L.g1b[i] * eta;
      if (TRANSIENT) {
        L.dva[i] = D[0] + D[3] * zeta + (D[2] + D[6] * zeta) * eta;
        L.dvb[i] = D[1] + D[5] * zeta + (D[4] + D[7] * zeta) * eta;
      }
    }
    {
      const double* Pc = sm + RC_P;
      L.pa = Pc[0] + Pc[3] * zeta + (Pc[2] + Pc[6] * zeta) * eta;
      L.pb = Pc[1] + Pc[5] * zeta + (Pc[4] + Pc[7] * zeta) * eta;
    }
    const double bet[3] = {beta[3 * e + 0], beta[3 * e + 1], beta[3 * e + 2]};
    const double nut = kp.nu_e ? kp.visc_factor * __ldg(kp.nu_e + e) : kp.nut;
    double Rf[3] = {0.0, 0.0, 0.0};
    ResSums s;
    if (!residual_line<TRANSIENT, FORCE, N1>(tab, q0, L, bet, nut, kp.tau, kp.f, s, Rf)) bad = 1u;
    double* o = share + ln;  // output t's share at o[t S]
    VMS_UNROLL
    for (int i = 0; i < 3; ++i) {
      const double sb = s.s1[i] + s.b0[i];
      o[(8 * i + 0) * S] = s.s0[i];
      o[(8 * i + 1) * S] = sb;
      o[(8 * i + 2) * S] = eta * s.s0[i] + s.c0[i];
      o[(8 * i + 3) * S] = zeta * s.s0[i] + s.d0[i];
      o[(8 * i + 4) * S] = eta * sb + s.c1[i];
      o[(8 * i + 5) * S] = zeta * sb + s.d1[i];
      o[(8 * i + 6) * S] = ez * s.s0[i] + zeta * s.c0[i] + eta * s.d0[i];
      o[(8 * i + 7) * S] = ez * sb + zeta * s.c1[i] + eta * s.d1[i];
      o[(32 + i) * S] = Rf[i];
    }
    o[24 * S] = s.t0;
    o[25 * S] = s.t1;
    o[26 * S] = eta * s.t0;
    o[27 * S] = zeta * s.t0;
    o[28 * S] = eta * s.t1;
    o[29 * S] = zeta * s.t1;
    o[30 * S] = ez * s.t0;
    o[31 * S] = ez * s.t1;
  }
  __syncwarp();
  if (valid)
    for (int t = ln; t < 35; t += S) {
      double v = share[t * S];
      VMS_UNROLL
      for (int l = 1; l < S; ++l) v += share[t * S + l];
      total[t] = v;
    }
  __syncwarp();
  if (valid) {
    if (ln < 4) {  // component ln: velocity 0..2, pressure 3
      double r[8];
      nodal8(total + 8 * ln, r);
      VMS_UNROLL
      for (int a = 0; a < 8; ++a) {
        const double v = 0.125 * r[a];
        if (!isfinite(v)) bad |= 4u;
        put(a, ln, v);
      }
    }
    for (int i = ln - 4 >= 0 ? ln - 4 : (S <= 4 ? ln : 3); i < 3; i += (S <= 4 ? S : 3)) {
      if (!isfinite(total[32 + i])) bad |= 4u;
      putf(i, total[32 + i]);
    }
  }
  __syncwarp();  // the element's shared memory may be reused
  return bad;
}

// Store the element residual in its 36-double record: R_cp (32, node-major), R_f (3), pad.
__device__ __forceinline__ void store_elem_residual(double* __restrict__ rec, const double Rcp[32],
                                                    const double Rf[3]) {
  double2* out = reinterpret_cast<double2*>(rec);
  VMS_UNROLL
  for (int k = 0; k < 16; ++k) out[k] = make_double2(Rcp[2 * k], Rcp[2 * k + 1]);
  out[16] = make_double2(Rf[0], Rf[1]);
  out[17] = make_double2(Rf[2], 0.0);
}
#endif

}  // namespace vms
