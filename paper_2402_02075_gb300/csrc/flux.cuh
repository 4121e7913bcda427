// The time-dependent gas-kinetic flux of a Gauss point (Eq. 2nd-flux of the paper, Sec. 2.3-2.4) in FP64.
//
// The FP64 pipe bounds it, so the form is the one with the fewest FP64 instructions found so far.  It
// evaluates the same integrals as point_flux (fine.cuh), which serves the other scalar types:
//  - gradients are primitive: for every direction k of the global frame (d rho, R_i = rho d u_i, d p).
//    The micro-slope of a Maxwellian is diagonal in them: with the peculiar velocity u - U,
//    h = p/rho and th = d p - h d rho,
//      a = (1/rho) [d rho + R.(u - U)/h + th/h (|u - U|^2 + xi^2 - (K + 3) h)/(2 h)],
//    and the Euler equations give its time slope in a few operations (dt rho = -u.d rho - tr R, ...);
//  - with m_k = <u_n^k> over the half space divided by rho, and beta = +-g(0)/rho, integration by parts
//    in u_n gives the normal moments of a slope (d, R_n, th) without any division or coefficient:
//      D_k = <u_n^k a> = m_k d + X_k R_n + Y_k th,
//      X = (beta, m_0, 2 m_1, 3 m_2, 4 m_3),  Y = (-beta U/(2 h), beta/2, m_0, 3 m_1, 6 m_2);
//    the tangential momentum row is m_k R, the energy row D_{k+2}/2 + (K+2)/2 (h D_k + m_k th), and the
//    moments of c a (c the tangential peculiar velocity) reuse the D_k of the tangential directions;
//  - no face frame: a vector is kept in the global frame, its normal component taken with n where it is
//    needed, so nothing is rotated in or out.  Tangential vectors may carry a normal component that
//    the final projection removes;
//  - both sides' moments are summed in the frame moving with the interface's tangential velocity, where
//    the heat flux of the Prandtl correction needs three of the time-integrated moments only.
// Measured on the 96x64x69 boundary layer (10.67 M points), CUDA events: 25.3 ms with the interface
// state, 23.4 ms the flux alone, against 37.6 and 35.6 ms by point_flux<double>.
#pragma once
#include "fastmath.cuh"
#include "kinetic.cuh"

// one side of the interface: state, half-space seeds
struct GksSide {
  double rho, r, u[3], U, ut[3];  // density, 1/rho, velocity, its normal and tangential parts
  double p, h, l2, sl;            // pressure, p/rho, rho/p, 1/sqrt(2 h)
  double m0, beta;                // half-space mass fraction, s g(0)/rho (s the side: u_n > 0 or < 0)
};

// s = +1 left, -1 right; false where the state is not physical
HD bool gks_side(const double w[5], const double n[3], double s, double gm1, const double* tab, GksSide& g) {
  g.rho = w[0];
  g.r = fast_rcp(w[0]);
#pragma unroll
  for (int d = 0; d < 3; ++d) g.u[d] = w[1 + d] * g.r;
  g.p = gm1 * (w[4] - 0.5 * (w[1] * g.u[0] + w[2] * g.u[1] + w[3] * g.u[2]));
  g.h = g.p * g.r;
  g.U = g.u[0] * n[0] + g.u[1] * n[1] + g.u[2] * n[2];
#pragma unroll
  for (int d = 0; d < 3; ++d) g.ut[d] = g.u[d] - g.U * n[d];
  g.sl = fast_rsqrt(2.0 * g.h);
  g.l2 = 2.0 * g.sl * g.sl;
  double e;
  half_gauss(-s * (g.sl * g.U), tab, g.m0, e);
  g.beta = (s * 0.56418958354775628695) * (e * g.sl);
  return positive(w[0]) && positive(g.p);
}

// time coefficients of Eq. 2nd-flux integrated over [0, dt] that multiply the two sides' moments
struct GksTime {
  double q4, q5, tq4;     // of g, of -(a.u) g and of -A g in the flux
  double edt, etd, etau;  // the same in the interface state at dt
};

// sums over both sides in the frame moving with the interface's tangential velocity: gradients of the
// interface equilibrium (mass, normal momentum, tangential momentum and energy, per direction) and the
// moments of the time-integrated flux (F), of the state at dt (W) and of the time-integrated state (I)
struct GksAcc {
  double rho[3], mn[3], T[3][3], e[3];
  double F0, F1, F4, FT[3], W0, W1, W4, WT[3], I0, I4;
};

// adds one side: G the conservative gradients (15), ut_c the interface's tangential velocity.  STATE: the
// state at dt as well; heat: the time-integrated state's rows that the Prandtl correction uses.  FIRST:
// the sums start with this side
template <bool STATE, bool FIRST>
HD void gks_add_side(const GksSide& g, const double G[15], const double n[3], const double utc[3], double gm1, double gamma,
                     double k2, const GksTime& t, bool heat, GksAcc& a) {
  double del[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) del[d] = g.ut[d] - utc[d];
  const double hd2 = 0.5 * (del[0] * del[0] + del[1] * del[1] + del[2] * del[2]);
  const double hu2 = 0.5 * (g.u[0] * g.u[0] + g.u[1] * g.u[1] + g.u[2] * g.u[2]);
  // primitive gradients
  double R[3][3], gp[3], th[3], Rn[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int i = 0; i < 3; ++i) R[i][k] = G[3 * (1 + i) + k] - g.u[i] * G[k];
    double x = G[12 + k] - hu2 * G[k];
    x -= g.u[0] * R[0][k];
    x -= g.u[1] * R[1][k];
    x -= g.u[2] * R[2][k];
    gp[k] = gm1 * x;
    th[k] = gp[k] - g.h * G[k];
    Rn[k] = n[0] * R[0][k] + n[1] * R[1][k] + n[2] * R[2][k];
  }
  // moments and the coefficients X_k, Y_k
  const double U = g.U, h = g.h, m0 = g.m0, beta = g.beta;
  const double m1 = U * m0 + h * beta;
  const double hm0 = h * m0, m2 = U * m1 + hm0;
  const double hm1 = h * m1, m3 = U * m2 + 2.0 * hm1;
  const double m4 = U * m3 + 3.0 * (h * m2);
  const double X2 = 2.0 * m1, X3 = 3.0 * m2, X4 = 4.0 * m3;
  const double Y0 = -0.5 * U * (beta * g.l2), Y1 = 0.5 * beta, Y3 = 3.0 * m1, Y4 = 2.0 * X3;
  const double kap = k2 * h, k2m0 = k2 * m0, k2m1 = k2 * m1, kd = kap + hd2;
  double dm0[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) dm0[d] = del[d] * m0;
  // gradients of the interface equilibrium; the D_0, D_1 of each direction serve below
  double D0[3], D1[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    D0[k] = m0 * G[k] + beta * Rn[k] + Y0 * th[k];
    D1[k] = m1 * G[k] + m0 * Rn[k] + Y1 * th[k];
    const double D2 = m2 * G[k] + X2 * Rn[k] + m0 * th[k];
    double e = FIRST ? 0.5 * D2 : a.e[k] + 0.5 * D2;
    e += kd * D0[k];
    e += k2m0 * th[k];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      e += dm0[i] * R[i][k];
      double T = FIRST ? m0 * R[i][k] : a.T[i][k] + m0 * R[i][k];
      a.T[i][k] = T + del[i] * D0[k];
    }
    a.e[k] = e;
    a.rho[k] = FIRST ? D0[k] : a.rho[k] + D0[k];
    a.mn[k] = FIRST ? D1[k] : a.mn[k] + D1[k];
  }
  // derivatives along n and along the tangential velocity
  const double rn = n[0] * G[0] + n[1] * G[1] + n[2] * G[2];
  const double pn = n[0] * gp[0] + n[1] * gp[1] + n[2] * gp[2];
  const double rS = g.ut[0] * G[0] + g.ut[1] * G[1] + g.ut[2] * G[2];
  const double pS = g.ut[0] * gp[0] + g.ut[1] * gp[1] + g.ut[2] * gp[2];
  double Rv[3], RS[3], Rt[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Rv[i] = n[0] * R[i][0] + n[1] * R[i][1] + n[2] * R[i][2];
    RS[i] = g.ut[0] * R[i][0] + g.ut[1] * R[i][1] + g.ut[2] * R[i][2];
    Rt[i] = U * Rv[i] + (RS[i] + gp[i]);
  }
  const double Rnn = n[0] * Rv[0] + n[1] * Rv[1] + n[2] * Rv[2];
  const double RnS = n[0] * RS[0] + n[1] * RS[1] + n[2] * RS[2];
  const double Rnt = n[0] * Rt[0] + n[1] * Rt[1] + n[2] * Rt[2];
  const double thn = pn - h * rn, thS = pS - h * rS;
  const double tr = R[0][0] + R[1][1] + R[2][2], Dv = tr - Rnn;
  // minus the time derivatives (Euler)
  const double rt = U * rn + (rS + tr);
  const double tht = U * pn + pS + (gamma * h) * tr - h * rt;
  // rows of <u_n^k (a.u) psi> (al) and of -<u_n^k A psi> (At), k = 0..3 for the powers of u_n and e0, e1
  // for the energy rows of k = 0, 1
  const double rSD = rS + Dv;
  double al0 = m1 * rn + m0 * Rnn + Y1 * thn;
  al0 += m0 * rSD;
  al0 += beta * RnS;
  al0 += Y0 * thS;
  double al1 = m2 * rn + X2 * Rnn + m0 * thn;
  al1 += m1 * rSD;
  al1 += m0 * RnS;
  al1 += Y1 * thS;
  double al2 = m3 * rn + X3 * Rnn + Y3 * thn;
  al2 += m2 * rSD;
  al2 += X2 * RnS;
  al2 += m0 * thS;
  double al3 = m4 * rn + X4 * Rnn + Y4 * thn;
  al3 += m3 * rSD;
  al3 += X3 * RnS;
  al3 += Y3 * thS;
  const double At0 = m0 * rt + beta * Rnt + Y0 * tht;
  const double At1 = m1 * rt + m0 * Rnt + Y1 * tht;
  const double At2 = m2 * rt + X2 * Rnt + m0 * tht;
  const double At3 = m3 * rt + X3 * Rnt + Y3 * tht;
  // tangential rows of a.u, k = 0, 1
  double Ta0[3], Ta1[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double b = RS[i] + th[i];
    Ta0[i] = m1 * Rv[i] + m0 * b + h * D0[i];
    Ta1[i] = m2 * Rv[i] + m1 * b + h * D1[i];
  }
  const double v4 = 0.5 * m2 + kap * m0, f4 = 0.5 * m3 + kap * m1;  // energy rows of psi and u psi
  {
    // flux: q4 <u psi> - q5 <u (a.u) psi> - tau q4 <u A psi>
    const double qr = t.q4 * g.rho, z1 = t.q5 * al1 - t.tq4 * At1, z2 = t.q5 * al2 - t.tq4 * At2,
                 z3 = t.q5 * al3 - t.tq4 * At3;
    const double hn = t.q5 * thn, hb = t.q5 * thS - t.tq4 * tht, dv = t.q5 * Dv;
    const double F0 = qr * m1 - z1, F1 = qr * m2 - z2;
    double F4 = qr * f4 - 0.5 * z3;
    F4 -= kap * z1;
    F4 -= (k2 * m2) * hn;
    F4 -= k2m1 * hb;
    F4 -= hm1 * dv;
    F4 += hd2 * F0;
    const double c = t.tq4 * m1;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double T = t.q5 * Ta1[i] - c * Rt[i];
      F4 -= del[i] * T;
      const double x = del[i] * F0 - T;
      a.FT[i] = FIRST ? x : a.FT[i] + x;
    }
    a.F0 = FIRST ? F0 : a.F0 + F0;
    a.F1 = FIRST ? F1 : a.F1 + F1;
    a.F4 = FIRST ? F4 : a.F4 + F4;
    if (heat) {
      const double z0 = t.q5 * al0 - t.tq4 * At0, I0 = qr * m0 - z0;
      double I4 = qr * v4 - 0.5 * z2;
      I4 -= kap * z0;
      I4 -= k2m1 * hn;
      I4 -= k2m0 * hb;
      I4 -= hm0 * dv;
      I4 += hd2 * I0;
      const double qT = t.q5 * (del[0] * Ta0[0] + del[1] * Ta0[1] + del[2] * Ta0[2]);
      const double qA = (t.tq4 * m0) * (del[0] * Rt[0] + del[1] * Rt[1] + del[2] * Rt[2]);
      I4 -= qT - qA;
      a.I0 = FIRST ? I0 : a.I0 + I0;
      a.I4 = FIRST ? I4 : a.I4 + I4;
    }
  }
  if (STATE) {
    const double qr = t.edt * g.rho, z0 = t.etd * al0 - t.etau * At0, z1 = t.etd * al1 - t.etau * At1,
                 z2 = t.etd * al2 - t.etau * At2;
    const double hn = t.etd * thn, hb = t.etd * thS - t.etau * tht, dv = t.etd * Dv;
    const double W0 = qr * m0 - z0, W1 = qr * m1 - z1;
    double W4 = qr * v4 - 0.5 * z2;
    W4 -= kap * z0;
    W4 -= k2m1 * hn;
    W4 -= k2m0 * hb;
    W4 -= hm0 * dv;
    W4 += hd2 * W0;
    const double c = t.etau * m0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double T = t.etd * Ta0[i] - c * Rt[i];
      W4 -= del[i] * T;
      const double x = del[i] * W0 - T;
      a.WT[i] = FIRST ? x : a.WT[i] + x;
    }
    a.W0 = FIRST ? W0 : a.W0 + W0;
    a.W1 = FIRST ? W1 : a.W1 + W1;
    a.W4 = FIRST ? W4 : a.W4 + W4;
  }
}

// moments (mass F0, normal momentum F1, tangential momentum T, energy F4) of the frame moving with the
// tangential velocity ut -> conservative vector of the global frame, times c
HD void gks_to_global(double F0, double F1, double F4, const double T[3], const double n[3], const double ut[3], double hut2,
                      double c, double out[5]) {
  out[0] = c * F0;
  const double x = F1 - (n[0] * T[0] + n[1] * T[1] + n[2] * T[2]);
  double e = F4 + hut2 * F0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    e += ut[i] * T[i];
    double v = T[i] + ut[i] * F0;
    v += x * n[i];
    out[1 + i] = c * v;
  }
  out[4] = c * e;
}

// mu(T), t = T/T_inf: fine.cuh
template <typename T>
HD T viscosity(const Phys& ph, T t);

// flux of one Gauss point: n the unit normal, weight the length of its area vector; WL, GL, WR, GR the
// states and gradients of both sides (global frame; on a boundary face the ghost's), dt the face's time
// step.  F: flux x weight averaged over dt; Wg (STATE): the interface state at dt; alpha (STATE): the
// compression factor (1 on boundary faces and with the factor off).  Returns 0, or the number of the
// check that failed (4 a side, 5 the interface state)
template <bool STATE>
HD int gks_flux(const double n[3], double weight, bool bnd, const double WL[5], const double GL[15], const double WR[5],
                const double GR[15], double dt, const Phys& ph, const double* tab, double F[5], double Wg[5],
                double& alpha) {
  const double gm1 = ph.gamma - 1.0, k2 = 0.5 * (ph.K + 2.0);
  GksSide gl, gr;
  const bool okl = gks_side(WL, n, 1.0, gm1, tab, gl), okr = gks_side(WR, n, -1.0, gm1, tab, gr);
  int bad = okl && okr ? 0 : 4;
  // interface equilibrium W^c = int_{u>0} psi g^l + int_{u<0} psi g^r (Eq. compatibility2)
  const double a0 = gl.rho * gl.m0, b0 = gr.rho * gr.m0;
  const double al1 = gl.U * gl.m0 + gl.h * gl.beta, ar1 = gr.U * gr.m0 + gr.h * gr.beta;
  const double rho = a0 + b0, Mn = gl.rho * al1 + gr.rho * ar1;
  const double r = fast_rcp(rho), U = Mn * r;
  double ut[3], jm2 = 0.0, jl2 = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    ut[d] = (a0 * gl.ut[d] + b0 * gr.ut[d]) * r;
    const double x = gl.ut[d] - ut[d], y = gr.ut[d] - ut[d];
    jl2 += x * x;
    jm2 += y * y;
  }
  // energy in the frame moving with the tangential velocity of the interface
  const double el = 0.5 * (gl.U * al1 + gl.h * gl.m0) + (k2 * gl.h + 0.5 * jl2) * gl.m0;
  const double er = 0.5 * (gr.U * ar1 + gr.h * gr.m0) + (k2 * gr.h + 0.5 * jm2) * gr.m0;
  const double E = gl.rho * el + gr.rho * er;
  const double p = gm1 * (E - 0.5 * Mn * U), h = p * r;
  if (!(positive(rho) && positive(p)) && !bad) bad = 5;
  // collision times (Sec. 2.3)
  const double jump = fabs((gl.p - gr.p) * fast_rcp(gl.p + gr.p));
  double tau, tn;
  if (ph.viscous) {
    tau = viscosity<double>(ph, ph.gamma * h) * fast_rcp(p);
    tn = tau + ph.c_press * jump * dt;
  } else {
    tn = (ph.eps_inviscid + ph.c_press * jump) * dt;
    tau = tn;
  }
  // exact integrals over [0, dt] of the time coefficients
  // (tn vanishes where the viscosity and the pressure jump do)
  const double edt = positive(tn) ? exp_neg(dt * fast_rcp(tn), tab) : 0.0, om = 1.0 - edt;
  const double q4 = tn * om, tte = tn * dt * edt;
  const double q1 = dt - q4, q5 = (tau + tn) * q4 - tte;
  const double q2 = q5 - tau * dt;
  const double q3 = 0.5 * dt * dt - tau * dt + tau * q4;
  const GksTime t{q4, q5, tau * q4, edt, edt * (tau + dt), edt * tau};
  const bool heat = ph.viscous && ph.prandtl != 1.0;
  alpha = 1.0;
  if (STATE && !bnd && ph.cf) {  // compression factor (interior faces), 1/sqrt(gamma h) = sl sqrt(2/gamma)
    const double dp = fabs(gl.p - gr.p);
    double dm = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double x = gl.u[d] * gl.sl - gr.u[d] * gr.sl;
      dm += x * x;
    }
    const double A = dp * (gl.r * gl.l2 + gr.r * gr.l2) + (2.0 / ph.gamma) * dm;
    alpha = fast_rcp(1.0 + A * A);
  }
  GksAcc a;
  gks_add_side<STATE, true>(gl, GL, n, ut, gm1, ph.gamma, k2, t, heat, a);
  gks_add_side<STATE, false>(gr, GR, n, ut, gm1, ph.gamma, k2, t, heat, a);
  // equilibrium part, full space: X = (0, 1, 2 m1, 3 m2, 4 m3), Y = (0, 0, 1, 3 m1, 6 m2)
  {
    double Rn[3], gp[3], th[3], Tn[3], TS[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      Rn[k] = a.mn[k] - U * a.rho[k];
      double x = a.e[k] - U * a.mn[k];
      x += (0.5 * U * U) * a.rho[k];
      gp[k] = gm1 * x;
      th[k] = gp[k] - h * a.rho[k];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      Tn[i] = n[0] * a.T[i][0] + n[1] * a.T[i][1] + n[2] * a.T[i][2];
      TS[i] = ut[0] * a.T[i][0] + ut[1] * a.T[i][1] + ut[2] * a.T[i][2];
    }
    const double rn = n[0] * a.rho[0] + n[1] * a.rho[1] + n[2] * a.rho[2];
    const double Rnn = n[0] * Rn[0] + n[1] * Rn[1] + n[2] * Rn[2];
    const double thn = n[0] * th[0] + n[1] * th[1] + n[2] * th[2];
    const double rS = ut[0] * a.rho[0] + ut[1] * a.rho[1] + ut[2] * a.rho[2];
    const double RnS = ut[0] * Rn[0] + ut[1] * Rn[1] + ut[2] * Rn[2];
    const double thS = ut[0] * th[0] + ut[1] * th[1] + ut[2] * th[2];
    const double Dv = (a.T[0][0] + a.T[1][1] + a.T[2][2]) - (n[0] * Tn[0] + n[1] * Tn[1] + n[2] * Tn[2]);
    const double m2 = U * U + h, m3 = U * m2 + 2.0 * h * U, m4 = U * m3 + 3.0 * h * m2;
    const double X2 = 2.0 * U, X3 = 3.0 * m2, X4 = 4.0 * m3, Y3 = 3.0 * U, Y4 = 2.0 * X3, kap = k2 * h;
    const double rSD = rS + Dv;
    const double c0 = U * rn + Rnn + rSD;  // <u^k (a.u)>: minus the time derivatives of mass, momentum, ...
    double c1 = m2 * rn + X2 * Rnn + thn;
    c1 += U * rSD;
    c1 += RnS;
    double c2 = m3 * rn + X3 * Rnn + Y3 * thn;
    c2 += m2 * rSD;
    c2 += X2 * RnS;
    c2 += thS;
    double c3 = m4 * rn + X4 * Rnn + Y4 * thn;
    c3 += m3 * rSD;
    c3 += X3 * RnS;
    c3 += Y3 * thS;
    double e0 = 0.5 * c2 + kap * c0;
    e0 += k2 * (U * thn + thS);
    e0 += h * Dv;
    double e1 = 0.5 * c3 + kap * c1;
    e1 += (k2 * m2) * thn;
    e1 += (k2 * U) * thS;
    e1 += (h * U) * Dv;
    double T0[3], T1[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      T0[i] = U * Tn[i] + (TS[i] + gp[i]);
      T1[i] = m2 * Tn[i] + h * a.mn[i];
      T1[i] += U * (TS[i] + th[i]);
    }
    // minus the time slope's rows in u psi
    const double Rt = c1 - U * c0;
    double pt = e0 - U * c1;
    pt += (0.5 * U * U) * c0;
    const double tht = gm1 * pt - h * c0;
    const double A2 = m2 * c0 + X2 * Rt + tht;
    const double A3 = m3 * c0 + X3 * Rt + Y3 * tht;
    double eA = 0.5 * A3 + kap * c1;
    eA += (k2 * U) * tht;
    const double q23 = q2 - q3;
    a.F0 += q1 * Mn;
    a.F0 += q23 * c1;
    a.F1 += q1 * (Mn * U + p);
    a.F1 += q2 * c2;
    a.F1 -= q3 * A2;
    a.F4 += (q1 * U) * (E + p);
    a.F4 += q2 * e1;
    a.F4 -= q3 * eA;
    const double q3U = q3 * U;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      a.FT[i] += q2 * T1[i];
      a.FT[i] -= q3U * T0[i];
    }
    if (STATE) {
      const double od = om * dt;
      a.W0 += om * rho;
      a.W0 -= od * c0;
      a.W1 += om * Mn;
      a.W1 -= od * c1;
      a.W4 += om * E;
      a.W4 -= od * e0;
#pragma unroll
      for (int i = 0; i < 3; ++i) a.WT[i] -= od * T0[i];
    }
    if (heat) {
      // heat flux about U^c of the time-integrated distribution, scaled by (1/Pr - 1); its normal
      // momentum is the mass flux F0
      const double I0 = a.I0 + q1 * rho + q23 * c0, I4 = a.I4 + q1 * E + q23 * e0;
      const double U2 = U * U;
      double qn = a.F4 - U * (a.F1 + I4);
      qn += (1.5 * U2) * a.F0;
      qn -= (0.5 * U2 * U) * I0;
      a.F4 += (1.0 / ph.prandtl - 1.0) * qn;
    }
  }
  const double hut2 = 0.5 * (ut[0] * ut[0] + ut[1] * ut[1] + ut[2] * ut[2]);
  gks_to_global(a.F0, a.F1, a.F4, a.FT, n, ut, hut2, weight * fast_rcp(dt), F);
  if (STATE) {
    gks_to_global(a.W0, a.W1, a.W4, a.WT, n, ut, hut2, 1.0, Wg);
  }
  return bad;
}
