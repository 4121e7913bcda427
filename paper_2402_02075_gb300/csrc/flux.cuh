// The time-dependent gas-kinetic flux of a Gauss point (Eq. 2nd-flux of the paper, Sec. 2.3-2.4) in FP64.
//
// The FP64 pipe bounds it, so the form is the one with the fewest FP64 instructions found so far.  It
// evaluates the same integrals as point_flux (flux_generic.cuh), the form that the tests compare it with:
//  - gradients are primitive: for every direction k of the global frame (d rho, R_i = rho d u_i, d p).
//    The micro-slope of a Maxwellian is diagonal in them: with the peculiar velocity u - U,
//    h = p/rho and th = d p - h d rho,
//      a = (1/rho) [d rho + R.(u - U)/h + th/h (|u - U|^2 + xi^2 - (K + 3) h)/(2 h)],
//    and the Euler equations give its time slope in a few operations (dt rho = -u.d rho - tr R, ...);
//  - with m_k = <u_n^k> over the half space divided by rho, and beta = +-g(0)/rho, integration by parts
//    in u_n gives the normal moments of a slope (d, R_n, th) without any division or coefficient:
//      D_k = <u_n^k a> = m_k d + X_k R_n + Y_k th,
//      X = (beta, m_0, 2 m_1, 3 m_2),  Y = (-beta U/(2 h), beta/2, m_0, 3 m_1);
//    the tangential momentum row is m_k R, the energy row D_{k+2}/2 + (K+2)/2 (h D_k + m_k th);
//  - with A the time slope, -A = u.d + ... as a slope (rt, Rt, tht), the rows of a.u are those of -A plus the
//    non-equilibrium part alone, which the recurrences of X and Y in k reduce to
//      a_k d_n th + h Y_k sig,  a_k = Y_{k+1} - U Y_k - X_k,  sig = 2 d_n R_n - (gamma - 1) tr R
//    (heat flux and normal stress) in the normal rows and h X_k (d_n R_i + d_i R_n) + h Y_k d_i th (shear) in
//    the tangential ones;
//  - no face frame: a vector is kept in the global frame, its normal component taken with n where it is
//    needed, so nothing is rotated in or out.  Tangential vectors may carry a normal component that
//    the final projection removes;
//  - both sides' moments are summed in the frame moving with the interface's tangential velocity, where
//    the heat flux of the Prandtl correction needs three of the time-integrated moments only.
// Measured on the 96x64x69 boundary layer (10.67 M points), CUDA events: 23.5 ms with the interface
// state, 21.2 ms the flux alone (1,256 and 1,135 FP64 instructions per point), against 37.6 and 35.6 ms
// (2,007 and 1,900) by point_flux<double>.  Blocks of 32, 64 and 128 threads take the same time; three or
// four blocks of 128 per SM (168 or 128 registers, with spills) 2 to 3 % more.
#pragma once
#include "fastmath.cuh"
#include "kinetic.cuh"

// The state dependence can be differentiated by dual numbers: S is the scalar of a side's state, T of
// what both sides and the time step enter (double for the flux itself; one of the sides or both DualD
// for a column of the linearisation); gradients stay double.

// one side of the interface: state, half-space seeds
template <typename S>
struct GksSide {
  S rho, r, u[3], U, ut[3];  // density, 1/rho, velocity, its normal and tangential parts
  S p, h, l2, sl;            // pressure, p/rho, rho/p, 1/sqrt(2 h)
  S m0, beta;                // half-space mass fraction, s g(0)/rho (s the side: u_n > 0 or < 0)
};

// s = +1 left, -1 right; false where the state is not physical
template <typename S>
HD bool gks_side(const S w[5], const double n[3], double s, double gm1, const double* tab, GksSide<S>& g) {
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
  S e;
  half_gauss(-s * (g.sl * g.U), tab, g.m0, e);
  g.beta = (s * 0.56418958354775628695) * (e * g.sl);
  return positive(w[0]) && positive(g.p);
}

// time coefficients of Eq. 2nd-flux integrated over [0, dt] that multiply the two sides' moments
template <typename T>
struct GksTime {
  T q4, q5, q54;    // in the flux: of g, of -(a.u) g, and that less the one of -A g
  T edt, etd, edd;  // the same in the interface state at dt
};

// sums over both sides in the frame moving with the interface's tangential velocity: gradients of the
// interface equilibrium (mass, normal momentum, tangential momentum and energy, per direction) and the
// moments of the time-integrated flux (F), of the state at dt (W) and of the time-integrated state (I)
template <typename T>
struct GksAcc {
  T rho[3], mn[3], Tm[3][3], e[3];
  T F0, F1, F4, FT[3], W0, W1, W4, WT[3], I0, I4;
};

// adds one side: G the conservative gradients (15), ut_c the interface's tangential velocity.  STATE: the
// state at dt as well; heat: the time-integrated state's rows that the Prandtl correction uses.  FIRST:
// the sums start with this side
template <bool STATE, bool FIRST, typename S, typename T>
HD void gks_add_side(const GksSide<S>& g, const double G[15], const double n[3], const T utc[3], double gm1, double gamma,
                     double k2, const GksTime<T>& t, bool heat, GksAcc<T>& a) {
  T del[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) del[d] = g.ut[d] - utc[d];
  const T hd2 = 0.5 * (del[0] * del[0] + del[1] * del[1] + del[2] * del[2]);
  const S hu2 = 0.5 * (g.u[0] * g.u[0] + g.u[1] * g.u[1] + g.u[2] * g.u[2]);
  // primitive gradients
  S R[3][3], gp[3], th[3], Rn[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int i = 0; i < 3; ++i) R[i][k] = G[3 * (1 + i) + k] - g.u[i] * G[k];
    S x = G[12 + k] - hu2 * G[k];
    x -= g.u[0] * R[0][k];
    x -= g.u[1] * R[1][k];
    x -= g.u[2] * R[2][k];
    gp[k] = gm1 * x;
    th[k] = gp[k] - g.h * G[k];
    Rn[k] = n[0] * R[0][k] + n[1] * R[1][k] + n[2] * R[2][k];
  }
  // moments and the coefficients X_k, Y_k
  const S U = g.U, h = g.h, m0 = g.m0, beta = g.beta;
  const S hb = h * beta, m1 = U * m0 + hb;
  const S hm0 = h * m0, m2 = U * m1 + hm0;
  const S hm1 = h * m1, m3 = U * m2 + 2.0 * hm1;
  const S X2 = 2.0 * m1, X3 = 3.0 * m2;
  const S Y0 = -0.5 * U * (beta * g.l2), Y1 = 0.5 * beta, Y3 = 3.0 * m1;
  const S kap = k2 * h, k2m0 = k2 * m0, k2m1 = k2 * m1;
  const T kd = hd2 + kap;
  T dm0[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) dm0[d] = del[d] * m0;
  // gradients of the interface equilibrium
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const S D0 = m0 * G[k] + beta * Rn[k] + Y0 * th[k];
    const S D1 = m1 * G[k] + m0 * Rn[k] + Y1 * th[k];
    const S D2 = m2 * G[k] + X2 * Rn[k] + m0 * th[k];
    T e = FIRST ? T(0.5 * D2) : a.e[k] + 0.5 * D2;
    e += kd * D0;
    e += k2m0 * th[k];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      e += dm0[i] * R[i][k];
      const T v = FIRST ? T(m0 * R[i][k]) : a.Tm[i][k] + m0 * R[i][k];
      a.Tm[i][k] = v + del[i] * D0;
    }
    a.e[k] = e;
    a.rho[k] = FIRST ? T(D0) : a.rho[k] + D0;
    a.mn[k] = FIRST ? T(D1) : a.mn[k] + D1;
  }
  // derivatives along n and along the tangential velocity
  const S rn = n[0] * G[0] + n[1] * G[1] + n[2] * G[2];
  const S thn = n[0] * th[0] + n[1] * th[1] + n[2] * th[2];
  const S rS = g.ut[0] * G[0] + g.ut[1] * G[1] + g.ut[2] * G[2];
  const S thS = g.ut[0] * th[0] + g.ut[1] * th[1] + g.ut[2] * th[2];
  S Rv[3], Rt[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Rv[i] = n[0] * R[i][0] + n[1] * R[i][1] + n[2] * R[i][2];
    S x = gp[i] + U * Rv[i];
    x += g.ut[0] * R[i][0];
    x += g.ut[1] * R[i][1];
    x += g.ut[2] * R[i][2];
    Rt[i] = x;
  }
  const S Rnn = n[0] * Rv[0] + n[1] * Rv[1] + n[2] * Rv[2];
  const S Rnt = n[0] * Rt[0] + n[1] * Rt[1] + n[2] * Rt[2];
  const S tr = R[0][0] + R[1][1] + R[2][2];
  // minus the time derivatives (Euler)
  const S rt = U * rn + (rS + tr);
  const S tht = U * thn + thS + (gm1 * h) * tr;
  // rows of -<u_n^k A psi>, k = 0..3, and the coefficients a_k, h Y_k of the non-equilibrium part
  const S At0 = m0 * rt + beta * Rnt + Y0 * tht;
  const S At1 = m1 * rt + m0 * Rnt + Y1 * tht;
  const S At2 = m2 * rt + X2 * Rnt + m0 * tht;
  const S At3 = m3 * rt + X3 * Rnt + Y3 * tht;
  const S a0 = U * Y0 + Y1, a1 = U * Y1, a3 = 3.0 * hm0;  // minus a_0, minus a_1; a_2 = h beta
  const S b0 = h * Y0, b1 = 0.5 * hb, b3 = 3.0 * hm1;     // b_2 = h m_0
  const S sig = 2.0 * Rnn - gm1 * tr, dvs = (1.0 - gm1 * k2) * tr - Rnn;
#pragma unroll
  for (int i = 0; i < 3; ++i) Rv[i] = Rv[i] + Rn[i];  // the shear d_n R_i + d_i R_n from here on
  const S v4 = 0.5 * m2 + kap * m0, f4 = 0.5 * m3 + kap * m1;  // energy rows of psi and u psi
  {
    // flux: q4 <u psi> - q5 <u (a.u) psi> - tau q4 <u A psi>
    const T qr = t.q4 * g.rho, hn = t.q5 * thn, hs = t.q5 * sig, hd = t.q5 * dvs, ht = t.q54 * tht;
    T z1 = t.q54 * At1 - a1 * hn;
    z1 += b1 * hs;
    T z2 = t.q54 * At2 + hb * hn;
    z2 += hm0 * hs;
    T z3 = t.q54 * At3 + a3 * hn;
    z3 += b3 * hs;
    const T F0 = qr * m1 - z1, F1 = qr * m2 - z2;
    T F4 = qr * f4 - 0.5 * z3;
    F4 -= kap * z1;
    F4 -= k2m1 * ht;
    F4 -= (kap * m0) * hn;
    F4 -= hm1 * hd;
    F4 += hd2 * F0;
    const T cA = t.q54 * m1, cS = t.q5 * hm0, ch = t.q5 * b1;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      T v = cA * Rt[i] + cS * Rv[i];
      v += ch * th[i];
      F4 -= del[i] * v;
      const T x = del[i] * F0 - v;
      a.FT[i] = FIRST ? x : a.FT[i] + x;
    }
    a.F0 = FIRST ? F0 : a.F0 + F0;
    a.F1 = FIRST ? F1 : a.F1 + F1;
    a.F4 = FIRST ? F4 : a.F4 + F4;
    if (heat) {
      T z0 = t.q54 * At0 - a0 * hn;
      z0 += b0 * hs;
      const T I0 = qr * m0 - z0;
      T I4 = qr * v4 - 0.5 * z2;
      I4 -= kap * z0;
      I4 -= k2m0 * ht;
      I4 -= (k2 * hb) * hn;
      I4 -= hm0 * hd;
      I4 += hd2 * I0;
      const T dA = t.q54 * m0, dS = t.q5 * hb, dh = t.q5 * b0;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        T v = dA * Rt[i] + dS * Rv[i];
        v += dh * th[i];
        I4 -= del[i] * v;
      }
      a.I0 = FIRST ? I0 : a.I0 + I0;
      a.I4 = FIRST ? I4 : a.I4 + I4;
    }
  }
  if (STATE) {
    const T qr = t.edt * g.rho, hn = t.etd * thn, hs = t.etd * sig, hd = t.etd * dvs, ht = t.edd * tht;
    T z0 = t.edd * At0 - a0 * hn;
    z0 += b0 * hs;
    T z1 = t.edd * At1 - a1 * hn;
    z1 += b1 * hs;
    T z2 = t.edd * At2 + hb * hn;
    z2 += hm0 * hs;
    const T W0 = qr * m0 - z0, W1 = qr * m1 - z1;
    T W4 = qr * v4 - 0.5 * z2;
    W4 -= kap * z0;
    W4 -= k2m0 * ht;
    W4 -= (k2 * hb) * hn;
    W4 -= hm0 * hd;
    W4 += hd2 * W0;
    const T dA = t.edd * m0, dS = t.etd * hb, dh = t.etd * b0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      T v = dA * Rt[i] + dS * Rv[i];
      v += dh * th[i];
      W4 -= del[i] * v;
      const T x = del[i] * W0 - v;
      a.WT[i] = FIRST ? x : a.WT[i] + x;
    }
    a.W0 = FIRST ? W0 : a.W0 + W0;
    a.W1 = FIRST ? W1 : a.W1 + W1;
    a.W4 = FIRST ? W4 : a.W4 + W4;
  }
}

// moments (mass F0, normal momentum F1, tangential momentum Ft, energy F4) of the frame moving with the
// tangential velocity ut -> conservative vector of the global frame, times c
template <typename T, typename C>
HD void gks_to_global(T F0, T F1, T F4, const T Ft[3], const double n[3], const T ut[3], T hut2, C c, T out[5]) {
  out[0] = c * F0;
  const T x = F1 - (n[0] * Ft[0] + n[1] * Ft[1] + n[2] * Ft[2]);
  T e = F4 + hut2 * F0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    e += ut[i] * Ft[i];
    T v = Ft[i] + ut[i] * F0;
    v += x * n[i];
    out[1 + i] = c * v;
  }
  out[4] = c * e;
}

// mu(T), t = T/T_inf: fine.cuh
template <typename T>
HD T viscosity(const Phys& ph, T t);

// what the equilibrium part of a flux and of a column of its linearisation share
template <typename T>
struct GksCentre {
  T rho, Mn, U, p, h, E, ut[3];            // density, momentum, velocity, ..., energy in the moving frame
  T om, q1, q2, q3, dt;                    // time coefficients of its terms, the time step
  GksTime<T> t;
};

// interface equilibrium W^c = int_{u>0} psi g^l + int_{u<0} psi g^r (Eq. compatibility2), the collision
// times and the integrals over [0, dt] of the time coefficients; false where the state is not physical
template <typename SL, typename SR, typename T, typename D>
HD bool gks_centre(const GksSide<SL>& gl, const GksSide<SR>& gr, D dt, const Phys& ph, const double* tab, GksCentre<T>& c) {
  const double gm1 = ph.gamma - 1.0, k2 = 0.5 * (ph.K + 2.0);
  const SL a0 = gl.rho * gl.m0, al1 = gl.U * gl.m0 + gl.h * gl.beta;
  const SR b0 = gr.rho * gr.m0, ar1 = gr.U * gr.m0 + gr.h * gr.beta;
  c.rho = a0 + b0;
  c.Mn = gl.rho * al1 + gr.rho * ar1;
  const T r = fast_rcp(c.rho);
  c.U = c.Mn * r;
  T jl2 = 0.0, jr2 = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    c.ut[d] = (a0 * gl.ut[d] + b0 * gr.ut[d]) * r;
    const T x = gl.ut[d] - c.ut[d], y = gr.ut[d] - c.ut[d];
    jl2 += x * x;
    jr2 += y * y;
  }
  // energy in the frame moving with the tangential velocity of the interface
  const T el = 0.5 * (gl.U * al1 + gl.h * gl.m0) + (0.5 * jl2 + k2 * gl.h) * gl.m0;
  const T er = 0.5 * (gr.U * ar1 + gr.h * gr.m0) + (0.5 * jr2 + k2 * gr.h) * gr.m0;
  c.E = gl.rho * el + gr.rho * er;
  c.p = gm1 * (c.E - 0.5 * c.Mn * c.U);
  c.h = c.p * r;
  // collision times (Sec. 2.3)
  const T jump = fabs((gl.p - gr.p) * fast_rcp(gl.p + gr.p));
  T tau, tn;
  if (ph.viscous) {
    tau = viscosity<T>(ph, ph.gamma * c.h) * fast_rcp(c.p);
    tn = tau + ph.c_press * jump * dt;
  } else {
    tn = (ph.eps_inviscid + ph.c_press * jump) * dt;
    tau = tn;
  }
  // exact integrals over [0, dt] of the time coefficients
  // (tn vanishes where the viscosity and the pressure jump do)
  T edt = 0.0;
  if (positive(tn)) edt = exp_neg(dt * fast_rcp(tn), tab);
  c.om = 1.0 - edt;
  c.dt = dt;
  const T q4 = tn * c.om, tte = tn * dt * edt;
  c.q1 = dt - q4;
  c.t.q4 = q4;
  c.t.q54 = tn * q4 - tte;
  c.t.q5 = c.t.q54 + tau * q4;
  c.t.edt = edt;
  c.t.edd = edt * dt;
  c.t.etd = c.t.edd + edt * tau;
  c.q2 = c.t.q5 - tau * dt;
  c.q3 = 0.5 * dt * dt - tau * dt + tau * q4;
  return positive(c.rho) && positive(c.p);
}

// flux of one Gauss point: n the unit normal, weight the length of its area vector; WL, GL, WR, GR the
// states and gradients of both sides (global frame; on a boundary face the ghost's), dt the face's time
// step.  F: flux x weight averaged over dt; Wg (STATE): the interface state at dt; alpha (STATE): the
// compression factor (1 on boundary faces and with the factor off).  Returns 0, or the number of the
// check that failed (4 a side, 5 the interface state).  T: the wider of the scalars of the sides and the time
// step; n, weight and the gradients are double.  gks_flux is the flux itself, gks_flux_t its dual form
template <bool STATE, typename SL, typename SR, typename T, typename D>
HD int gks_flux_t(const double n[3], double weight, bool bnd, const SL WL[5], const double GL[15], const SR WR[5],
                  const double GR[15], D dt, const Phys& ph, const double* tab, T F[5], T Wg[5], T& alpha) {
  const double gm1 = ph.gamma - 1.0, k2 = 0.5 * (ph.K + 2.0);
  GksSide<SL> gl;
  GksSide<SR> gr;
  const bool okl = gks_side(WL, n, 1.0, gm1, tab, gl), okr = gks_side(WR, n, -1.0, gm1, tab, gr);
  GksCentre<T> c;
  const bool okc = gks_centre<SL, SR, T, D>(gl, gr, dt, ph, tab, c);
  const int bad = !(okl && okr) ? 4 : (okc ? 0 : 5);
  const T rho = c.rho, Mn = c.Mn, U = c.U, p = c.p, h = c.h, E = c.E, om = c.om, q1 = c.q1, q2 = c.q2, q3 = c.q3;
  const T(&ut)[3] = c.ut;
  const GksTime<T>& t = c.t;
  const bool heat = ph.viscous && ph.prandtl != 1.0;
  alpha = 1.0;
  if (STATE && !bnd && ph.cf) {  // compression factor (interior faces), 1/sqrt(gamma h) = sl sqrt(2/gamma)
    const T dp = fabs(gl.p - gr.p);
    T dm = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const T x = gl.u[d] * gl.sl - gr.u[d] * gr.sl;
      dm += x * x;
    }
    const T A = dp * (gl.r * gl.l2 + gr.r * gr.l2) + (2.0 / ph.gamma) * dm;
    alpha = fast_rcp(1.0 + A * A);
  }
  GksAcc<T> a;
  gks_add_side<STATE, true, SL, T>(gl, GL, n, ut, gm1, ph.gamma, k2, t, heat, a);
  gks_add_side<STATE, false, SR, T>(gr, GR, n, ut, gm1, ph.gamma, k2, t, heat, a);
  // equilibrium part, full space: X = (0, 1, 2 m1, 3 m2), Y = (0, 0, 1, 3 m1)
  {
    T Rn[3], th[3], Tn[3], T0[3];
    const T hU2 = 0.5 * U * U;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      Rn[k] = a.mn[k] - U * a.rho[k];
      T x = a.e[k] - U * a.mn[k];
      x += hU2 * a.rho[k];
      T0[k] = gm1 * x;  // pressure gradient, then minus the tangential momentum's time derivative
      th[k] = T0[k] - h * a.rho[k];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      Tn[i] = n[0] * a.Tm[i][0] + n[1] * a.Tm[i][1] + n[2] * a.Tm[i][2];
      T0[i] += U * Tn[i];
      T0[i] += ut[0] * a.Tm[i][0];
      T0[i] += ut[1] * a.Tm[i][1];
      T0[i] += ut[2] * a.Tm[i][2];
    }
    const T rn = n[0] * a.rho[0] + n[1] * a.rho[1] + n[2] * a.rho[2];
    const T Rnn = n[0] * Rn[0] + n[1] * Rn[1] + n[2] * Rn[2];
    const T thn = n[0] * th[0] + n[1] * th[1] + n[2] * th[2];
    const T rS = ut[0] * a.rho[0] + ut[1] * a.rho[1] + ut[2] * a.rho[2];
    const T RnS = ut[0] * Rn[0] + ut[1] * Rn[1] + ut[2] * Rn[2];
    const T thS = ut[0] * th[0] + ut[1] * th[1] + ut[2] * th[2];
    const T Dv = (a.Tm[0][0] + a.Tm[1][1] + a.Tm[2][2]) - (n[0] * Tn[0] + n[1] * Tn[1] + n[2] * Tn[2]);
    const T tr = Dv + Rnn;
    const T m2 = U * U + h, m3 = U * m2 + 2.0 * h * U, kap = k2 * h;
    // minus the time derivatives: mass, normal momentum (Rt, c1 with the mass's), th
    const T c0 = U * rn + (rS + tr);
    T Rt = U * Rnn + (RnS + thn);
    Rt += h * rn;
    const T c1 = U * c0 + Rt;
    const T tht = U * thn + thS + (gm1 * h) * tr;
    const T sig = 2.0 * Rnn - gm1 * tr, dvs = (1.0 - gm1 * k2) * tr - Rnn;
    T A2 = m2 * c0 + tht;
    A2 += (2.0 * U) * Rt;
    T A3 = m3 * c0 + (3.0 * m2) * Rt;
    A3 += (3.0 * U) * tht;
    T eA = 0.5 * A3 + kap * c1;
    eA += (k2 * U) * tht;
    T e1 = (k2 + 1.5) * thn + (1.5 * U) * sig;  // non-equilibrium energy flux over h
    e1 += U * dvs;
    const T q23 = q2 - q3, q2h = q2 * h;
    a.F0 += q1 * Mn;
    a.F0 += q23 * c1;
    a.F1 += q1 * (Mn * U + p);
    a.F1 += q23 * A2;
    a.F1 += q2h * sig;
    a.F4 += (q1 * U) * (E + p);
    a.F4 += q23 * eA;
    a.F4 += q2h * e1;
    const T qU = q23 * U;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      a.FT[i] += qU * T0[i];
      a.FT[i] += q2h * (Tn[i] + Rn[i]);
    }
    T e0 = 0.5 * A2 + kap * c0;  // energy's time derivative (minus)
    e0 += k2 * tht;
    e0 += h * (dvs + 0.5 * sig);
    if (STATE) {
      const T od = om * c.dt;
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
      const T I0 = a.I0 + q1 * rho + q23 * c0, I4 = a.I4 + q1 * E + q23 * e0;
      const T U2 = U * U;
      T qn = a.F4 - U * (a.F1 + I4);
      qn += (1.5 * U2) * a.F0;
      qn -= (0.5 * U2 * U) * I0;
      a.F4 += (1.0 / ph.prandtl - 1.0) * qn;
    }
  }
  const T hut2 = 0.5 * (ut[0] * ut[0] + ut[1] * ut[1] + ut[2] * ut[2]);
  gks_to_global(a.F0, a.F1, a.F4, a.FT, n, ut, hut2, weight * fast_rcp(dt), F);
  if (STATE) {
    gks_to_global(a.W0, a.W1, a.W4, a.WT, n, ut, hut2, 1.0, Wg);
  }
  return bad;
}

// the flux itself
template <bool STATE>
HD int gks_flux(const double n[3], double weight, bool bnd, const double WL[5], const double GL[15], const double WR[5],
                const double GR[15], double dt, const Phys& ph, const double* tab, double F[5], double Wg[5],
                double& alpha) {
  return gks_flux_t<STATE, double, double, double, double>(n, weight, bnd, WL, GL, WR, GR, dt, ph, tab, F, Wg, alpha);
}

// response of a point's time-averaged flux x weight / dt (out 0..4) and interface state (out 5..9), both
// linear in the gradients, to a unit of the gradient dW = A along the direction d (d W_q/dx_k = A_q d_k) of
// one side: gks_flux with a gradient of rank one, where every derivative is that amplitude times n.d, u_t.d
// or d itself
HD void gks_gradient_column(const GksSide<double>& g, const GksCentre<double>& c, const double A[5], const double d[3],
                            const double n[3], double sdt, const Phys& ph, double out[10]) {
  const double gm1 = ph.gamma - 1.0, k2 = 0.5 * (ph.K + 2.0);
  const double U = g.U, h = g.h, m0 = g.m0, beta = g.beta;
  double del[3], R[3];
  const double hu2 = 0.5 * (g.u[0] * g.u[0] + g.u[1] * g.u[1] + g.u[2] * g.u[2]);
  double x = A[4] - hu2 * A[0];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    del[i] = g.ut[i] - c.ut[i];
    R[i] = A[1 + i] - g.u[i] * A[0];
    x -= g.u[i] * R[i];
  }
  const double hd2 = 0.5 * (del[0] * del[0] + del[1] * del[1] + del[2] * del[2]);
  const double gr = A[0], gp = gm1 * x, th = gp - h * gr, Rn = n[0] * R[0] + n[1] * R[1] + n[2] * R[2];
  const double dn = n[0] * d[0] + n[1] * d[1] + n[2] * d[2];
  const double ds = g.ut[0] * d[0] + g.ut[1] * d[1] + g.ut[2] * d[2], ud = U * dn + ds;
  const double hb = h * beta, m1 = U * m0 + hb, hm0 = h * m0, m2 = U * m1 + hm0, hm1 = h * m1, m3 = U * m2 + 2.0 * hm1;
  const double X2 = 2.0 * m1, X3 = 3.0 * m2, Y0 = -0.5 * U * (beta * g.l2), Y1 = 0.5 * beta, Y3 = 3.0 * m1;
  const double kap = k2 * h, k2m0 = k2 * m0, k2m1 = k2 * m1;
  const double D0 = m0 * gr + beta * Rn + Y0 * th, D1 = m1 * gr + m0 * Rn + Y1 * th, D2 = m2 * gr + X2 * Rn + m0 * th;
  const double tr = R[0] * d[0] + R[1] * d[1] + R[2] * d[2], Rnn = dn * Rn;
  const double rt = ud * gr + tr, Rnt = ud * Rn + gp * dn, tht = ud * th + (gm1 * h) * tr, thn = dn * th;
  const double At0 = m0 * rt + beta * Rnt + Y0 * tht, At1 = m1 * rt + m0 * Rnt + Y1 * tht,
               At2 = m2 * rt + X2 * Rnt + m0 * tht, At3 = m3 * rt + X3 * Rnt + Y3 * tht;
  const double a0 = -(U * Y0 + Y1), a1 = -(U * Y1), a3 = 3.0 * hm0, b0 = h * Y0, b1 = 0.5 * hb, b3 = 3.0 * hm1;
  const double sig = 2.0 * Rnn - gm1 * tr, dvs = (1.0 - gm1 * k2) * tr - Rnn;
  double F0, F1, F4, FT[3], W0, W1, W4, WT[3], I0 = 0.0, I4 = 0.0;
  const bool heat = ph.viscous && ph.prandtl != 1.0;
  {
    const GksTime<double>& t = c.t;
    const double hn = t.q5 * thn, hs = t.q5 * sig, hd = t.q5 * dvs, ht = t.q54 * tht;
    const double wn = t.etd * thn, ws = t.etd * sig, wd = t.etd * dvs, wt = t.edd * tht;
    const double z0 = t.q54 * At0 + a0 * hn + b0 * hs, z1 = t.q54 * At1 + a1 * hn + b1 * hs,
                 z2 = t.q54 * At2 + hb * hn + hm0 * hs, z3 = t.q54 * At3 + a3 * hn + b3 * hs;
    const double y0 = t.edd * At0 + a0 * wn + b0 * ws, y1 = t.edd * At1 + a1 * wn + b1 * ws,
                 y2 = t.edd * At2 + hb * wn + hm0 * ws;
    F0 = -z1;
    F1 = -z2;
    F4 = hd2 * F0 - (0.5 * z3 + kap * z1 + k2m1 * ht + (kap * m0) * hn + hm1 * hd);
    W0 = -y0;
    W1 = -y1;
    W4 = hd2 * W0 - (0.5 * y2 + kap * y0 + k2m0 * wt + (k2 * hb) * wn + hm0 * wd);
    if (heat) {
      I0 = -z0;
      I4 = hd2 * I0 - (0.5 * z2 + kap * z0 + k2m0 * ht + (k2 * hb) * hn + hm0 * hd);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double Rt = ud * R[i] + gp * d[i], Sh = dn * R[i] + Rn * d[i], thi = th * d[i];
      const double v = (t.q54 * m1) * Rt + (t.q5 * hm0) * Sh + (t.q5 * b1) * thi;
      const double y = (t.edd * m0) * Rt + (t.etd * hb) * Sh + (t.etd * b0) * thi;
      F4 -= del[i] * v;
      FT[i] = del[i] * F0 - v;
      W4 -= del[i] * y;
      WT[i] = del[i] * W0 - y;
      if (heat) I4 -= del[i] * ((t.q54 * m0) * Rt + (t.q5 * hb) * Sh + (t.q5 * b0) * thi);
    }
  }
  // the interface equilibrium's gradient (amplitudes along d) and its terms
  {
    const double Uc = c.U, hc = c.h, kc = k2 * hc;
    double T[3];
    double e = 0.5 * D2 + (kap + hd2) * D0 + k2m0 * th;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      T[i] = m0 * R[i] + del[i] * D0;
      e += (del[i] * m0) * R[i];
    }
    const double Rc = D1 - Uc * D0, pc = gm1 * (e - Uc * D1 + (0.5 * Uc * Uc) * D0), tc = pc - hc * D0;
    const double dc = c.ut[0] * d[0] + c.ut[1] * d[1] + c.ut[2] * d[2], uc = Uc * dn + dc;
    const double nT = n[0] * T[0] + n[1] * T[1] + n[2] * T[2], rc = dn * Rc;
    const double t2 = (T[0] * d[0] + T[1] * d[1] + T[2] * d[2]) - dn * nT + rc;
    const double n2 = Uc * Uc + hc, n3 = Uc * n2 + 2.0 * hc * Uc;
    const double c0 = uc * D0 + t2, Rt = uc * Rc + pc * dn, c1 = Uc * c0 + Rt, tt = uc * tc + (gm1 * hc) * t2, tn = dn * tc;
    const double sc = 2.0 * rc - gm1 * t2, dv = (1.0 - gm1 * k2) * t2 - rc;
    const double A2 = n2 * c0 + 2.0 * Uc * Rt + tt, A3 = n3 * c0 + 3.0 * n2 * Rt + 3.0 * Uc * tt;
    const double eA = 0.5 * A3 + kc * c1 + (k2 * Uc) * tt, e1 = (k2 + 1.5) * tn + (1.5 * Uc) * sc + Uc * dv;
    const double e0 = 0.5 * A2 + kc * c0 + k2 * tt + hc * (dv + 0.5 * sc);
    const double q23 = c.q2 - c.q3, od = c.om * c.dt, q2h = c.q2 * hc;
    F0 += q23 * c1;
    F1 += q23 * A2 + q2h * sc;
    F4 += q23 * eA + q2h * e1;
    W0 -= od * c0;
    W1 -= od * c1;
    W4 -= od * e0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double T0 = uc * T[i] + pc * d[i];
      FT[i] += (q23 * Uc) * T0 + q2h * (dn * T[i] + Rc * d[i]);
      WT[i] -= od * T0;
    }
    if (heat) {
      I0 += q23 * c0;
      I4 += q23 * e0;
      const double qn = F4 - Uc * (F1 + I4) + (1.5 * Uc * Uc) * F0 - (0.5 * Uc * Uc * Uc) * I0;
      F4 += (1.0 / ph.prandtl - 1.0) * qn;
    }
  }
  const double hut2 = 0.5 * (c.ut[0] * c.ut[0] + c.ut[1] * c.ut[1] + c.ut[2] * c.ut[2]);
  gks_to_global(F0, F1, F4, FT, n, c.ut, hut2, sdt, out);
  gks_to_global(W0, W1, W4, WT, n, c.ut, hut2, 1.0, out + 5);
}
