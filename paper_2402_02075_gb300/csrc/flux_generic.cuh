// The gas-kinetic flux of a Gauss point in a second, independent form on any scalar type: face frame, explicit
// micro-slopes and sparse moment matrices, where flux.cuh has primitive gradients.  The kernels run gks_flux
// (flux.cuh) and the library does not contain this file; the host tests hold gks_flux and its linearisation
// against it in long double and on dual numbers, and the oracle against it in double.
#pragma once
#include "kinetic.cuh"

HD double rsqrt_hd(double x) { return fast_rsqrt(x); }
HD DualD rsqrt_hd(DualD x) { return fast_rsqrt(x); }

// branchless orthonormal basis (t1, t2) completing the unit normal n (Duff et al., JCGT 6(1), 2017)
template <typename T>
HD void face_frame(const T n[3], T t1[3], T t2[3]) {
  const T sign = n[2] >= T(0) ? T(1) : T(-1);
  const T a = T(-1) / (sign + n[2]);
  const T b = n[0] * n[1] * a;
  t1[0] = T(1) + sign * n[0] * n[0] * a;
  t1[1] = sign * b;
  t1[2] = -sign * n[0];
  t2[0] = b;
  t2[1] = sign + n[1] * n[1] * a;
  t2[2] = -n[1];
}

// conservative vector into the face frame and out of it
template <typename T>
HD void rotate_in(const T W[5], const T n[3], const T t1[3], const T t2[3], T w[5]) {
  w[0] = W[0];
  w[1] = W[1] * n[0] + W[2] * n[1] + W[3] * n[2];
  w[2] = W[1] * t1[0] + W[2] * t1[1] + W[3] * t1[2];
  w[3] = W[1] * t2[0] + W[2] * t2[1] + W[3] * t2[2];
  w[4] = W[4];
}

template <typename T>
HD void rotate_out(const T f[5], const T n[3], const T t1[3], const T t2[3], T F[5]) {
  F[0] = f[0];
  F[1] = f[1] * n[0] + f[2] * t1[0] + f[3] * t2[0];
  F[2] = f[1] * n[1] + f[2] * t1[1] + f[3] * t2[1];
  F[3] = f[1] * n[2] + f[2] * t1[2] + f[3] * t2[2];
  F[4] = f[4];
}

// a Maxwellian in the face frame with the reciprocals and products the moments and slopes need
template <typename T>
struct Maxw {
  T rho, U, V, W;  // density, velocity (normal, tangential 1, tangential 2)
  T r, p, h;       // 1/rho, pressure, h = p/rho = 1/(2 lambda)
  T l2, q2;        // 2 lambda = 1/h, |U|^2 + (K+3) h
  T lr, ckr, hq2;  // 2 lambda / rho, 4 lambda^2 / ((K+3) rho), q2 / 2: the slope solve's coefficients
  T hu2, rH;       // |U|^2 / 2, (E + p) / rho: the Euler-flux derivative's
};

// iK3 = 1/(K+3)
template <typename T>
HD bool make_maxw(const T w[5], T gm1, T K, T iK3, Maxw<T>& g) {
  g.rho = w[0];
  g.r = 1.0 / w[0];
  g.U = w[1] * g.r;
  g.V = w[2] * g.r;
  g.W = w[3] * g.r;
  g.p = gm1 * (w[4] - 0.5 * (w[1] * g.U + w[2] * g.V + w[3] * g.W));
  g.h = g.p * g.r;
  g.l2 = 1.0 / g.h;
  const T u2 = g.U * g.U + g.V * g.V + g.W * g.W;
  g.q2 = u2 + (K + 3.0) * g.h;
  g.lr = g.l2 * g.r;
  g.ckr = g.l2 * g.l2 * iK3 * g.r;
  g.hq2 = 0.5 * g.q2;
  g.hu2 = 0.5 * u2;
  g.rH = (w[4] + g.p) * g.r;
  return w[0] > 0.0 && g.p > 0.0;
}

// <u^0>, <u^1> over u > 0 (side +1) or u < 0 (side -1), normalised by rho:
// 1/2 erfc(-s sqrt(lambda) U) and U <u^0> + s exp(-lambda U^2) / (2 sqrt(pi lambda))
template <typename T>
HD void half_seeds(const Maxw<T>& g, T side, T& m0, T& m1) {
  const T lam = 0.5 * g.l2;
  const T isl = rsqrt_hd(lam);
  const T sl = lam * isl;
  m0 = 0.5 * erfc(-side * sl * g.U);
  m1 = g.U * m0 + side * (0.5 * 0.56418958354775628695) * exp(-lam * g.U * g.U) * isl;
}

// micro-slope s with <s psi> = dW under the full Maxwellian g (closed form of the 5x5 system, with
// d = dW / rho: s4 = 4 lambda^2/(K+3) (2 d4 - q2 d0 - 2 U.(d - U d0)), s_i = 2 lambda (d_i - U_i d0)
// - U_i s4, s0 = d0 - U.s - q2 s4 / 2); the 1/rho of d rides in the coefficients lr and ckr
template <typename T>
HD void slope_solve(const Maxw<T>& g, const T dW[5], T s[5]) {
  const T R1 = dW[1] - g.U * dW[0], R2 = dW[2] - g.V * dW[0], R3 = dW[3] - g.W * dW[0];
  const T R4 = 2.0 * dW[4] - g.q2 * dW[0];
  s[4] = g.ckr * (R4 - 2.0 * (g.U * R1 + g.V * R2 + g.W * R3));
  s[1] = g.lr * R1 - g.U * s[4];
  s[2] = g.lr * R2 - g.V * s[4];
  s[3] = g.lr * R3 - g.W * s[4];
  s[0] = g.r * dW[0] - g.U * s[1] - g.V * s[2] - g.W * s[3] - g.hq2 * s[4];
}

// directional derivative of the Euler flux through the k-th axis of the face frame along dW:
// equals <u_k (a . psi) psi> under the full Maxwellian when <a psi> = dW.  With e_j = rho du_j =
// dW_{1+j} - u_j dW_0: d(rho u_k u_j) = dW_{1+k} u_j + u_k e_j, d(u_k (E + p)) = e_k (E + p)/rho +
// u_k (dE + dp)
template <typename T>
HD void euler_jvp(const Maxw<T>& g, T gm1, int k, const T dW[5], T out[5]) {
  const T u[3] = {g.U, g.V, g.W};
  const T e[3] = {dW[1] - u[0] * dW[0], dW[2] - u[1] * dW[0], dW[3] - u[2] * dW[0]};
  const T dp = gm1 * (dW[4] - (u[0] * dW[1] + u[1] * dW[2] + u[2] * dW[3]) + g.hu2 * dW[0]);
  const T dmk = dW[1 + k];
  out[0] = dmk;
#pragma unroll
  for (int j = 0; j < 3; ++j) out[1 + j] = dmk * u[j] + u[k] * e[j];
  out[1 + k] += dp;
  out[4] = e[k] * g.rH + u[k] * (dW[4] + dp);
}

// directional derivatives along (n, t1, t2) of the frame-rotated conservative variables
template <typename T>
HD void rotate_gradient(const T Gq[15], const T* e[3], T D[3][5]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const T* dir = e[k];
    T gs[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) gs[q] = Gq[3 * q] * dir[0] + Gq[3 * q + 1] * dir[1] + Gq[3 * q + 2] * dir[2];
    D[k][0] = gs[0];
    D[k][4] = gs[4];
#pragma unroll
    for (int j = 0; j < 3; ++j) D[k][1 + j] = e[j][0] * gs[1] + e[j][1] * gs[2] + e[j][2] * gs[3];
  }
}

// ---- moments in the frame moving with the tangential velocity --------------------------------
// With c = v - V, d = w - W (full-space Gaussians of variance h), psi = T psi' where
// psi' = (1, u, c, d, (u^2 + c^2 + d^2 + xi^2)/2) and T adds V, W, (V^2 + W^2)/2 terms.  Odd moments of
// c and d vanish, so the matrices <u^k psi' psi'^T>, <u^k c psi' psi'^T>, <u^k d psi' psi'^T> are sparse;
// a slope s becomes s' = T^T s and a moment vector o' becomes T o'.
template <typename T>
struct MomP {
  T M[7];            // rho <u^k>, k = 0..6 (half or full space)
  T h, sig, tau4;    // h = p/rho, sig = h + <xi^2>/2, tau4 = 2 h^2 + h <xi^2> + <xi^4>/4
  T hs;              // h (2 h + <xi^2>/2)
  T V, W, E;         // tangential velocity and (V^2 + W^2)/2
  // the matrix entries the products below share, formed once per moment set: P_k = M_{k+2}/2 +
  // sig M_k (<u^k psi'_0 psi'_4>; <u^k psi'_1 psi'_4> is P_{k+1}), R_k = M_{k+4}/4 + sig M_{k+2} +
  // tau4 M_k (<u^k psi'_4 psi'_4>), h M_k, and S_k = h M_{k+2}/2 + hs M_k (<u^k c psi'_2 psi'_4>)
  T Pm[4], Rm[3], hM[4], S4[2];
};

template <typename T>
HD void make_momp(const Maxw<T>& g, T m0, T m1, T K, MomP<T>& P) {
  T* M = P.M;
  const T h = g.h;
  M[0] = g.rho * m0;
  M[1] = g.rho * m1;
#pragma unroll
  for (int n = 0; n + 2 < 7; ++n) M[n + 2] = g.U * M[n + 1] + T(n + 1) * h * M[n];
  const T x2 = K * h, x4 = K * (K + 2.0) * h * h;
  P.h = h;
  P.sig = h + 0.5 * x2;
  P.tau4 = 2.0 * h * h + h * x2 + 0.25 * x4;
  P.hs = h * (2.0 * h + 0.5 * x2);
  P.V = g.V;
  P.W = g.W;
  P.E = 0.5 * (g.V * g.V + g.W * g.W);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    P.Pm[k] = 0.5 * M[k + 2] + P.sig * M[k];
    P.hM[k] = h * M[k];
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) P.Rm[k] = 0.25 * M[k + 4] + P.sig * M[k + 2] + P.tau4 * M[k];
#pragma unroll
  for (int k = 0; k < 2; ++k) P.S4[k] = 0.5 * P.hM[k + 2] + P.hs * M[k];
}

// s' = T^T s
template <typename T>
HD void to_primed(const MomP<T>& P, const T s[5], T sp[5]) {
  sp[0] = s[0] + P.V * s[2] + P.W * s[3] + P.E * s[4];
  sp[1] = s[1];
  sp[2] = s[2] + P.V * s[4];
  sp[3] = s[3] + P.W * s[4];
  sp[4] = s[4];
}

// out += T o' (the energy row added term by term, one fused multiply-add each)
template <typename T>
HD void add_from_primed(const MomP<T>& P, const T o[5], T out[5]) {
  out[0] += o[0];
  out[1] += o[1];
  out[2] += P.V * o[0] + o[2];
  out[3] += P.W * o[0] + o[3];
  out[4] += P.E * o[0];
  out[4] += P.V * o[2];
  out[4] += P.W * o[3];
  out[4] += o[4];
}

// out = T o'
template <typename T>
HD void from_primed(const MomP<T>& P, const T o[5], T out[5]) {
  out[0] = o[0];
  out[1] = o[1];
  out[2] = P.V * o[0] + o[2];
  out[3] = P.W * o[0] + o[3];
  out[4] = P.E * o[0] + P.V * o[2] + P.W * o[3] + o[4];
}

// o' = <u^k (s' . psi') psi'>
template <typename T, int k>
HD void papp(const MomP<T>& P, const T s[5], T o[5]) {
  const T* M = P.M;
  const T Pk = P.Pm[k], Qk = P.Pm[k + 1], Rk = P.Rm[k], hM = P.hM[k];
  o[0] = M[k] * s[0] + M[k + 1] * s[1] + Pk * s[4];
  o[1] = M[k + 1] * s[0] + M[k + 2] * s[1] + Qk * s[4];
  o[2] = hM * s[2];
  o[3] = hM * s[3];
  o[4] = Pk * s[0] + Qk * s[1] + Rk * s[4];
}

// o' += <u^k c (s' . psi') psi'> (J = 2) or <u^k d (s' . psi') psi'> (J = 3)
template <typename T, int k, int J>
HD void papp_t_add(const MomP<T>& P, const T s[5], T o[5]) {
  const T hM0 = P.hM[k], hM1 = P.hM[k + 1], S4 = P.S4[k];
  o[0] += hM0 * s[J];
  o[1] += hM1 * s[J];
  o[J] += hM0 * s[0];
  o[J] += hM1 * s[1];
  o[J] += S4 * s[4];
  o[4] += S4 * s[J];
}

// o' = <u^k (a . u) psi'> with the three slopes in primed form: u a_n + v a_t1 + w a_t2,
// v = V + c, w = W + d
template <typename T, int k>
HD void papp_au(const MomP<T>& P, const T an[5], const T a1[5], const T a2[5], T o[5]) {
  T comb[5], t[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) comb[q] = P.V * a1[q] + P.W * a2[q];
  papp<T, k + 1>(P, an, o);
  papp<T, k>(P, comb, t);
#pragma unroll
  for (int q = 0; q < 5; ++q) o[q] += t[q];
  papp_t_add<T, k, 2>(P, a1, o);
  papp_t_add<T, k, 3>(P, a2, o);
}

// one side of the interface: micro-slopes of the initial distribution, its contribution to the
// equilibrium slopes, the time-integrated flux, the state at dt and the time-integrated state
template <typename T>
HD void side_terms(const T D[3][5], const Maxw<T>& g, T m0, T m1, T K, T gm1, T tau, T q4, T q5, T edt, T dtf, T dWc[3][5],
                   T Facc[5], T Wacc[5], T Iacc[5]) {
  MomP<T> P;
  make_momp<T>(g, m0, m1, K, P);
  T a[3][5];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T s[5];
    slope_solve<T>(g, D[k], s);
    to_primed<T>(P, s, a[k]);
  }
  // time slope A from <A + a.u> = 0 under the full Maxwellian: <(a.u) psi> = sum_k J_k dW_k
  T Ap[5];
  {
    T t0[5], t1[5], t2[5], au[5], A[5];
    euler_jvp<T>(g, gm1, 0, D[0], t0);
    euler_jvp<T>(g, gm1, 1, D[1], t1);
    euler_jvp<T>(g, gm1, 2, D[2], t2);
#pragma unroll
    for (int q = 0; q < 5; ++q) au[q] = -(t0[q] + t1[q] + t2[q]);
    slope_solve<T>(g, au, A);
    to_primed<T>(P, A, Ap);
  }
  // half-space moments: equilibrium-slope contributions <a_k psi>
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T t[5];
    papp<T, 0>(P, a[k], t);
    add_from_primed<T>(P, t, dWc[k]);
  }
  // <(a.u) psi>, <u (a.u) psi>, <A psi>, <u A psi>, <psi>, <u psi>
  T Va[5], Fa[5], VA[5], FA[5];
  papp_au<T, 0>(P, a[0], a[1], a[2], Va);
  papp_au<T, 1>(P, a[0], a[1], a[2], Fa);
  papp<T, 0>(P, Ap, VA);
  papp<T, 1>(P, Ap, FA);
  const T* M = P.M;
  const T V0[5] = {M[0], M[1], 0.0, 0.0, 0.5 * M[2] + P.sig * M[0]};
  const T F0[5] = {M[1], M[2], 0.0, 0.0, 0.5 * M[3] + P.sig * M[1]};
  const T tq4 = tau * q4;
  const T etd = edt * (tau + dtf), etau = edt * tau;
  T f[5], s[5], i[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    f[q] = q4 * F0[q] - q5 * Fa[q] - tq4 * FA[q];
    s[q] = edt * V0[q] - etd * Va[q] - etau * VA[q];
    i[q] = q4 * V0[q] - q5 * Va[q] - tq4 * VA[q];
  }
  add_from_primed<T>(P, f, Facc);
  add_from_primed<T>(P, s, Wacc);
  add_from_primed<T>(P, i, Iacc);
}

// the gas-kinetic flux of one Gauss point (flux x weight / dt and interface state x area, both in
// the global frame) and its compression factor, from the point's left and right states and
// gradients; on a boundary face (bnd) the right side is the ghost of the left
template <typename T>
HD void point_flux(const double nd[3], double iw, bool bnd, int tag, const T WLg[5], const T GLg[15], const T WRi[5],
                   const T GRi[15], T dtf, const Phys& ph, T Fg[5], T Wg[5], T& alpha, DevErr* err, int64_t f) {
  T n[3], t1[3], t2[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) n[d] = nd[d];
  face_frame<T>(n, t1, t2);
  const T* e[3] = {n, t1, t2};
  const T K = ph.K, gm1 = ph.gamma - 1.0, iK3 = 1.0 / (ph.K + 3.0);
  T WRg[5], GRg[15];
  if (!bnd) {
#pragma unroll
    for (int q = 0; q < 5; ++q) WRg[q] = WRi[q];
#pragma unroll
    for (int j = 0; j < 15; ++j) GRg[j] = GRi[j];
  } else if (!bc_ghost<T>(tag, n, WLg, GLg, WRg, GRg, T(ph.gamma), ph.Winf)) {
    set_err(err, CGKS_ENAN, (int)f, 3);
  }
  T wl[5], wr[5];
  rotate_in<T>(WLg, n, t1, t2, wl);
  rotate_in<T>(WRg, n, t1, t2, wr);
  Maxw<T> gl, gr;
  const bool okl = make_maxw<T>(wl, gm1, K, iK3, gl), okr = make_maxw<T>(wr, gm1, K, iK3, gr);
  if (!(okl && okr)) set_err(err, CGKS_ENAN, (int)f, 4);
  // half-space seeds of both sides, and the interface equilibrium
  // W^c = int_{u>0} psi g^l + int_{u<0} psi g^r (Eq. compatibility2)
  T ml0, ml1, mr0, mr1;
  half_seeds<T>(gl, 1.0, ml0, ml1);
  half_seeds<T>(gr, -1.0, mr0, mr1);
  T wc[5];
  {
    const T ml2 = gl.U * ml1 + gl.h * ml0, mr2 = gr.U * mr1 + gr.h * mr0;
    const T ql = gl.V * gl.V + gl.W * gl.W + (ph.K + 2.0) * gl.h;
    const T qr = gr.V * gr.V + gr.W * gr.W + (ph.K + 2.0) * gr.h;
    wc[0] = gl.rho * ml0 + gr.rho * mr0;
    wc[1] = gl.rho * ml1 + gr.rho * mr1;
    wc[2] = gl.rho * gl.V * ml0 + gr.rho * gr.V * mr0;
    wc[3] = gl.rho * gl.W * ml0 + gr.rho * gr.W * mr0;
    wc[4] = 0.5 * (gl.rho * (ml2 + ml0 * ql) + gr.rho * (mr2 + mr0 * qr));
  }
  Maxw<T> gc;
  if (!make_maxw<T>(wc, gm1, K, iK3, gc)) set_err(err, CGKS_ENAN, (int)f, 5);
  // collision times (Sec. 2.3)
  const T jump = fabs((gl.p - gr.p) / (gl.p + gr.p));
  T tau, tn;
  if (ph.viscous) {
    tau = viscosity<T>(ph, ph.gamma * gc.h) * (gc.r * gc.l2);  // mu(T^c) / p^c, p^c/rho^c = 1/(2 lambda^c)
    tn = tau + ph.c_press * jump * dtf;
  } else {
    tn = (ph.eps_inviscid + ph.c_press * jump) * dtf;
    tau = tn;
  }
  // exact integrals over [0, dt] of the time coefficients of Eq. 2nd-flux
  const T edt = exp(-dtf / tn), om = 1.0 - edt;
  const T q1 = dtf - tn * om;
  const T q2 = (tn * tn + tau * tn) * om - tn * dtf * edt - tau * dtf;
  const T q3 = 0.5 * dtf * dtf - tau * dtf + tau * tn * om;
  const T q4 = tn * om;
  const T q5 = (tau * tn + tn * tn) * om - tn * dtf * edt;
  // compression factor of this Gauss point (interior faces only), 1/p = l2 / rho
  alpha = 1.0;
  if (!bnd && ph.cf) {
    const T icl = rsqrt_hd(ph.gamma * gl.h), icr = rsqrt_hd(ph.gamma * gr.h);
    const T dp = fabs(gl.p - gr.p);
    const T dn = gl.U * icl - gr.U * icr, d1 = gl.V * icl - gr.V * icr, d2 = gl.W * icl - gr.W * icr;
    const T A = dp * (gl.r * gl.l2 + gr.r * gr.l2) + dn * dn + (d1 * d1 + d2 * d2);
    alpha = 1.0 / (1.0 + A * A);
  }
  T dWc[3][5], Facc[5], Wacc[5], Iacc[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    dWc[0][q] = dWc[1][q] = dWc[2][q] = 0.0;
    Facc[q] = Wacc[q] = Iacc[q] = 0.0;
  }
  {
    T D[3][5];
    rotate_gradient<T>(GLg, e, D);
    side_terms<T>(D, gl, ml0, ml1, K, gm1, tau, q4, q5, edt, dtf, dWc, Facc, Wacc, Iacc);
    rotate_gradient<T>(GRg, e, D);
    side_terms<T>(D, gr, mr0, mr1, K, gm1, tau, q4, q5, edt, dtf, dWc, Facc, Wacc, Iacc);
  }
  // equilibrium part: slopes a^c from the kinetic-weighted interface gradients; A^c from
  // <A + a.u> = 0; full-space moments through the Euler-flux Jacobians
  T ac[3][5];
#pragma unroll
  for (int k = 0; k < 3; ++k) slope_solve<T>(gc, dWc[k], ac[k]);
  T cu[5];  // <(a^c . u) psi>_c = sum_k J_k dW^c_k
  {
    T u0[5], u1[5], u2[5];
    euler_jvp<T>(gc, gm1, 0, dWc[0], u0);
    euler_jvp<T>(gc, gm1, 1, dWc[1], u1);
    euler_jvp<T>(gc, gm1, 2, dWc[2], u2);
#pragma unroll
    for (int q = 0; q < 5; ++q) cu[q] = u0[q] + u1[q] + u2[q];
  }
  T Fc0[5], FcA[5], Fca[5];
  {
    // <u psi>_c is the Euler flux of W^c; <u A^c psi>_c = J_n <A^c psi>_c = -J_n <(a^c . u) psi>_c
    Fc0[0] = wc[1];
    Fc0[1] = wc[1] * gc.U + gc.p;
    Fc0[2] = wc[2] * gc.U;
    Fc0[3] = wc[3] * gc.U;
    Fc0[4] = (wc[4] + gc.p) * gc.U;
    euler_jvp<T>(gc, gm1, 0, cu, FcA);
#pragma unroll
    for (int q = 0; q < 5; ++q) FcA[q] = -FcA[q];
    // <u (a^c . u) psi>_c in the frame moving with the tangential velocity
    MomP<T> P;
    make_momp<T>(gc, 1.0, gc.U, K, P);
    T a0[5], a1[5], a2[5], o[5];
    to_primed<T>(P, ac[0], a0);
    to_primed<T>(P, ac[1], a1);
    to_primed<T>(P, ac[2], a2);
    papp_au<T, 1>(P, a0, a1, a2, o);
    from_primed<T>(P, o, Fca);
  }
  const T q23 = q2 - q3;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    Facc[q] += q1 * Fc0[q];
    Facc[q] += q2 * Fca[q];
    Facc[q] += q3 * FcA[q];
    Wacc[q] += om * (wc[q] - dtf * cu[q]);
    Iacc[q] += q1 * wc[q];
    Iacc[q] += q23 * cu[q];
  }
  if (ph.viscous && ph.prandtl != 1.0) {
    // heat flux about U^c of the time-integrated distribution, scaled by (1/Pr - 1)
    const T Ub[3] = {gc.U, gc.V, gc.W};
    const T U2 = Ub[0] * Ub[0] + Ub[1] * Ub[1] + Ub[2] * Ub[2];
    const T qn = Facc[4] - (Ub[0] * Facc[1] + Ub[1] * Facc[2] + Ub[2] * Facc[3]) + 0.5 * U2 * Facc[0] -
                 Ub[0] * (Iacc[4] - (Ub[0] * Iacc[1] + Ub[1] * Iacc[2] + Ub[2] * Iacc[3]) + 0.5 * U2 * Iacc[0]);
    Facc[4] += (1.0 / ph.prandtl - 1.0) * qn;
  }
  const T sdt = 1.0 / (iw * dtf);  // weight / dt
#pragma unroll
  for (int q = 0; q < 5; ++q) Facc[q] *= sdt;
  rotate_out<T>(Facc, n, t1, t2, Fg);
  rotate_out<T>(Wacc, n, t1, t2, Wg);
}
