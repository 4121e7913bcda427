// Bodies of the fine-level CGKS kernels (Sec. 2-3 of the paper), FP64, written as host+device
// functions over argument structs; fine.cu wraps them in kernels.
//   reconstruct_body : per cell, HWENO p^2 (constrained least-squares operator), Green-Gauss p^1
//                      scaled by the compression factor, least-squares gradient, smoothness
//                      indicators, non-linear WENO weights -> 10 coefficients per variable; local dt
//   gks_point_body   : per face Gauss point, the time-dependent gas distribution of Eq. 2nd-flux:
//                      flux averaged over dt, interface state at dt (Sec. 2.4), compression factor
//                      alpha_{p,k} (Sec. 3.3)
//   gather_body      : per cell, fixed-order sums of the Gauss-point records -> residual,
//                      Gauss-Green gradient times the compression factor, optional explicit update
// The FP64 pipe bounds this path (FP64 runs at 1/62 of the FP32 rate on this GPU), so the code is
// written for few FP64 instructions; the flux itself is in flux.cuh.
#pragma once
#include <cstring>

#include "flux.cuh"
#include "internal.cuh"
#include "kinetic.cuh"

// sizes of the stored linearisation (the adjoint): inputs and outputs of one Gauss point; of one
// cell's reconstruction: its own slot dense (20 inputs (W, grad W) x 51 outputs, the coefficients and
// the time step), and per neighbour slot (up to 6) one block per variable q, 4 inputs (W_q and its
// gradient) x its 10 coefficients -- each variable is reconstructed on its own, so a neighbour's
// variable q reaches no other variable's coefficients (only the cell's own ghosts couple them)
#define CGKS_PJ_IN 41
#define CGKS_PJ_OUT 10
#define CGKS_RJ_OUT 51
#define CGKS_RJ_SELF (20 * CGKS_RJ_OUT)
#define CGKS_RJ_NB (5 * 4 * 10)
#define CGKS_RJ_ROWS (CGKS_RJ_SELF + 6 * CGKS_RJ_NB)

// dynamic viscosity at temperature ratio t = T/T_inf = gamma p/rho (free stream rho 1, p 1/gamma):
// constant, or Sutherland's law mu_inf t^(3/2) (1 + s)/(t + s)
template <typename T>
HD T viscosity(const Phys& ph, T t) {
  if (ph.suth == 0.0) return T(ph.mu);
  return ph.mu * t * sqrt(t) * (1.0 + ph.suth) / (t + ph.suth);
}

#ifndef CGKS_LIBRARY
#include "flux_generic.cuh"  // host tests
#endif

struct ReconArgs {
  int64_t nc, nf;
  const int8_t* ctype;
  const int32_t *cf, *fL, *fR, *ftag;
  const int8_t* cside;
  const double *fnrm, *Kop, *ggw, *lsw, *aux, *dtw, *vol, *W, *G, *alpha;
  double *rc, *dt;
  Phys ph;
  DevErr* err;
  const int32_t* nbr;  // [6][nc] cell across each local face, -1 on the boundary (null: from the faces)
};

// local time step of cell i from its average Q0: CFL |Omega| / sum_p S_p (|U.n_p| + c + 2 nu S_p / |Omega|)
template <typename T>
HD T time_step(int64_t i, const ReconArgs& a, const T Q0[5]) {
  const int64_t nc = a.nc;
  const int nt = a.ctype[i] == 7 ? 5 : a.ctype[i];
  const Phys& ph = a.ph;
  const T r = 1.0 / Q0[0];
  const T u[3] = {Q0[1] * r, Q0[2] * r, Q0[3] * r};
  const T p = (ph.gamma - 1.0) * (Q0[4] - 0.5 * Q0[0] * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]));
  const T c = sqrt(ph.gamma * p * r);
  const double V = a.vol[i];
  const T nu2 = ph.viscous ? 2.0 * viscosity<T>(ph, ph.gamma * p * r) * r / V : T(0.0);
  T s = 0.0;
  for (int m = 0; m < nt; ++m) {
    const double S = a.dtw[(4 * m + 3) * nc + i];
    const T un = fabs(u[0] * a.dtw[(4 * m) * nc + i] + u[1] * a.dtw[(4 * m + 1) * nc + i] +
                      u[2] * a.dtw[(4 * m + 2) * nc + i]);
    s += un + S * c + nu2 * S * S;
  }
  if (!(Q0[0] > 0.0) || !(p > 0.0) || !isfinite(Q0[4])) set_err(a.err, CGKS_ENAN, (int)i, 2);
  return ph.cfl_fine * V / s;
}

// stencil sums of one variable of cell i: the p^2 coefficients b, Green-Gauss and least-squares gradients;
// v[m] = (W_q, gradient of W_q) of slot m.  Each neighbour's difference and gradient are added into a
// coefficient on their own (one fused multiply-add per operator entry).  Green-Gauss from the differences:
// the outward S n / |Omega| of a closed cell sum to zero, so sum (Q_m + Q_0) w_m = sum (Q_m - Q_0) w_m,
// without the cancellation
HD void recon_sums(int64_t i, int nt, double Q0, const ReconArgs& a, const double v[6][4], double b[9], double gg[3],
                   double gl[3]) {
  const int64_t nc = a.nc;
#pragma unroll
  for (int j = 0; j < 9; ++j) b[j] = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) gg[d] = gl[d] = 0.0;
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    if (m >= nt) continue;
    const double dQ = v[m][0] - Q0;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      b[j] += a.Kop[(j * 24 + m) * nc + i] * dQ;
      b[j] += a.Kop[(j * 24 + 6 + 3 * m) * nc + i] * v[m][1];
      b[j] += a.Kop[(j * 24 + 7 + 3 * m) * nc + i] * v[m][2];
      b[j] += a.Kop[(j * 24 + 8 + 3 * m) * nc + i] * v[m][3];
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      gg[d] += a.ggw[(3 * m + d) * nc + i] * dQ;
      gl[d] += a.lsw[(3 * m + d) * nc + i] * dQ;
    }
  }
}

// the non-linear combination of one variable (Sec. 3.4): b the p^2 coefficients of X,Y,Z,X^2,Y^2,Z^2,XY,
// YZ,XZ, p1 the compressed Green-Gauss gradient, gl the least-squares gradient -> its 10 coefficients.
// The indicator's first part, sum_d <(d_d p2)^2> = |b_0..2|^2 + tr(M H^2), takes the squared Hessian once
HD void weno_variable(double Q0, const double b[9], const double p1[3], const double gl[3], double V23, double V43,
                      const double M2[6], double eps, double out[10]) {
  const double a0 = Q0 - (b[3] * M2[0] + b[4] * M2[1] + b[5] * M2[2] + b[6] * M2[3] + b[7] * M2[4] + b[8] * M2[5]);
  const double bGG = V23 * (p1[0] * p1[0] + p1[1] * p1[1] + p1[2] * p1[2]);
  const double bLS = V23 * (gl[0] * gl[0] + gl[1] * gl[1] + gl[2] * gl[2]);
  const double beta1 = min_positive(bGG, bLS);
  const double s6 = b[6] * b[6], s7 = b[7] * b[7], s8 = b[8] * b[8];
  const double c6 = s6 + s8, c7 = s6 + s7, c8 = s7 + s8;
  const double hxx = 4.0 * b[3] * b[3] + c6, hyy = 4.0 * b[4] * b[4] + c7, hzz = 4.0 * b[5] * b[5] + c8;
  // twice the off-diagonal entries of the squared Hessian, half of each
  const double hxy = 2.0 * b[6] * (b[3] + b[4]) + b[8] * b[7];
  const double hyz = 2.0 * b[7] * (b[4] + b[5]) + b[6] * b[8];
  const double hxz = 2.0 * b[8] * (b[3] + b[5]) + b[6] * b[7];
  double off = M2[3] * hxy;
  off += M2[4] * hyz;
  off += M2[5] * hxz;
  double first = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
  first += M2[0] * hxx;
  first += M2[1] * hyy;
  first += M2[2] * hzz;
  first += 2.0 * off;
  // 4 (b_3^2 + b_4^2 + b_5^2) + b_6^2 + b_7^2 + b_8^2
  const double second = (hxx + hyy + hzz) - (c6 + s7);
  const double beta2 = V23 * first + V43 * second;
  const double rden = fast_rcp(Q0 * Q0 + beta1 + 1e-40);
  const double bt1 = beta1 * rden, bt2 = beta2 * rden;
  const double sig = bt2 - bt1;
  // w_m = g_m (1 + (sig/d_m)^2) with d_m = eps + beta~_m and g_1 = g_2 = 1/2, normalised with one
  // reciprocal: w_1 : w_2 = (d_1^2 + sig^2) d_2^2 : (d_2^2 + sig^2) d_1^2
  const double d1 = eps + bt1, d2 = eps + bt2;
  const double s2 = sig * sig, d11 = d1 * d1, d22 = d2 * d2;
  const double A1 = (d11 + s2) * d22, A2 = (d22 + s2) * d11;
  const double inv = fast_rcp(A1 + A2);
  const double w1 = A1 * inv, w2 = A2 * inv;
  const double c2 = 2.0 * w2, c1 = w1 - w2;
  out[0] = c2 * a0 + c1 * Q0;
#pragma unroll
  for (int d = 0; d < 3; ++d) out[1 + d] = c2 * b[d] + c1 * p1[d];
#pragma unroll
  for (int j = 3; j < 9; ++j) out[1 + j] = c2 * b[j];
}

// ghost average and gradient (W 5, grad W 15) of boundary slot m of cell i
HD void recon_ghost(int64_t i, int m, const ReconArgs& a, double Wg[5], double Gg[15]) {
  const int64_t nc = a.nc, nf = a.nf, f = a.cf[(int64_t)m * nc + i];
  double Q0[5], G0[15];
#pragma unroll
  for (int q = 0; q < 5; ++q) Q0[q] = a.W[q * nc + i];
#pragma unroll
  for (int j = 0; j < 15; ++j) G0[j] = a.G[j * nc + i];
  const double n[3] = {a.fnrm[f], a.fnrm[nf + f], a.fnrm[2 * nf + f]};
  if (!bc_ghost<double>(a.ftag[f], n, Q0, G0, Wg, Gg, a.ph.gamma, a.ph.Winf)) set_err(a.err, CGKS_ENAN, (int)i, 1);
}

// cell across local face m of cell i, -1 on the boundary
HD int32_t recon_neighbour(int64_t i, int m, const ReconArgs& a) {
  const int64_t k = (int64_t)m * a.nc + i;
  if (a.nbr) return a.nbr[k];
  const int64_t f = a.cf[k];
  return a.fR[f] < 0 ? -1 : (a.cside[k] ? a.fL[f] : a.fR[f]);
}

// reconstruction of variable q of cell i.  ghost(m, v) gives the boundary slot's (W_q, gradient of W_q)
template <typename Ghost>
HD void reconstruct_variable(int64_t i, int q, const ReconArgs& a, const Ghost& ghost, double out[10]) {
  const int64_t nc = a.nc;
  const int nt = a.ctype[i] == 7 ? 5 : a.ctype[i];  // faces: pyramids (type 7) have 5
  const double Q0 = a.W[q * nc + i];
  int32_t nb[6];
#pragma unroll
  for (int m = 0; m < 6; ++m) nb[m] = m < nt ? recon_neighbour(i, m, a) : 0;
  double v[6][4];
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    if (m >= nt) continue;
    if (nb[m] >= 0) {
      v[m][0] = a.W[q * nc + nb[m]];
#pragma unroll
      for (int d = 0; d < 3; ++d) v[m][1 + d] = a.G[(3 * q + d) * nc + nb[m]];
    } else {
      ghost(m, v[m]);
    }
  }
  double b[9], gg[3], gl[3];
  recon_sums(i, nt, Q0, a, v, b, gg, gl);
  double M2[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) M2[j] = a.aux[(2 + j) * nc + i];
  const double al = a.alpha[i];
  const double p1[3] = {al * gg[0], al * gg[1], al * gg[2]};
  weno_variable(Q0, b, p1, gl, a.aux[i], a.aux[nc + i], M2, a.ph.weno_eps, out);
}

HD void reconstruct_body(int64_t i, const ReconArgs& a) {
  const auto ghost_of = [&](int q) {
    return [&a, i, q](int m, double v[4]) {
      double Wg[5], Gg[15];
      recon_ghost(i, m, a, Wg, Gg);
      v[0] = Wg[q];
      for (int d = 0; d < 3; ++d) v[1 + d] = Gg[3 * q + d];
    };
  };
  for (int q = 0; q < 5; ++q) reconstruct_variable(i, q, a, ghost_of(q), a.rc + (int64_t)CGKS_RC * i + 10 * q);
  double Q0[5];
  for (int q = 0; q < 5; ++q) Q0[q] = a.W[q * a.nc + i];
  a.dt[i] = time_step<double>(i, a, Q0);
}

// the non-linear combination of one variable at its stencil sums, and its linearisation.  The outputs are
// (c2 a0 + c1 Q0, c2 b_d + c1 p1_d, c2 b_j) with c1 = 1 - c2 (the weights add up to one), so all of the
// nonlinearity is the derivative of c2 = 2 w_2: gb, gp, gl, gQ with respect to b, p1, the least-squares
// gradient and Q0, by reverse mode (the minimum in beta_1 takes the smaller branch, half of each at a tie)
struct WenoLin {
  double c2, c1, a0, p1[3], gb[9], gp[3], gl[3], gQ;
};

HD void weno_linear(double Q0, const double b[9], const double gg[3], const double gl[3], double al, double V23, double V43,
                    const double M2[6], double eps, WenoLin& w) {
  w.a0 = Q0 - (b[3] * M2[0] + b[4] * M2[1] + b[5] * M2[2] + b[6] * M2[3] + b[7] * M2[4] + b[8] * M2[5]);
  for (int d = 0; d < 3; ++d) w.p1[d] = al * gg[d];
  const double bGG = V23 * (w.p1[0] * w.p1[0] + w.p1[1] * w.p1[1] + w.p1[2] * w.p1[2]);
  const double bLS = V23 * (gl[0] * gl[0] + gl[1] * gl[1] + gl[2] * gl[2]);
  const double beta1 = fmin(bGG, bLS);
  const double vv[3][3] = {{2.0 * b[3], b[6], b[8]}, {b[6], 2.0 * b[4], b[7]}, {b[8], b[7], 2.0 * b[5]}};
  double first = 0.0, vb[3][3];
  for (int d = 0; d < 3; ++d) {
    const double* x = vv[d];
    const double Mx[3] = {M2[0] * x[0] + M2[3] * x[1] + M2[5] * x[2], M2[3] * x[0] + M2[1] * x[1] + M2[4] * x[2],
                          M2[5] * x[0] + M2[4] * x[1] + M2[2] * x[2]};
    first += b[d] * b[d] + x[0] * Mx[0] + x[1] * Mx[1] + x[2] * Mx[2];
    for (int e = 0; e < 3; ++e) vb[d][e] = 2.0 * Mx[e];
  }
  const double second = 4.0 * (b[3] * b[3] + b[4] * b[4] + b[5] * b[5]) + b[6] * b[6] + b[7] * b[7] + b[8] * b[8];
  const double beta2 = V23 * first + V43 * second;
  const double rden = 1.0 / (Q0 * Q0 + beta1 + 1e-40);
  const double bt1 = beta1 * rden, bt2 = beta2 * rden, dif = bt2 - bt1;
  const double d1 = eps + bt1, d2 = eps + bt2;
  const double s2 = dif * dif, d11 = d1 * d1, d22 = d2 * d2;
  const double A1 = (d11 + s2) * d22, A2 = (d22 + s2) * d11;
  const double inv = 1.0 / (A1 + A2);
  const double w1 = A1 * inv, w2 = A2 * inv;
  w.c2 = 2.0 * w2;
  w.c1 = w1 - w2;
  // d c2 = 2 d w2 = 2 inv (w1 dA2 - w2 dA1)
  const double A1b = -2.0 * inv * w2, A2b = 2.0 * inv * w1;
  const double d11b = A1b * d22 + A2b * (d22 + s2), d22b = A1b * (d11 + s2) + A2b * d11;
  const double s2b = A1b * d22 + A2b * d11;
  const double bt1b = 2.0 * d1 * d11b - 2.0 * dif * s2b, bt2b = 2.0 * d2 * d22b + 2.0 * dif * s2b;
  const double rdenb = bt1b * beta1 + bt2b * beta2, dr = -rden * rden * rdenb;
  w.gQ = 2.0 * Q0 * dr;
  const double beta1b = bt1b * rden + dr, beta2b = bt2b * rden;
  const double f1 = V23 * beta2b, f2 = V43 * beta2b;
  for (int d = 0; d < 3; ++d) w.gb[d] = 2.0 * b[d] * f1;
  for (int d = 0; d < 3; ++d) w.gb[3 + d] = 2.0 * vb[d][d] * f1 + 8.0 * b[3 + d] * f2;
  w.gb[6] = (vb[0][1] + vb[1][0]) * f1 + 2.0 * b[6] * f2;
  w.gb[7] = (vb[1][2] + vb[2][1]) * f1 + 2.0 * b[7] * f2;
  w.gb[8] = (vb[0][2] + vb[2][0]) * f1 + 2.0 * b[8] * f2;
  const double share = bGG < bLS ? 1.0 : (bGG > bLS ? 0.0 : 0.5);
  for (int d = 0; d < 3; ++d) {
    w.gp[d] = 2.0 * V23 * w.p1[d] * (share * beta1b);
    w.gl[d] = 2.0 * V23 * gl[d] * ((1.0 - share) * beta1b);
  }
}

// derivatives of a variable's 10 coefficients along a change (db, dgg, dgl, dQ0) of its sums
HD void weno_column(const WenoLin& w, const double b[9], double Q0, double al, const double M2[6], const double db[9],
                    const double dgg[3], const double dgl[3], double dQ0, double out[10]) {
  double dc = w.gQ * dQ0, da0 = dQ0;
#pragma unroll
  for (int j = 0; j < 9; ++j) dc += w.gb[j] * db[j];
#pragma unroll
  for (int j = 0; j < 6; ++j) da0 -= db[3 + j] * M2[j];
  double dp[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    dp[d] = al * dgg[d];
    dc += w.gp[d] * dp[d];
    dc += w.gl[d] * dgl[d];
  }
  out[0] = w.c2 * da0 + w.c1 * dQ0 + dc * (w.a0 - Q0);
#pragma unroll
  for (int d = 0; d < 3; ++d) out[1 + d] = w.c2 * db[d] + w.c1 * dp[d] + dc * (b[d] - w.p1[d]);
#pragma unroll
  for (int j = 3; j < 9; ++j) out[1 + j] = w.c2 * db[j] + dc * b[j];
}

HD bool ghost_mixes(int tag) { return tag <= 3; }  // boundary kinds 1 and 2 (walls), 3 (farfield)

// linearisation of variable q (0..4) of cell i, or of its time step (5), into Jr [CGKS_RJ_ROWS][nc]: rows
// 51 c + o of the own slot (input c of (W, grad W), output o of (50 coefficients, time step)), then
// for neighbour slot s = 1..6 the rows CGKS_RJ_SELF + ((s - 1) 5 + q) 40 + 10 c4 + j: input c4 of
// (W_q, d/dx, d/dy, d/dz of W_q), output coefficient j of variable q.  Only the rows that can differ
// from zero are written (the array starts at zero and which these are is the mesh's): absent slots and
// boundary faces have no neighbour rows; of the own slot a variable has the rows of its own average, of
// its own gradient next to a boundary face, and of all 20 inputs where the ghost mixes the variables
// (walls and farfield).
// Each stencil input is a column of the cell's linear maps (weno_column), so the whole takes about 4,500
// FP64 operations per cell; evaluating the reconstruction on dual numbers once per input took 140 times
// the reconstruction
HD void recon_jacobian_variable(int64_t i, int q, const ReconArgs& a, double* Jr) {
  const int64_t nc = a.nc, nf = a.nf;
  const int nt = a.ctype[i] == 7 ? 5 : a.ctype[i];
  if (q == 5) {
    for (int k = 0; k < 5; ++k) {
      DualD Q[5];
      for (int c = 0; c < 5; ++c) Q[c] = DualD(a.W[c * nc + i], c == k ? 1.0 : 0.0);
      Jr[(int64_t)(CGKS_RJ_OUT * k + CGKS_RC) * nc + i] = time_step<DualD>(i, a, Q).d;
    }
    return;
  }
  const double Q0 = a.W[q * nc + i];
  double v[6][4];
  unsigned bnd = 0;
  bool mixed = false;
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    if (m >= nt) continue;
    const int32_t nb = recon_neighbour(i, m, a);
    if (nb >= 0) {
      v[m][0] = a.W[q * nc + nb];
#pragma unroll
      for (int d = 0; d < 3; ++d) v[m][1 + d] = a.G[(3 * q + d) * nc + nb];
    } else {
      bnd |= 1u << m;
      mixed = mixed || ghost_mixes(a.ftag[a.cf[(int64_t)m * nc + i]]);
      double Wg[5], Gg[15];
      recon_ghost(i, m, a, Wg, Gg);
#pragma unroll
      for (int c = 0; c < 5; ++c)
        if (c == q) {
          v[m][0] = Wg[c];
#pragma unroll
          for (int d = 0; d < 3; ++d) v[m][1 + d] = Gg[3 * c + d];
        }
    }
  }
  double b[9], gg[3], gl[3], M2[6];
  recon_sums(i, nt, Q0, a, v, b, gg, gl);
#pragma unroll
  for (int j = 0; j < 6; ++j) M2[j] = a.aux[(2 + j) * nc + i];
  const double al = a.alpha[i];
  WenoLin w;
  weno_linear(Q0, b, gg, gl, al, a.aux[i], a.aux[nc + i], M2, a.ph.weno_eps, w);
  const double zero[3] = {0.0, 0.0, 0.0};
  double sb[9], sg[3], sl[3];  // minus the sums of the value columns: the change with Q0
#pragma unroll
  for (int j = 0; j < 9; ++j) sb[j] = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) sg[d] = sl[d] = 0.0;
  for (int m = 0; m < nt; ++m) {
    double db[9], dg[3], dl[3], out[10];
#pragma unroll
    for (int j = 0; j < 9; ++j) sb[j] -= db[j] = a.Kop[(j * 24 + m) * nc + i];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      sg[d] -= dg[d] = a.ggw[(3 * m + d) * nc + i];
      sl[d] -= dl[d] = a.lsw[(3 * m + d) * nc + i];
    }
    if (bnd >> m & 1) continue;
    const int64_t row = CGKS_RJ_SELF + (m * 5 + q) * 40;
    weno_column(w, b, Q0, al, M2, db, dg, dl, 0.0, out);
#pragma unroll
    for (int j = 0; j < 10; ++j) Jr[(row + j) * nc + i] = out[j];
    for (int e = 0; e < 3; ++e) {
#pragma unroll
      for (int j = 0; j < 9; ++j) db[j] = a.Kop[(j * 24 + 6 + 3 * m + e) * nc + i];
      weno_column(w, b, Q0, al, M2, db, zero, zero, 0.0, out);
#pragma unroll
      for (int j = 0; j < 10; ++j) Jr[(row + 10 * (1 + e) + j) * nc + i] = out[j];
    }
  }
  for (int c = 0; c < 20; ++c) {
    if (c != q && !mixed && !(bnd && c >= 5 && (c - 5) / 3 == q)) continue;
    double db[9], dg[3], dl[3], out[10];
    const double own = c == q ? 1.0 : 0.0;
#pragma unroll
    for (int j = 0; j < 9; ++j) db[j] = own * sb[j];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      dg[d] = own * sg[d];
      dl[d] = own * sl[d];
    }
    for (int m = 0; m < nt; ++m) {
      if (!(bnd >> m & 1)) continue;
      const int64_t f = a.cf[(int64_t)m * nc + i];
      const DualD n[3] = {DualD(a.fnrm[f]), DualD(a.fnrm[nf + f]), DualD(a.fnrm[2 * nf + f])};
      DualD Wd[5], Gd[15], Wg[5], Gg[15];
      for (int k = 0; k < 5; ++k) Wd[k] = DualD(a.W[k * nc + i], c == k ? 1.0 : 0.0);
      for (int k = 0; k < 15; ++k) Gd[k] = DualD(a.G[k * nc + i], c == 5 + k ? 1.0 : 0.0);
      bc_ghost<DualD>(a.ftag[f], n, Wd, Gd, Wg, Gg, DualD(a.ph.gamma), a.ph.Winf);
      double x = 0.0, y[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int k = 0; k < 5; ++k)
        if (k == q) {
          x = Wg[k].d;
#pragma unroll
          for (int d = 0; d < 3; ++d) y[d] = Gg[3 * k + d].d;
        }
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        db[j] += a.Kop[(j * 24 + m) * nc + i] * x;
#pragma unroll
        for (int d = 0; d < 3; ++d) db[j] += a.Kop[(j * 24 + 6 + 3 * m + d) * nc + i] * y[d];
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        dg[d] += a.ggw[(3 * m + d) * nc + i] * x;
        dl[d] += a.lsw[(3 * m + d) * nc + i] * x;
      }
    }
    weno_column(w, b, Q0, al, M2, db, dg, dl, own, out);
#pragma unroll
    for (int j = 0; j < 10; ++j) Jr[(int64_t)(CGKS_RJ_OUT * c + 10 * q + j) * nc + i] = out[j];
  }
}

HD void recon_jacobian_body(int64_t i, const ReconArgs& a, double* Jr) {
  for (int q = 0; q < 6; ++q) recon_jacobian_variable(i, q, a, Jr);
}

// ---- gas-kinetic point flux -------------------------------------------------------------------

// gradient (global frame) of a reconstruction polynomial at offset X from its centroid
HD void eval_gradient(const double* rcp, const double X[3], double Gq[15]) {
  const double X2[3] = {2.0 * X[0], 2.0 * X[1], 2.0 * X[2]};
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const double2* c2 = reinterpret_cast<const double2*>(rcp + 10 * q);
    const double2 A = c2[0], B = c2[1], C = c2[2], D = c2[3], E = c2[4];
    // (r0 r1) (r2 r3) (r4 r5) (r6 r7) (r8 r9): 1 X Y Z X^2 Y^2 Z^2 XY YZ XZ
    Gq[3 * q + 0] = A.y + C.x * X2[0] + D.y * X[1] + E.y * X[2];
    Gq[3 * q + 1] = B.x + C.y * X2[1] + D.y * X[0] + E.x * X[2];
    Gq[3 * q + 2] = B.y + D.x * X2[2] + E.x * X[1] + E.y * X[0];
  }
}

HD void eval_value(const double* rcp, const double X[3], double Wv[5]) {
  const double xx = X[0] * X[0], yy = X[1] * X[1], zz = X[2] * X[2], xy = X[0] * X[1], yz = X[1] * X[2], xz = X[0] * X[2];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const double2* c2 = reinterpret_cast<const double2*>(rcp + 10 * q);
    const double2 A = c2[0], B = c2[1], C = c2[2], D = c2[3], E = c2[4];
    Wv[q] = A.x + A.y * X[0] + B.x * X[1] + B.y * X[2] + C.x * xx + C.y * yy + D.x * zz + D.y * xy + E.x * yz + E.y * xz;
  }
}

struct PointArgs {
  int64_t ngp, nf, nc;
  const int32_t *gp_face, *fL, *fR, *ftag;
  const double *gp_x, *gp_A, *fshift, *ctr, *rc, *dt;
  double* gpr;  // [ngp][CGKS_GPR] records: flux x weight / dt (5), interface state (5), area vector (3), alpha
  Phys ph;
  DevErr* err;
  const double* tab;  // table of half_gauss (device)
};

// inputs of one Gauss point: unit normal n, 1/|weight x area|, face, cells, the left and right
// states and gradients at the point (global frame) and the face's time step
struct PointIn {
  double n[3], iw;
  int64_t f, L, R;
  double WL[5], GL[15], WR[5], GR[15], dtf;
};

HD void point_inputs(int64_t g, const PointArgs& a, PointIn& p) {
  const int64_t ngp = a.ngp, nf = a.nf, nc = a.nc;
  const int64_t f = a.gp_face[g];
  const int64_t L = a.fL[f], R = a.fR[f];
  p.f = f;
  p.L = L;
  p.R = R;
  const double x[3] = {a.gp_x[g], a.gp_x[ngp + g], a.gp_x[2 * ngp + g]};
  const double Av[3] = {a.gp_A[g], a.gp_A[ngp + g], a.gp_A[2 * ngp + g]};
  p.iw = fast_rsqrt(Av[0] * Av[0] + Av[1] * Av[1] + Av[2] * Av[2]);
#pragma unroll
  for (int d = 0; d < 3; ++d) p.n[d] = Av[d] * p.iw;
  const double* rcL = a.rc + (int64_t)CGKS_RC * L;
  const double XL[3] = {x[0] - a.ctr[L], x[1] - a.ctr[nc + L], x[2] - a.ctr[2 * nc + L]};
  eval_value(rcL, XL, p.WL);
  eval_gradient(rcL, XL, p.GL);
  if (R >= 0) {
    const double* rcR = a.rc + (int64_t)CGKS_RC * R;
    double XR[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) XR[d] = x[d] - a.fshift[d * nf + f] - a.ctr[d * nc + R];
    eval_value(rcR, XR, p.WR);
    eval_gradient(rcR, XR, p.GR);
    p.dtf = fmin(a.dt[L], a.dt[R]);
  } else {
    p.dtf = a.dt[L];
  }
}

// value and gradient (global frame) of a reconstruction polynomial at offset X from its centroid: with
// t_d = c_d + (H X)_d / 2 (H the Hessian) the gradient is 2 t - c and the value c_0 + X.t
HD void eval_both(const double* rcp, const double X[3], double Wv[5], double Gq[15]) {
  const double hx = 0.5 * X[0], hy = 0.5 * X[1], hz = 0.5 * X[2];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const double2* c2 = reinterpret_cast<const double2*>(rcp + 10 * q);
    const double2 A = c2[0], B = c2[1], C = c2[2], D = c2[3], E = c2[4];
    // (A.x A.y) (B.x B.y) ...: 1 X Y Z X^2 Y^2 Z^2 XY YZ XZ
    const double tx = A.y + C.x * X[0] + D.y * hy + E.y * hz;
    const double ty = B.x + C.y * X[1] + D.y * hx + E.x * hz;
    const double tz = B.y + D.x * X[2] + E.x * hy + E.y * hx;
    Wv[q] = A.x + X[0] * tx + X[1] * ty + X[2] * tz;
    Gq[3 * q + 0] = 2.0 * tx - A.y;
    Gq[3 * q + 1] = 2.0 * ty - B.x;
    Gq[3 * q + 2] = 2.0 * tz - B.y;
  }
}

// one contiguous record per point, so that the gather reads a face's points as one segment; STATE
// false (the defect of the V-cycle): the flux alone, in the record's first five entries
template <bool STATE = true>
HD void gks_point_body(int64_t g, const PointArgs& a) {
  const int64_t ngp = a.ngp, nf = a.nf, nc = a.nc;
  const int64_t f = a.gp_face[g];
  const int64_t L = a.fL[f], R = a.fR[f];
  const int tag = a.ftag[f];
  const double x[3] = {a.gp_x[g], a.gp_x[ngp + g], a.gp_x[2 * ngp + g]};
  const double Av[3] = {a.gp_A[g], a.gp_A[ngp + g], a.gp_A[2 * ngp + g]};
  const double a2 = Av[0] * Av[0] + Av[1] * Av[1] + Av[2] * Av[2], iw = fast_rsqrt(a2);
  const double n[3] = {Av[0] * iw, Av[1] * iw, Av[2] * iw};
  double WL[5], GL[15], WR[5], GR[15], X[3], dtf = a.dt[L];
#pragma unroll
  for (int d = 0; d < 3; ++d) X[d] = x[d] - a.ctr[d * nc + L];
  eval_both(a.rc + (int64_t)CGKS_RC * L, X, WL, GL);
  if (R >= 0) {
#pragma unroll
    for (int d = 0; d < 3; ++d) X[d] = x[d] - a.ctr[d * nc + R];
    if (tag >= 0)  // a periodic face
#pragma unroll
      for (int d = 0; d < 3; ++d) X[d] -= a.fshift[d * nf + f];
    eval_both(a.rc + (int64_t)CGKS_RC * R, X, WR, GR);
    dtf = min_positive(dtf, a.dt[R]);
  } else if (!bc_ghost<double>(tag, n, WL, GL, WR, GR, a.ph.gamma, a.ph.Winf)) {
    set_err(a.err, CGKS_ENAN, (int)f, 3);
  }
  double Fg[5], Wg[5], alpha;
  const int bad = gks_flux<STATE>(n, a2 * iw, R < 0, WL, GL, WR, GR, dtf, a.ph, a.tab, Fg, Wg, alpha);
  if (bad) set_err(a.err, CGKS_ENAN, (int)f, bad);
  double2* dst = reinterpret_cast<double2*>(a.gpr + (int64_t)CGKS_GPR * g);
  dst[0] = make_double2(Fg[0], Fg[1]);
  dst[1] = make_double2(Fg[2], Fg[3]);
  if (!STATE) {
    a.gpr[(int64_t)CGKS_GPR * g + 4] = Fg[4];
    return;
  }
  dst[2] = make_double2(Fg[4], Wg[0]);
  dst[3] = make_double2(Wg[1], Wg[2]);
  dst[4] = make_double2(Wg[3], Wg[4]);
  dst[5] = make_double2(Av[0], Av[1]);
  dst[6] = make_double2(Av[2], alpha);
}

// linearisation of one Gauss point: Jp[(10 k + o) ngp + g] = d out_o / d in_k with inputs k = (W_L 5,
// grad W_L 15, W_R 5, grad W_R 15, dt_f) at the point and outputs o = (flux 5, interface state 5) as
// gks_point_body stores them; the right-side columns of a boundary point are zero (its ghost is a function
// of the left side).
// The flux is linear in the gradients, so their 30 columns are responses to gradients of rank one
// (gks_gradient_column, about 250 FP64 operations each); the ten columns of the states are dual evaluations
// of one side (a right column is a left one seen from the other side: F_n(L, R) = -F_-n(R, L)), about 3,000
// each; the time step's is a dual evaluation with passive states.  Evaluating all 41 on dual numbers took
// 246,000 FP64 operations per point
HD void point_jacobian_body(int64_t g, const PointArgs& a, double* Jp) {
  PointIn p;
  point_inputs(g, a, p);
  const bool bnd = p.R < 0;
  const int tag = a.ftag[p.f];
  const int64_t ngp = a.ngp;
  const Phys& ph = a.ph;
  const double weight = 1.0 / p.iw, sdt = weight * fast_rcp(p.dtf);
  const auto store = [&](int k, const double col[10], double sf, double sw) {
#pragma unroll
    for (int o = 0; o < 10; ++o) Jp[(int64_t)(10 * k + o) * ngp + g] = (o < 5 ? sf : sw) * col[o];
  };
  if (bnd && !bc_ghost<double>(tag, p.n, p.WL, p.GL, p.WR, p.GR, ph.gamma, ph.Winf)) set_err(a.err, CGKS_ENAN, (int)p.f, 3);
  const double nm[3] = {-p.n[0], -p.n[1], -p.n[2]};
  // states
  for (int k = 0; k < 10; ++k) {
    const bool right = k >= 5;
    const int q = right ? k - 5 : k;
    double col[10];
    DualD F[5], Wg[5], al, W[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) W[c] = DualD(right ? p.WR[c] : p.WL[c], c == q ? 1.0 : 0.0);
    if (right && bnd) {
#pragma unroll
      for (int o = 0; o < 10; ++o) col[o] = 0.0;
      store(20 + q, col, 1.0, 1.0);
      continue;
    }
    if (bnd) {
      DualD G[15], Wr[5], Gr[15];
      const DualD nd[3] = {DualD(p.n[0]), DualD(p.n[1]), DualD(p.n[2])};
#pragma unroll
      for (int j = 0; j < 15; ++j) G[j] = DualD(p.GL[j]);
      bc_ghost<DualD>(tag, nd, W, G, Wr, Gr, DualD(ph.gamma), ph.Winf);  // the ghost gradient is linear in G alone
      const int bad = gks_flux_t<true, DualD, DualD, DualD, DualD>(p.n, weight, true, W, p.GL, Wr, p.GR, DualD(p.dtf), ph,
                                                                   a.tab, F, Wg, al);
      if (bad) set_err(a.err, CGKS_ENAN, (int)p.f, bad);
    } else {
      const int bad = gks_flux_t<true, DualD, double, DualD, double>(right ? nm : p.n, weight, false, W, right ? p.GR : p.GL,
                                                                     right ? p.WL : p.WR, right ? p.GL : p.GR, p.dtf, ph,
                                                                     a.tab, F, Wg, al);
      if (bad) set_err(a.err, CGKS_ENAN, (int)p.f, bad);
    }
#pragma unroll
    for (int o = 0; o < 5; ++o) {
      col[o] = F[o].d;
      col[5 + o] = Wg[o].d;
    }
    store(right ? 20 + q : q, col, right ? -1.0 : 1.0, 1.0);
  }
  // time step
  {
    DualD WL[5], WR[5], F[5], Wg[5], al;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      WL[q] = DualD(p.WL[q]);
      WR[q] = DualD(p.WR[q]);
    }
    gks_flux_t<true, DualD, DualD, DualD, DualD>(p.n, weight, bnd, WL, p.GL, WR, p.GR, DualD(p.dtf, 1.0), ph, a.tab, F, Wg,
                                                 al);
    double col[10];
#pragma unroll
    for (int o = 0; o < 5; ++o) {
      col[o] = F[o].d;
      col[5 + o] = Wg[o].d;
    }
    store(40, col, 1.0, 1.0);
  }
  // gradients: unit e_q along the axis d; on a boundary the ghost's gradient is another of rank one
  GksSide<double> gl, gr;
  GksCentre<double> c;
  const double gm1 = ph.gamma - 1.0;
  gks_side<double>(p.WL, p.n, 1.0, gm1, a.tab, gl);
  gks_side<double>(p.WR, p.n, -1.0, gm1, a.tab, gr);
  gks_centre<double, double, double, double>(gl, gr, p.dtf, ph, a.tab, c);
  for (int j = 0; j < 15; ++j) {
    const int q = j / 3;
    double A[5], B[5], d[3], r[3], col[10], add[10];
#pragma unroll
    for (int k = 0; k < 5; ++k) A[k] = B[k] = k == q ? 1.0 : 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) r[k] = d[k] = k == j % 3 ? 1.0 : 0.0;
    gks_gradient_column(gl, c, A, d, p.n, sdt, ph, col);
    if (!bnd) {
      store(5 + j, col, 1.0, 1.0);
      gks_gradient_column(gr, c, A, d, p.n, sdt, ph, col);
      store(25 + j, col, 1.0, 1.0);
      continue;
    }
    if (tag == 1 || tag == 2 || tag == 5) {
      if (tag != 5) {
        const double dn = d[0] * p.n[0] + d[1] * p.n[1] + d[2] * p.n[2];
        const double an = A[1] * p.n[0] + A[2] * p.n[1] + A[3] * p.n[2];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          r[k] = d[k] - 2.0 * dn * p.n[k];
          B[1 + k] = tag == 1 ? A[1 + k] - 2.0 * an * p.n[k] : -A[1 + k];
        }
      }
      gks_gradient_column(gr, c, B, r, p.n, sdt, ph, add);
#pragma unroll
      for (int o = 0; o < 10; ++o) col[o] += add[o];
    }
    store(5 + j, col, 1.0, 1.0);
#pragma unroll
    for (int o = 0; o < 10; ++o) col[o] = 0.0;
    store(25 + j, col, 1.0, 1.0);
  }
}

struct GatherArgs {
  int64_t nc, ngp;
  const int8_t *ctype, *cside;
  const int32_t *cf, *gp_ptr;
  const double *gpr, *vol, *dt, *W_in;
  double *W_out, *res, *G_out, *alpha_out;
  int update;
  double gamma;
  DevErr* err;
};

// running sums of one cell: residual, Gauss-Green gradient sums, compression-factor product
struct GatherAcc {
  double r[5], gs[15], al;
};

HD void gather_init(GatherAcc& c) {
#pragma unroll
  for (int q = 0; q < 5; ++q) c.r[q] = 0.0;
#pragma unroll
  for (int j = 0; j < 15; ++j) c.gs[j] = 0.0;
  c.al = 1.0;
}

// x with its sign bit xor-ed with `mask` (0 or the sign bit): an exact change of sign done by an
// integer operation, so that it takes no FP64 issue slot (those bound the gather on GB300)
HD double xor_sign(double x, uint64_t mask) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(__double_as_longlong(x) ^ (long long)mask);
#else
  uint64_t u;
  memcpy(&u, &x, sizeof u);
  u ^= mask;
  memcpy(&x, &u, sizeof x);
  return x;
#endif
}

// adds the ng consecutive Gauss-point records `rec` of one face, seen from its left cell (right:
// false) or from its right cell (the flux and the area vector change sign), in ascending point order
template <bool GRAD = true>
HD void gather_face(const double* rec, int ng, bool right, GatherAcc& c) {
  const uint64_t m = right ? 0x8000000000000000ull : 0ull;
  for (int k = 0; k < ng; ++k) {
    const double* v = rec + (int64_t)CGKS_GPR * k;
    if (!GRAD) {  // the residual alone (the defect of the V-cycle)
#pragma unroll
      for (int q = 0; q < 5; ++q) c.r[q] -= xor_sign(v[q], m);
      continue;
    }
    const double A[3] = {xor_sign(v[10], m), xor_sign(v[11], m), xor_sign(v[12], m)};
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      c.r[q] -= xor_sign(v[q], m);
      const double wq = v[5 + q];
#pragma unroll
      for (int d = 0; d < 3; ++d) c.gs[3 * q + d] += wq * A[d];
    }
    c.al *= v[13];
  }
}

// the cell's outputs from its sums: residual, alpha x Gauss-Green gradient / |Omega|, alpha, and
// the optional explicit update W += dt/|Omega| Res
HD void gather_store(int64_t i, const GatherArgs& a, const GatherAcc& c) {
  const int64_t nc = a.nc;
  const double rv = 1.0 / a.vol[i];
  if (a.res)
#pragma unroll
    for (int q = 0; q < 5; ++q) a.res[q * nc + i] = c.r[q];
  if (a.G_out) {
    const double k = c.al * rv;
#pragma unroll
    for (int j = 0; j < 15; ++j) a.G_out[j * nc + i] = k * c.gs[j];
  }
  if (a.alpha_out) a.alpha_out[i] = c.al;
  if (a.update) {
    const double h = a.dt[i] * rv;
    double w[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      w[q] = a.W_in[q * nc + i] + h * c.r[q];
      a.W_out[q * nc + i] = w[q];
    }
    const double p = (a.gamma - 1.0) * (w[4] - 0.5 * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]) / w[0]);
    if (!(w[0] > 0.0) || !(p > 0.0) || !isfinite(p)) set_err(a.err, CGKS_ENAN, (int)i, 6);
  }
}

// the gather of cell i, one face after the other in local-face order (the reference order: the
// device kernel stages the same records through shared memory and sums them in the same order)
HD void gather_body(int64_t i, const GatherArgs& a) {
  const int64_t nc = a.nc;
  GatherAcc c;
  gather_init(c);
  const int nt = a.ctype[i] == 7 ? 5 : a.ctype[i];  // faces: pyramids (type 7) have 5
  for (int m = 0; m < nt; ++m) {
    const int64_t f = a.cf[(int64_t)m * nc + i];
    const int64_t g0 = a.gp_ptr[f];
    const double* rec = a.gpr + (int64_t)CGKS_GPR * g0;
    const int ng = (int)(a.gp_ptr[f + 1] - g0);
    const bool right = a.cside[(int64_t)m * nc + i] != 0;
    if (a.G_out || a.alpha_out || a.update)
      gather_face<true>(rec, ng, right, c);
    else
      gather_face<false>(rec, ng, right, c);
  }
  gather_store(i, a, c);
}
