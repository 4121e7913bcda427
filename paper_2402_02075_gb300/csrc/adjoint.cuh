// Bodies of the adjoint's transposed-product kernels, per Gauss point and per cell (host+device, so
// that their arithmetic can be exercised without a device); adjoint.cu wraps them in kernels.
#pragma once
#include "fine.cuh"

// point cotangents are one record per Gauss point (41 values padded to 42 doubles, 336 bytes: the
// per-cell kernel gathers its faces' points, so each reads 21 contiguous 16-byte pairs instead of 41
// scattered words); neighbour records are one 20-double record per face side
#define CGKS_PB 42

struct VjpArgs {
  int64_t nc, nf, ngp;
  const int8_t *ctype, *cside;
  const int32_t *cf, *fL, *fR, *gp_face, *gp_ptr;
  const double *gp_x, *gp_A, *fshift, *ctr, *vol, *dt, *Jp, *Jr;
  const double *rbar, *gbar;  // cotangents of Res [5][nc] and Gnew [15][nc]
  double *pbar, *self, *rec;  // [ngp][42] (41 used), [20][nc], [2 nf][20]
  double* cbuf;               // [51][nc]: cotangents of each cell's coefficients and time step
  double *out;                // [20][nc]: cotangents of (W, G)
  const int32_t* ftag;        // face tags (null: every boundary face counts as mixing)
};

// what the own inputs of cell i reach besides their own average's coefficients: 0 nothing (no boundary
// face), 1 their own variable's (ghosts are functions of the gradient too), 2 every variable's (a ghost
// that mixes them)
HD int vjp_cell_kind(int64_t i, const VjpArgs& a) {
  const int nt = a.ctype[i] == 7 ? 5 : a.ctype[i];
  int kind = 0;
  for (int m = 0; m < nt; ++m) {
    const int64_t f = a.cf[(int64_t)m * a.nc + i];
    if (a.fR[f] < 0) kind = !a.ftag || ghost_mixes(a.ftag[f]) ? 2 : (kind > 1 ? kind : 1);
    if (kind == 2) break;
  }
  return kind;
}

// per Gauss point: cotangents of (flux, interface state) from those of (Res, Gnew) of its two cells,
// times Jp^T -> cotangents of the point inputs
HD void vjp_point_body(int64_t g, const VjpArgs& a) {
  const int64_t ngp = a.ngp, nc = a.nc;
  const int64_t f = a.gp_face[g], L = a.fL[f], R = a.fR[f];
  const double A[3] = {a.gp_A[g], a.gp_A[ngp + g], a.gp_A[2 * ngp + g]};
  // the left cell takes -flux and +A x state / |Omega|; the right cell the opposite
  double ub[10];
  // (the FP64 pipe bounds this kernel: 410 multiply-adds per point, and 60 here instead of 75)
  const double rvL = fast_rcp(a.vol[L]), rvR = R >= 0 ? fast_rcp(a.vol[R]) : 0.0;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    double u = -a.rbar[q * nc + L];
    double s = rvL * (A[0] * a.gbar[(3 * q) * nc + L] + A[1] * a.gbar[(3 * q + 1) * nc + L] + A[2] * a.gbar[(3 * q + 2) * nc + L]);
    if (R >= 0) {
      u += a.rbar[q * nc + R];
      s -= rvR * (A[0] * a.gbar[(3 * q) * nc + R] + A[1] * a.gbar[(3 * q + 1) * nc + R] + A[2] * a.gbar[(3 * q + 2) * nc + R]);
    }
    ub[q] = u;
    ub[5 + q] = s;
  }
  for (int k = 0; k < CGKS_PJ_IN; ++k) {
    if (R < 0 && k >= 20 && k < 40) continue;  // no right side (and no reader of its cotangents)
    const double* J = a.Jp + (int64_t)(CGKS_PJ_OUT * k) * ngp + g;
    double s = 0.0;
#pragma unroll
    for (int o = 0; o < CGKS_PJ_OUT; ++o) s += J[(int64_t)o * ngp] * ub[o];
    a.pbar[(int64_t)g * CGKS_PB + k] = s;
  }
}

// phase 1, per cell: cotangents of its 50 coefficients and its time step from its faces' points (the
// transposed evaluation of the polynomial and its gradient) -> cbuf [51][nc]
HD void vjp_coef_body(int64_t i, const VjpArgs& a) {
  const int64_t nc = a.nc, nf = a.nf, ngp = a.ngp;
  const int nt = a.ctype[i] == 7 ? 5 : a.ctype[i];
  double cb[CGKS_RJ_OUT];
#pragma unroll
  for (int o = 0; o < CGKS_RJ_OUT; ++o) cb[o] = 0.0;
  for (int m = 0; m < nt; ++m) {
    const int64_t f = a.cf[(int64_t)m * nc + i];
    const int side = a.cside[(int64_t)m * nc + i];
    const int64_t L = a.fL[f], R = a.fR[f];
    const int base = side ? 20 : 0;
    // the face time step is the smaller of the two cells' (shared equally at a tie, as a central
    // difference of the minimum sees it)
    const double own = side ? a.dt[R] : a.dt[L], other = side ? a.dt[L] : a.dt[R];
    const double w_dt = R < 0 ? 1.0 : (own < other ? 1.0 : (own > other ? 0.0 : 0.5));
    for (int64_t g = a.gp_ptr[f]; g < a.gp_ptr[f + 1]; ++g) {
      double X[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) X[d] = a.gp_x[d * ngp + g] - (side ? a.fshift[d * nf + f] : 0.0) - a.ctr[d * nc + i];
      const double2* pb2 = reinterpret_cast<const double2*>(a.pbar + (int64_t)g * CGKS_PB + base);
      double pb[20];
#pragma unroll
      for (int k = 0; k < 10; ++k) {
        const double2 v = pb2[k];
        pb[2 * k] = v.x;
        pb[2 * k + 1] = v.y;
      }
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const double w = pb[q], gx = pb[5 + 3 * q], gy = pb[6 + 3 * q], gz = pb[7 + 3 * q];
        // basis 1, X, Y, Z, X^2, Y^2, Z^2, XY, YZ, XZ and its gradient, through w X + g (the FP64 pipe
        // bounds this kernel: 19 operations per variable instead of 31)
        double* c = cb + 10 * q;
        const double ax = w * X[0] + gx, ay = w * X[1] + gy, az = w * X[2] + gz;
        c[0] += w;
        c[1] += ax;
        c[2] += ay;
        c[3] += az;
        c[4] += X[0] * (ax + gx);
        c[5] += X[1] * (ay + gy);
        c[6] += X[2] * (az + gz);
        c[7] += X[1] * ax;
        c[7] += X[0] * gy;
        c[8] += X[2] * ay;
        c[8] += X[1] * gz;
        c[9] += X[2] * ax;
        c[9] += X[0] * gz;
      }
      cb[CGKS_RC] += w_dt * a.pbar[(int64_t)g * CGKS_PB + 40];
    }
  }
#pragma unroll
  for (int o = 0; o < CGKS_RJ_OUT; ++o) a.cbuf[(int64_t)o * nc + i] = cb[o];
}

// phase 2, per cell and row group g with the cell's 51 cotangents cb[o * cs]:
//   g < 20   own-slot input c = g: self[c][i] = sum_o Jr[51 c + o][i] cb[o]; over the rows that
//            can differ from zero (kind, vjp_cell_kind): all, its variable's 10 coefficients and the time
//            step, or for a gradient none
//   g >= 20  neighbour slot s = 1 + (g - 20) / 5, variable q = (g - 20) % 5: its 4 inputs (W_q and the
//            gradient of W_q) into the record of the slot's face for the cell across it (absent
//            slots and boundary faces write nothing)
HD void vjp_slot_body(int64_t i, int g, const VjpArgs& a, const double* cb, int cs, int kind) {
  const int64_t nc = a.nc;
  if (g < 20) {
    const double* J = a.Jr + (int64_t)(CGKS_RJ_OUT * g) * nc + i;
    double v = g < 5 ? J[(int64_t)CGKS_RC * nc] * cb[CGKS_RC * cs] : 0.0;
    if (kind == 2) {
#pragma unroll 10
      for (int o = 0; o < CGKS_RC; ++o) v += J[(int64_t)o * nc] * cb[o * cs];
    } else if (kind == 1 || g < 5) {
      const int o0 = 10 * (g < 5 ? g : (g - 5) / 3);
#pragma unroll
      for (int o = 0; o < 10; ++o) v += J[(int64_t)(o0 + o) * nc] * cb[(o0 + o) * cs];
    }
    a.self[(int64_t)g * nc + i] = v;
    return;
  }
  const int s = 1 + (g - 20) / 5, q = (g - 20) % 5;
  const int nt = a.ctype[i] == 7 ? 5 : a.ctype[i];
  if (s > nt) return;
  const int64_t f = a.cf[(int64_t)(s - 1) * nc + i];
  if (a.fR[f] < 0) return;
  const int side = a.cside[(int64_t)(s - 1) * nc + i];
  double* rec = a.rec + (2 * f + side) * 20;
#pragma unroll
  for (int c4 = 0; c4 < 4; ++c4) {
    const double* J = a.Jr + (int64_t)(CGKS_RJ_SELF + ((s - 1) * 5 + q) * 40 + 10 * c4) * nc + i;
    double v = 0.0;
#pragma unroll
    for (int j = 0; j < 10; ++j) v += J[(int64_t)j * nc] * cb[(10 * q + j) * cs];
    rec[c4 == 0 ? q : 5 + 3 * q + (c4 - 1)] = v;
  }
}

HD void vjp_slot_body(int64_t i, int g, const VjpArgs& a, const double* cb, int cs) {
  vjp_slot_body(i, g, a, cb, cs, vjp_cell_kind(i, a));
}

// per cell, the reconstruction's part of the transposed product recomputed from the state instead of
// read from the stored linearisation (adjoint_recompute 1).  cb (stride cs) holds the cotangents of
// the cell's 50 coefficients and of its time step; out: the cotangents of its own (W, grad W) ->
// self, and those of each interior neighbour's (W_q, grad W_q) -> the record of that face side.  Per
// variable the transposed linearisation of the WENO combination of Sec. 3.4 (weno_linear, at the same
// stencil sums as the stored one), then the linear maps of p^2 (Sec. 3.1), Green-Gauss and least squares;
// then the ghost states of boundary faces (a function of the cell's own W and grad W: their transposed
// Jacobian from forward-mode duals) and the local time step.
HD void vjp_recon_body(int64_t i, const ReconArgs& a, const VjpArgs& v, const double* cb, int64_t cs) {
  const int64_t nc = a.nc, nf = a.nf;
  const int nt = a.ctype[i] == 7 ? 5 : a.ctype[i];
  const Phys& ph = a.ph;
  double Q0[5], G0[15], self[20];
#pragma unroll
  for (int q = 0; q < 5; ++q) Q0[q] = a.W[q * nc + i];
#pragma unroll
  for (int j = 0; j < 15; ++j) G0[j] = a.G[j * nc + i];
#pragma unroll
  for (int c = 0; c < 20; ++c) self[c] = 0.0;
  // ghost states of boundary slots (primal) and their cotangents
  double gval[6][20], gcot[6][20];
  for (int m = 0; m < nt; ++m) {
    const int64_t f = a.cf[(int64_t)m * nc + i];
    for (int c = 0; c < 20; ++c) gcot[m][c] = 0.0;
    if (a.fR[f] < 0) {
      const double n[3] = {a.fnrm[f], a.fnrm[nf + f], a.fnrm[2 * nf + f]};
      bc_ghost<double>(a.ftag[f], n, Q0, G0, gval[m], gval[m] + 5, ph.gamma, ph.Winf);
    }
  }
  const double V23 = a.aux[i], V43 = a.aux[nc + i], al = a.alpha[i];
  double M2[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) M2[j] = a.aux[(2 + j) * nc + i];
  for (int q = 0; q < 5; ++q) {
    // stencil of variable q, its sums and the linearised combination
    double v4[6][4], b[9], gg[3], gl[3];
    for (int m = 0; m < nt; ++m) {
      const int32_t nb = recon_neighbour(i, m, a);
      v4[m][0] = nb >= 0 ? a.W[q * nc + nb] : gval[m][q];
      for (int e = 0; e < 3; ++e) v4[m][1 + e] = nb >= 0 ? a.G[(3 * q + e) * nc + nb] : gval[m][5 + 3 * q + e];
    }
    recon_sums(i, nt, Q0[q], a, v4, b, gg, gl);
    WenoLin w;
    weno_linear(Q0[q], b, gg, gl, al, V23, V43, M2, ph.weno_eps, w);
    // out[0] = c2 a0 + c1 Q0, out[1+d] = c2 b[d] + c1 p1[d] (d < 3), out[1+j] = c2 b[j] (j >= 3), c1 = 1 - c2
    double ob[10];
    for (int k = 0; k < 10; ++k) ob[k] = cb[(10 * q + k) * cs];
    double c2b = ob[0] * (w.a0 - Q0[q]);
    for (int d = 0; d < 3; ++d) c2b += ob[1 + d] * (b[d] - w.p1[d]);
    for (int j = 3; j < 9; ++j) c2b += ob[1 + j] * b[j];
    const double a0b = w.c2 * ob[0];
    double q0b = w.c1 * ob[0] + w.gQ * c2b + a0b, bb[9], glb[3], ggb[3];
    for (int j = 0; j < 9; ++j) bb[j] = w.c2 * ob[1 + j] + w.gb[j] * c2b;
    for (int j = 3; j < 9; ++j) bb[j] -= a0b * M2[j - 3];
    for (int d = 0; d < 3; ++d) {
      glb[d] = w.gl[d] * c2b;
      ggb[d] = al * (w.c1 * ob[1 + d] + w.gp[d] * c2b);
    }
    // the linear maps, slot by slot
    for (int m = 0; m < nt; ++m) {
      const int64_t f = a.cf[(int64_t)m * nc + i];
      double dQb = 0.0, Gnb[3] = {0, 0, 0};
      for (int j = 0; j < 9; ++j) {
        dQb += a.Kop[(j * 24 + m) * nc + i] * bb[j];
        for (int e = 0; e < 3; ++e) Gnb[e] += a.Kop[(j * 24 + 6 + 3 * m + e) * nc + i] * bb[j];
      }
      double ggsum = 0.0;
      for (int d = 0; d < 3; ++d) {
        dQb += a.lsw[(3 * m + d) * nc + i] * glb[d];
        ggsum += a.ggw[(3 * m + d) * nc + i] * ggb[d];
      }
      const double Qnb = dQb + ggsum;
      q0b -= Qnb;
      if (a.fR[f] >= 0) {
        double* rec = v.rec + (2 * f + a.cside[(int64_t)m * nc + i]) * 20;
        rec[q] = Qnb;
        for (int e = 0; e < 3; ++e) rec[5 + 3 * q + e] = Gnb[e];
      } else {
        gcot[m][q] += Qnb;
        for (int e = 0; e < 3; ++e) gcot[m][5 + 3 * q + e] += Gnb[e];
      }
    }
    self[q] += q0b;
  }
  // ghost states: their transposed Jacobian in the cell's own (W, grad W), one dual seed per input
  for (int m = 0; m < nt; ++m) {
    const int64_t f = a.cf[(int64_t)m * nc + i];
    if (a.fR[f] >= 0) continue;
    const DualD n[3] = {DualD(a.fnrm[f]), DualD(a.fnrm[nf + f]), DualD(a.fnrm[2 * nf + f])};
    for (int c = 0; c < 20; ++c) {
      DualD Wd[5], Gd[15], Wg[5], Gg[15];
      for (int q = 0; q < 5; ++q) Wd[q] = DualD(Q0[q], c == q ? 1.0 : 0.0);
      for (int j = 0; j < 15; ++j) Gd[j] = DualD(G0[j], c == 5 + j ? 1.0 : 0.0);
      bc_ghost<DualD>(a.ftag[f], n, Wd, Gd, Wg, Gg, DualD(ph.gamma), ph.Winf);
      double sacc = 0.0;
      for (int q = 0; q < 5; ++q) sacc += Wg[q].d * gcot[m][q];
      for (int j = 0; j < 15; ++j) sacc += Gg[j].d * gcot[m][5 + j];
      self[c] += sacc;
    }
  }
  // local time step
  const double dtb = cb[CGKS_RC * cs];
  for (int c = 0; c < 5; ++c) {
    DualD Qd[5];
    for (int q = 0; q < 5; ++q) Qd[q] = DualD(Q0[q], q == c ? 1.0 : 0.0);
    self[c] += time_step<DualD>(i, a, Qd).d * dtb;
  }
  for (int c = 0; c < 20; ++c) v.self[(int64_t)c * nc + i] = self[c];
}

// per cell: own part plus the records its neighbours wrote for it -> cotangents of its (W, G)
HD void vjp_cell_body(int64_t i, const VjpArgs& a) {
  const int64_t nc = a.nc;
  const int nt = a.ctype[i] == 7 ? 5 : a.ctype[i];
  double v[20];
#pragma unroll
  for (int c = 0; c < 20; ++c) v[c] = a.self[(int64_t)c * nc + i];
  for (int m = 0; m < nt; ++m) {
    const int64_t f = a.cf[(int64_t)m * nc + i];
    if (a.fR[f] < 0) continue;
    const int other = 1 - a.cside[(int64_t)m * nc + i];
    const double2* rec = reinterpret_cast<const double2*>(a.rec + (2 * f + other) * 20);
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      const double2 r = rec[k];
      v[2 * k] += r.x;
      v[2 * k + 1] += r.y;
    }
  }
#pragma unroll
  for (int c = 0; c < 20; ++c) a.out[(int64_t)c * nc + i] = v[c];
}
