// Per-cell precompute of the reconstruction operators (Sec. 3): the constrained least-squares p^2
// map, Green-Gauss and least-squares gradient weights, indicator constants and time-step weights,
// as host+device functions (mesh.cu runs them in a kernel; the host can run them on the same
// arrays).
#pragma once
#include "internal.cuh"

__host__ __device__ __forceinline__ int cell_nfaces(int t) { return t == 7 ? 5 : t; }

// ---- dense helpers of the reconstruction-operator precompute (per thread, column-major) --------
//
// The number of faces is a template parameter, so that every loop is unrolled and every index known: the
// matrices then live in registers and in spill slots that are read once or twice.  With run-time sizes
// all of them (5.5 KB per thread) were local memory read at every multiply-add: 17.0 ms for the
// 1.51 M cells of the 96x64x69 boundary layer against 12.0 now, the FP64 pipe 91 % busy.

// s / d from r = 1/d: the product and one correction by its residual (P. W. Markstein, IBM J. Res. Dev. 34,
// 1990), as accurate as a division (within an ulp) and 3 FP64 instructions against 9; the operators take
// about 190 quotients by 25 divisors per cell.
__host__ __device__ __forceinline__ double quotient(double s, double d, double r) {
  const double q = s * r;
  return fma(fma(-q, d, s), r, q);
}

// Householder QR of A (M x N, M >= N, column-major, leading dimension M): R in the upper triangle,
// reflector k stored in A[k+1:, k] with an implicit unit leading entry, scale in tau[k].
template <int M, int N>
__host__ __device__ __forceinline__ bool house_qr(double* A, double* tau) {
  bool ok = true;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    double* a = A + k * M;
    double s = 0.0;
#pragma unroll
    for (int i = k + 1; i < M; ++i) s += a[i] * a[i];
    const double x0 = a[k];
    const double nrm = sqrt(x0 * x0 + s);
    ok = ok && nrm != 0.0;
    const double beta = x0 >= 0.0 ? -nrm : nrm;
    const double v0 = x0 - beta, rv = 1.0 / v0;
#pragma unroll
    for (int i = k + 1; i < M; ++i) a[i] = quotient(a[i], v0, rv);
    tau[k] = (beta - x0) / beta;
    a[k] = beta;
#pragma unroll
    for (int j = k + 1; j < N; ++j) {
      double* b = A + j * M;
      double d = b[k];
#pragma unroll
      for (int i = k + 1; i < M; ++i) d += a[i] * b[i];
      d *= tau[k];
      b[k] -= d;
#pragma unroll
      for (int i = k + 1; i < M; ++i) b[i] -= d * a[i];
    }
  }
  return ok;
}

// y <- Q y (Q = H_0 H_1 ... H_{N-1}) or y <- Q^T y
template <int M, int N, bool TRANSPOSE>
__host__ __device__ __forceinline__ void house_apply(const double* A, const double* tau, double* y) {
#pragma unroll
  for (int kk = 0; kk < N; ++kk) {
    const int k = TRANSPOSE ? kk : N - 1 - kk;
    const double* a = A + k * M;
    double d = y[k];
#pragma unroll
    for (int i = k + 1; i < M; ++i) d += a[i] * y[i];
    d *= tau[k];
    y[k] -= d;
#pragma unroll
    for (int i = k + 1; i < M; ++i) y[i] -= d * a[i];
  }
}

// p^2 operator, Green-Gauss and least-squares weights, smoothness-indicator constants and
// time-step weights of every cell.  Stencil: the cell and its face neighbours; a boundary face
// contributes the mirror image of the cell in the face plane (ghost cell).
struct ROArgs {
  int64_t nc, nf;
  const int8_t* ctype;
  const int32_t* cf;
  const int8_t* cside;
  const int32_t *fL, *fR;
  const double *vol, *ctr, *m2, *Sn, *area, *fshift, *fctr, *fnrm;
  double *Kop, *ggw, *lsw, *aux, *dtw;
  DevErr* err;
};

template <int nt>
__host__ __device__ __forceinline__ void recon_ops_cell(int64_t i, const ROArgs& A_) {
  const int64_t nc = A_.nc, nf = A_.nf;
  const int32_t* cf = A_.cf;
  const int8_t* cside = A_.cside;
  const int32_t *fL = A_.fL, *fR = A_.fR;
  const double *vol = A_.vol, *ctr = A_.ctr, *m2 = A_.m2, *Sn = A_.Sn, *area = A_.area, *fshift = A_.fshift,
               *fctr = A_.fctr, *fnrm = A_.fnrm;
  double *Kop = A_.Kop, *ggw = A_.ggw, *lsw = A_.lsw, *aux = A_.aux, *dtw = A_.dtw;
  DevErr* err = A_.err;
  const double V = vol[i];
  double c0[3], M0[6];
  for (int d = 0; d < 3; ++d) c0[d] = ctr[d * nc + i];
  for (int j = 0; j < 6; ++j) M0[j] = m2[j * nc + i];
  double dl[nt][3], Mn[nt][6];
#pragma unroll
  for (int m = 0; m < nt; ++m) {
    const int64_t f = cf[(int64_t)m * nc + i];
    const bool side = cside[(int64_t)m * nc + i] != 0;
    const double sg = side ? -1.0 : 1.0;
    double S[3];
    for (int d = 0; d < 3; ++d) S[d] = sg * Sn[d * nf + f];
    const double sn = sqrt(S[0] * S[0] + S[1] * S[1] + S[2] * S[2]);
    for (int d = 0; d < 3; ++d) {
      ggw[(3 * m + d) * nc + i] = S[d] / (2.0 * V);
      dtw[(4 * m + d) * nc + i] = S[d] * (area[f] / sn);
    }
    dtw[(4 * m + 3) * nc + i] = area[f];
    if (fR[f] >= 0) {
      const int64_t nb = side ? fL[f] : fR[f];
      for (int d = 0; d < 3; ++d) dl[m][d] = ctr[d * nc + nb] + sg * fshift[d * nf + f] - c0[d];
      for (int j = 0; j < 6; ++j) Mn[m][j] = m2[j * nc + nb];
    } else {
      double n[3], h = 0.0;
      for (int d = 0; d < 3; ++d) {
        n[d] = fnrm[d * nf + f];
        h += (c0[d] - fctr[d * nf + f]) * n[d];
      }
      for (int d = 0; d < 3; ++d) dl[m][d] = -2.0 * h * n[d];
      // mirrored moments R M R, R = I - 2 n n^T
      const double A[3][3] = {{M0[0], M0[3], M0[5]}, {M0[3], M0[1], M0[4]}, {M0[5], M0[4], M0[2]}};
      double An[3], nAn = 0.0;
      for (int r = 0; r < 3; ++r) {
        An[r] = A[r][0] * n[0] + A[r][1] * n[1] + A[r][2] * n[2];
        nAn += n[r] * An[r];
      }
      double B[3][3];
      for (int r = 0; r < 3; ++r)
        for (int s = 0; s < 3; ++s) B[r][s] = A[r][s] - 2.0 * (n[r] * An[s] + An[r] * n[s]) + 4.0 * nAn * n[r] * n[s];
      Mn[m][0] = B[0][0];
      Mn[m][1] = B[1][1];
      Mn[m][2] = B[2][2];
      Mn[m][3] = B[0][1];
      Mn[m][4] = B[1][2];
      Mn[m][5] = B[0][2];
    }
  }
  for (int m = nt; m < 6; ++m) {
    for (int d = 0; d < 3; ++d) ggw[(3 * m + d) * nc + i] = 0.0;
    for (int d = 0; d < 4; ++d) dtw[(4 * m + d) * nc + i] = 0.0;
  }
  // C (nt x 9): averages of the basis X,Y,Z,X^2,Y^2,Z^2,XY,YZ,XZ over the neighbour minus over the cell
  constexpr int mb = 3 * nt, nz = 9 - nt;
  double Ct[9 * nt];  // C^T, column-major 9 x nt
#pragma unroll
  for (int m = 0; m < nt; ++m) {
    const double* x = dl[m];
    const double* M = Mn[m];
    const double row[9] = {x[0], x[1], x[2], M[0] + x[0] * x[0] - M0[0], M[1] + x[1] * x[1] - M0[1],
                           M[2] + x[2] * x[2] - M0[2], M[3] + x[0] * x[1] - M0[3], M[4] + x[1] * x[2] - M0[4],
                           M[5] + x[0] * x[2] - M0[5]};
#pragma unroll
    for (int j = 0; j < 9; ++j) Ct[m * 9 + j] = row[j];
  }
  // product of row 3 m + d of B (3nt x 9) with y: averages of the derivatives of the basis over neighbour
  // m, 4 of the 9 not zero
  const auto B_row = [&dl](int m, int d, const double* y) {
    const double* x = dl[m];
    double s = y[d];
    s += 2 * x[d] * y[3 + d];
    s += d == 0 ? x[1] * y[6] : d == 1 ? x[0] * y[6] : x[1] * y[7];
    s += d == 0 ? x[2] * y[8] : d == 1 ? x[2] * y[7] : x[0] * y[8];
    return s;
  };
  double tc[nt];
  if (!house_qr<9, nt>(Ct, tc)) {
    set_err(err, CGKS_EMESH, (int)i, 50);
    return;
  }
  // A1 = Q1 R^{-T} (9 x nt), Q1 the first nt columns of Q: each row x of A1 solves R x^T = (row of Q1)^T,
  // back substitution; R[k][j] is stored at Ct[j*9 + k]
  double A1[9 * nt];
#pragma unroll
  for (int col = 0; col < nt; ++col) {
    double* y = A1 + col * 9;
#pragma unroll
    for (int r = 0; r < 9; ++r) y[r] = r == col ? 1.0 : 0.0;
    house_apply<9, nt, false>(Ct, tc, y);
  }
  double rc[nt];
#pragma unroll
  for (int k = 0; k < nt; ++k) rc[k] = 1.0 / Ct[k * 9 + k];
#pragma unroll
  for (int r = 0; r < 9; ++r)
#pragma unroll
    for (int k = nt - 1; k >= 0; --k) {
      double s = A1[k * 9 + r];
#pragma unroll
      for (int j = k + 1; j < nt; ++j) s -= Ct[j * 9 + k] * A1[j * 9 + r];
      A1[k * 9 + r] = quotient(s, Ct[k * 9 + k], rc[k]);
    }
  double BA[nt * mb];  // B A1 (mb x nt)
#pragma unroll
  for (int k = 0; k < nt; ++k)
#pragma unroll
    for (int r = 0; r < mb; ++r) BA[k * mb + r] = B_row(r / 3, r % 3, A1 + k * 9);
  // Q2 (9 x nz), the other columns of Q, and B Q2 (mb x nz)
  double Q2[9 * nz], BQ2[mb * nz], tb[nz];
#pragma unroll
  for (int c = 0; c < nz; ++c) {
    double* y = Q2 + c * 9;
#pragma unroll
    for (int r = 0; r < 9; ++r) y[r] = r == nt + c ? 1.0 : 0.0;
    house_apply<9, nt, false>(Ct, tc, y);
#pragma unroll
    for (int r = 0; r < mb; ++r) BQ2[c * mb + r] = B_row(r / 3, r % 3, y);
  }
  if (!house_qr<mb, nz>(BQ2, tb)) {
    set_err(err, CGKS_EMESH, (int)i, 51);
    return;
  }
  // P2 = (BQ2)^+ = Rb^{-1} Qb^T (nz x mb): the first nz columns of Qb, then back substitution per row of
  // Qb (forming all of Qb^T from the identity would take three times the operations)
  double P2[nz * mb];
#pragma unroll
  for (int col = 0; col < nz; ++col) {
    double* y = P2 + col * mb;
#pragma unroll
    for (int r = 0; r < mb; ++r) y[r] = r == col ? 1.0 : 0.0;
    house_apply<mb, nz, false>(BQ2, tb, y);
  }
  double rb[nz];
#pragma unroll
  for (int r = 0; r < nz; ++r) rb[r] = 1.0 / BQ2[r * mb + r];
#pragma unroll
  for (int col = 0; col < mb; ++col)
#pragma unroll
    for (int r = nz - 1; r >= 0; --r) {
      double s = P2[r * mb + col];
#pragma unroll
      for (int j = r + 1; j < nz; ++j) s -= BQ2[j * mb + r] * P2[j * mb + col];
      P2[r * mb + col] = quotient(s, BQ2[r * mb + r], rb[r]);
    }
  // row by row: Kg = Q2 P2 (9 x mb), KdQ = A1 - Kg (B A1) (9 x nt)
#pragma unroll
  for (int r = 0; r < 9; ++r) {
    double dq[nt];
#pragma unroll
    for (int k = 0; k < nt; ++k) dq[k] = A1[k * 9 + r];
#pragma unroll
    for (int col = 0; col < mb; ++col) {
      double s = 0.0;
#pragma unroll
      for (int j = 0; j < nz; ++j) s += Q2[j * 9 + r] * P2[j * mb + col];
      Kop[(r * 24 + 6 + col) * nc + i] = s;
#pragma unroll
      for (int k = 0; k < nt; ++k) dq[k] -= s * BA[k * mb + col];
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) Kop[(r * 24 + k) * nc + i] = k < nt ? dq[k < nt ? k : 0] : 0.0;
#pragma unroll
    for (int col = mb; col < 18; ++col) Kop[(r * 24 + 6 + col) * nc + i] = 0.0;
  }
  // least-squares gradient weights: D^+ with D = [dl_m] (nt x 3)
  double D[nt * 3], td[3];
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int m = 0; m < nt; ++m) D[d * nt + m] = dl[m][d];
  if (!house_qr<nt, 3>(D, td)) {
    set_err(err, CGKS_EMESH, (int)i, 52);
    return;
  }
  double rd[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) rd[r] = 1.0 / D[r * nt + r];
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    double y[nt], g[3] = {0.0, 0.0, 0.0};
    if (m < nt) {
#pragma unroll
      for (int r = 0; r < nt; ++r) y[r] = r == m ? 1.0 : 0.0;
      house_apply<nt, 3, true>(D, td, y);
#pragma unroll
      for (int r = 2; r >= 0; --r) {
        double s = y[r];
#pragma unroll
        for (int j = r + 1; j < 3; ++j) s -= D[j * nt + r] * g[j];
        g[r] = quotient(s, D[r * nt + r], rd[r]);
      }
    }
    for (int d = 0; d < 3; ++d) lsw[(3 * m + d) * nc + i] = g[d];
  }
  const double c13 = cbrt(V);
  aux[0 * nc + i] = c13 * c13;  // |Omega|^(2/3)
  aux[1 * nc + i] = V * c13;    // |Omega|^(4/3)
  for (int j = 0; j < 6; ++j) aux[(2 + j) * nc + i] = M0[j];
}

__host__ __device__ inline void recon_ops_body(int64_t i, const ROArgs& a) {
  switch (cell_nfaces(a.ctype[i])) {
    case 4: recon_ops_cell<4>(i, a); break;
    case 5: recon_ops_cell<5>(i, a); break;
    default: recon_ops_cell<6>(i, a); break;
  }
}
