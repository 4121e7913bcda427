// Coarse levels of the V-cycle (Sec. 4.2 of the paper): first-order KFVS residual, local time
// steps, FAS forcing and forward-Euler smoothing, volume-weighted state restriction, summed
// residual restriction, injection correction, and the residual norm.  All sums run in a fixed
// order (no floating-point atomics), so results are bitwise reproducible.
#include "internal.cuh"
#include "kinetic.cuh"

// KFVS face fluxes x area (FP64)
__global__ void k_kfvs_faces(int64_t nf, const int32_t* __restrict__ fL, const int32_t* __restrict__ fR,
                             const int32_t* __restrict__ ftag, const double* __restrict__ nS, int64_t nc,
                             const double* W, double* ff, Phys ph, DevErr* err, const double* __restrict__ tab) {
  const int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool live = f < nf;
  const double s = live ? nS[3 * nf + f] : 0.0;
  const double n[3] = {live ? nS[f] : 0.0, live ? nS[nf + f] : 0.0, live ? nS[2 * nf + f] : 0.0};
  const int64_t L = live ? fL[f] : 0, R = live ? fR[f] : 0;
  const int32_t tag = live && R < 0 ? ftag[f] : 0;
  wait_prior();
  if (!live) return;
  if (s == 0.0) {  // a coarse face whose summed area vectors cancel carries no flux
#pragma unroll
    for (int q = 0; q < 5; ++q) ff[q * nf + f] = 0.0;
    return;
  }
  double WL[5], WR[5], F[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) WL[q] = W[q * nc + L];
  if (R >= 0) {
#pragma unroll
    for (int q = 0; q < 5; ++q) WR[q] = W[q * nc + R];
  } else if (!bc_ghost<double>(tag, n, WL, nullptr, WR, nullptr, ph.gamma, ph.Winf)) {
    set_err(err, CGKS_ENAN, (int)L, 20);
  }
  if (!kfvs_flux<double>(WL, WR, n, ph.K, ph.gamma - 1.0, F, tab)) set_err(err, CGKS_ENAN, (int)L, 21);
#pragma unroll
  for (int q = 0; q < 5; ++q) ff[q * nf + f] = s * F[q];
}

// Directional derivative of the KFVS face fluxes x area at the state W0 in the direction dW, in
// FP32 forward mode: dW = X - W0 when x_is_state, else X.  The boundary ghost state is
// differentiated with the cell state it is built from.
__global__ void k_kfvs_jvp_faces(int64_t nf, const int32_t* __restrict__ fL, const int32_t* __restrict__ fR,
                                 const int32_t* __restrict__ ftag, const double* __restrict__ Sn, int64_t nc,
                                 const double* W0, const double* X, int x_is_state, float* ff, Phys ph, DevErr* err) {
  using D = Dual<float>;
  wait_prior();
  const int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (f >= nf) return;
  const float S[3] = {float(Sn[f]), float(Sn[nf + f]), float(Sn[2 * nf + f])};
  const float s = sqrtf(S[0] * S[0] + S[1] * S[1] + S[2] * S[2]);
  if (s == 0.0f) {  // no net area, no flux
#pragma unroll
    for (int q = 0; q < 5; ++q) ff[q * nf + f] = 0.0f;
    return;
  }
  const D n[3] = {D(S[0] / s), D(S[1] / s), D(S[2] / s)};
  const int64_t L = fL[f], R = fR[f];
  D WL[5], WR[5], F[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const double w = W0[q * nc + L], x = X[q * nc + L];
    WL[q] = D(float(w), float(x_is_state ? x - w : x));
  }
  if (R >= 0) {
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const double w = W0[q * nc + R], x = X[q * nc + R];
      WR[q] = D(float(w), float(x_is_state ? x - w : x));
    }
  } else if (!bc_ghost<D>(ftag[f], n, WL, nullptr, WR, nullptr, D(ph.gamma), ph.Winf)) {
    set_err(err, CGKS_ENAN, (int)L, 23);
  }
  if (!kfvs_flux<D>(WL, WR, n, D(ph.K), D(ph.gamma - 1.0), F)) set_err(err, CGKS_ENAN, (int)L, 24);
#pragma unroll
  for (int q = 0; q < 5; ++q) ff[q * nf + f] = s * F[q].d;
}

// ---- sums over a coarse cell's faces -------------------------------------------------------------
//
// A coarse cell has 10 to 40 faces, read through its face list: a thread that walks them alone takes
// as many dependent trips to L2.  Where a level is small, eight threads share a cell's faces and add their
// partial sums in a fixed tree; above that one thread per cell is faster, since a warp's FP64 addition takes
// as long for a few active lanes as for 32.  Per launch, with one thread and with eight, in us (the mean
// over the launches of two levels, whose mean number of cells is given):
//   step       9,500 cells 23.5 and 21.8,  11,200 23.7 and 24.6,  14,700 23.9 and 30.4,  21,300 26.0 and 40.3
//   time step 11,200 cells 16.3 and 13.4,  14,700 15.8 and 15.7,  17,100 16.8 and 18.2,  21,300 15.8 and 19.9
//   gather    11,400 cells 21.9 and 14.9,  18,500 22.2 and 20.7,  21,300 20.1 and 19.3,  26,200 20.5 and 20.9
// The step's line depends on the faces per cell: 10,500 cells on a first coarse level (about 12 faces), 13,700
// on a second (about 22); it is put where one thread is the faster on both.
#define STEP_LANE_CELLS 96  // cells per SM below which eight threads share a cell
#define DT_LANE_CELLS 96
#define GATHER_LANE_CELLS 128
inline bool share_cells(int64_t nc, int n_sm, int cells) { return nc < (int64_t)n_sm * cells; }

template <int LANES>
__device__ __forceinline__ double lane_sum(double v) {
#pragma unroll
  for (int d = LANES / 2; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// res = -(sum of outward face fluxes) in FP64
template <typename T, int LANES>
__global__ void k_kfvs_gather(int64_t nc, int64_t nf, const int32_t* __restrict__ ptr, const int32_t* __restrict__ c2f,
                              const int32_t* __restrict__ fL, const int32_t* __restrict__ fR, const T* ff,
                              double* res) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, c = t / LANES;
  const int sub = (int)(t % LANES);
  const bool live = c < nc;
  double r[5] = {0, 0, 0, 0, 0};
  const int32_t e = live ? ptr[c + 1] : 0;
  int32_t k = live ? ptr[c] + sub : 0;
  wait_prior();
  for (; k < e; k += LANES) {
    const int64_t f = c2f[k];
    const int32_t a = fL[f], b = fR[f];
    if (a == b) continue;  // a cell's periodic image of itself: the two sides cancel
    const double s = a == c ? 1.0 : -1.0;
#pragma unroll
    for (int q = 0; q < 5; ++q) r[q] -= s * (double)ff[q * nf + f];
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) r[q] = lane_sum<LANES>(r[q]);
  if (live && sub == 0)
#pragma unroll
    for (int q = 0; q < 5; ++q) res[q * nc + c] = r[q];
}

// velocity and sound speed of a coarse cell's state
__device__ __forceinline__ double coarse_sound(const double w[5], double gamma, double u[3]) {
  const double r = fast_rcp(w[0]);
#pragma unroll
  for (int d = 0; d < 3; ++d) u[d] = w[1 + d] * r;
  const double p = (gamma - 1.0) * (w[4] - 0.5 * (w[1] * u[0] + w[2] * u[1] + w[3] * u[2]));
  return sqrt(gamma * p * r);
}

// local time step CFL |Omega| / sum_p A_p (|u . n_p| + c): A_p the area of the coarse face (the sum
// of its fine faces' areas), n_p the direction of its summed area vector (nS; zero, so no |u . n|
// term, when that vector cancels)
template <int LANES>
__global__ void k_coarse_dt(int64_t nc, int64_t nf, const int32_t* __restrict__ ptr, const int32_t* __restrict__ c2f,
                            const double* __restrict__ nS, const double* __restrict__ area,
                            const double* __restrict__ vol, const double* W, double* dt, double gamma, double cfl) {
  wait_prior();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, c = t / LANES;
  const int sub = (int)(t % LANES);
  const bool live = c < nc;
  double w[5], u[3], s = 0.0;
#pragma unroll
  for (int q = 0; q < 5; ++q) w[q] = live ? W[q * nc + c] : 1.0;
  const double snd = coarse_sound(w, gamma, u);
  const int32_t e = live ? ptr[c + 1] : 0;
  for (int32_t k = live ? ptr[c] + sub : 0; k < e; k += LANES) {
    const int64_t f = c2f[k];
    const double un = fabs(u[0] * nS[f] + u[1] * nS[nf + f] + u[2] * nS[2 * nf + f]);
    s += area[f] * (un + snd);
  }
  s = lane_sum<LANES>(s);
  if (live && sub == 0) dt[c] = cfl * vol[c] / s;
}

// One forward-Euler step of a coarse level from its face fluxes, in one pass over each cell's faces: the
// residual R (the gather), the local time step (k_coarse_dt), on a level's first step the forcing
// F = Res* - R (stored), and W += dt / |Omega| (R + F).  GATHER false (first step of the mixed cycle):
// R = 0 and F = Res*.  An update that would make rho or p non-positive is skipped for that cell
// (counted), a non-finite one is an error.  The faces' fluxes are those of W before the step, so W is
// updated in place.  Bound by its FP64 additions, with lanes idle where a warp's cells differ in faces
// (48-byte face and flux records instead of component arrays changed nothing).  One launch instead of four
// (gather, forcing, time step, update), and the cell's face list is read once: 0.23 ms per step of the
// 96x64x69 boundary layer (0.58 M cells on average) against 0.31, 12 us against 45 on the 24x4x24 one
// (2,231 cells).
struct CoarseStep {
  int64_t nc, nf;
  const int32_t *ptr, *c2f, *fL, *fR;
  const double *nS, *area, *Rs;
  double *F, *W;
  double gamma, cfl;
  int first;
  unsigned long long* skipped;
  DevErr* err;
};

// what the step needs of face entry k of cell c from the mesh alone
struct StepFace {
  int64_t f;
  int32_t l, r;
  double n[3], area;
};

template <bool GATHER>
__device__ __forceinline__ StepFace step_face(const CoarseStep& a, int32_t k, int32_t e) {
  StepFace F{};
  if (k >= e) return F;
  F.f = a.c2f[k];
#pragma unroll
  for (int d = 0; d < 3; ++d) F.n[d] = a.nS[d * a.nf + F.f];
  F.area = a.area[F.f];
  if (GATHER) F.l = a.fL[F.f], F.r = a.fR[F.f];
  return F;
}

template <typename T, int LANES, bool GATHER>
__global__ void k_coarse_step(CoarseStep a, const T* ff) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, c = t / LANES;
  const int64_t nc = a.nc, nf = a.nf;
  const int sub = (int)(t % LANES);
  const bool live = c < nc;
  double w[5], u[3], s = 0.0, r[5] = {0, 0, 0, 0, 0};
  const int32_t e = live ? a.ptr[c + 1] : 0;
  int32_t k = live ? a.ptr[c] + sub : 0;
  StepFace F = step_face<GATHER>(a, k, e);
  wait_prior();
#pragma unroll
  for (int q = 0; q < 5; ++q) w[q] = live ? a.W[q * nc + c] : 1.0;
  const double snd = coarse_sound(w, a.gamma, u);
  while (k < e) {
    k += LANES;
    const StepFace next = step_face<GATHER>(a, k, e);
    s += F.area * (fabs(u[0] * F.n[0] + u[1] * F.n[1] + u[2] * F.n[2]) + snd);
    if (GATHER && F.l != F.r) {  // not a cell's periodic image of itself
      const double sg = F.l == c ? 1.0 : -1.0;
#pragma unroll
      for (int q = 0; q < 5; ++q) r[q] -= sg * (double)ff[q * nf + F.f];
    }
    F = next;
  }
  s = lane_sum<LANES>(s);
  if (GATHER)
#pragma unroll
    for (int q = 0; q < 5; ++q) r[q] = lane_sum<LANES>(r[q]);
  if (!live || sub != 0) return;
  const double h = a.cfl / s;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    double F = a.first ? a.Rs[q * nc + c] : a.F[q * nc + c];
    if (GATHER && a.first) a.F[q * nc + c] = F = F - r[q];
    w[q] += h * (r[q] + F);
  }
  const double p = (a.gamma - 1.0) * (w[4] - 0.5 * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]) / w[0]);
  if (!(isfinite(w[0]) && isfinite(w[1]) && isfinite(w[2]) && isfinite(w[3]) && isfinite(w[4]))) {
    set_err(a.err, CGKS_ENAN, (int)c, 22);
  } else if (w[0] > 0.0 && p > 0.0) {
#pragma unroll
    for (int q = 0; q < 5; ++q) a.W[q * nc + c] = w[q];
  } else {
    atomicAdd(a.skipped, 1ULL);
  }
}

// F = Rs - R  (FAS forcing term)
__global__ void k_forcing(int64_t n5, const double* Rs, const double* R, double* F) {
  wait_prior();
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j < n5) F[j] = Rs[j] - R[j];
}

// W += dt / V (R + F); an update that would make rho or p non-positive is skipped for that cell
// (counted), a non-finite one is an error
__global__ void k_fe_update(int64_t nc, const double* __restrict__ dt, const double* __restrict__ vol,
                            const double* __restrict__ R, const double* __restrict__ F, double* __restrict__ W,
                            double gamma, unsigned long long* skipped, DevErr* err) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= nc) return;
  const double h = dt[c] / vol[c];
  double w[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) w[q] = W[q * nc + c] + h * (R[q * nc + c] + F[q * nc + c]);
  const double p = (gamma - 1.0) * (w[4] - 0.5 * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]) / w[0]);
  if (!(isfinite(w[0]) && isfinite(w[1]) && isfinite(w[2]) && isfinite(w[3]) && isfinite(w[4]))) {
    set_err(err, CGKS_ENAN, (int)c, 22);
  } else if (w[0] > 0.0 && p > 0.0) {
#pragma unroll
    for (int q = 0; q < 5; ++q) W[q * nc + c] = w[q];
  } else {
    atomicAdd(skipped, 1ULL);
  }
}

// coarse state = sum V_i W_i / V_c (and its copy W^0) and coarse defect = sum (R_i [+ F_i]) over the
// finer cells of each coarse cell, in ascending finer-cell order, by one of two kernels with the same sums:
// a thread per coarse cell and variable where the level is small, since an agglomerate has a handful of
// members and the time of a small launch is that of the dependent loads of one thread (four members
// are in flight at once); a thread for all five variables above RESTRICT_CELLS coarse cells per SM, since
// there the member lists and volumes are read from memory once instead of five times.  Per launch (the
// mean of both levels' restrictions), by variable and by cell: 340 cells 6.6 and 10.8 us, 33,945 cells 11.3
// and 13.3, 143,000 cells 26.6 and 26.6, 205,000 cells 35.8 and 32.9, 554,000 cells 83.9 and 71.7.
#define RESTRICT_CELLS 1024

__global__ void k_restrict_vars(int64_t ncc, int64_t ncf, const int32_t* __restrict__ aptr,
                                const int32_t* __restrict__ agg, const double* __restrict__ vf,
                                const double* __restrict__ vc, const double* Wf, const double* Rf, const double* Ff,
                                double* Wc, double* Wc0, double* Rc) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int q = blockIdx.y;
  const bool live = c < ncc;
  double w = 0.0, r = 0.0;
  const int32_t e = live ? aptr[c + 1] : 0, k0 = live ? aptr[c] : 0;
  const double rv = live ? 1.0 / vc[c] : 0.0;
  wait_prior();
  if (!live) return;
  for (int32_t k = k0; k < e; k += 4) {
    double v[4], x[4], y[4], z[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t i = agg[k + j < e ? k + j : e - 1];
      v[j] = vf[i];
      x[j] = Wf[q * ncf + i];
      y[j] = Rf[q * ncf + i];
      z[j] = Ff ? Ff[q * ncf + i] : 0.0;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (k + j < e) {
        w += v[j] * x[j];
        r += Ff ? y[j] + z[j] : y[j];
      }
  }
  w *= rv;
  Wc[q * ncc + c] = w;
  Wc0[q * ncc + c] = w;
  Rc[q * ncc + c] = r;
}

__global__ void k_restrict_cells(int64_t ncc, int64_t ncf, const int32_t* __restrict__ aptr,
                                 const int32_t* __restrict__ agg, const double* __restrict__ vf,
                                 const double* __restrict__ vc, const double* Wf, const double* Rf, const double* Ff,
                                 double* Wc, double* Wc0, double* Rc) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool live = c < ncc;
  double w[5] = {0, 0, 0, 0, 0}, r[5] = {0, 0, 0, 0, 0};
  const int32_t e = live ? aptr[c + 1] : 0, k0 = live ? aptr[c] : 0;
  const double rv = live ? 1.0 / vc[c] : 0.0;
  wait_prior();
  if (!live) return;
  for (int32_t k = k0; k < e; ++k) {
    const int64_t i = agg[k];
    const double v = vf[i];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      w[q] += v * Wf[q * ncf + i];
      r[q] += Ff ? Rf[q * ncf + i] + Ff[q * ncf + i] : Rf[q * ncf + i];
    }
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    w[q] *= rv;
    Wc[q * ncc + c] = w[q];
    Wc0[q * ncc + c] = w[q];
    Rc[q * ncc + c] = r[q];
  }
}

// restriction from a finer level of n cells (volumes vf, state W, residual R and forcing F or null) to level l
static cgks_status restrict_to(cgks_ctx* ctx, int l, int64_t n, const double* vf, const double* W, const double* R,
                               const double* F) {
  const Level& L = ctx->L[l];
  CoarseBuf& B = ctx->C[l];
  ProfScope ps(ctx, PK_RESTRICT, (double)n, n * (F ? 132.0 : 92.0) + L.nc * 132.0);
  if (L.nc <= (int64_t)ctx->n_sm * RESTRICT_CELLS)
    CK(launch_overlapped(k_restrict_vars, dim3(grid_for(L.nc, 128), 5), 128, ctx->stream, L.nc, n, L.agg_ptr, L.agg, vf,
                         L.vol, W, R, F, B.W, B.W0, B.Rs));
  else
    CK(launch_overlapped(k_restrict_cells, grid_for(L.nc, 256), 256, ctx->stream, L.nc, n, L.agg_ptr, L.agg, vf, L.vol, W,
                         R, F, B.W, B.W0, B.Rs));
  return CGKS_OK;
}

// W_f += r (W_c - W_c^0) (injection, r = correction_relax); a correction that would make rho or p
// non-positive is skipped
__global__ void k_prolong(int64_t ncf, int64_t ncc, const int32_t* __restrict__ f2c, const double* Wc,
                          const double* Wc0, double* Wf, double gamma, double relax, unsigned long long* skipped) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t c = i < ncf ? f2c[i] : 0;
  wait_prior();
  if (i >= ncf) return;
  double w[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) w[q] = Wf[q * ncf + i] + relax * (Wc[q * ncc + c] - Wc0[q * ncc + c]);
  const double p = (gamma - 1.0) * (w[4] - 0.5 * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]) / w[0]);
  if (w[0] > 0.0 && p > 0.0) {
#pragma unroll
    for (int q = 0; q < 5; ++q) Wf[q * ncf + i] = w[q];
  } else {
    atomicAdd(skipped, 1ULL);
  }
}

// prolongation 1: cell i of the receiving level takes the volume-weighted mean of the injected
// corrections of itself and its face neighbours (in ascending face order), then W += relax x that
__global__ void k_prolong_smooth(int64_t ncf, int64_t ncc, const int32_t* __restrict__ ptr,
                                 const int32_t* __restrict__ c2f, const int32_t* __restrict__ fL,
                                 const int32_t* __restrict__ fR, const double* __restrict__ vol,
                                 const int32_t* __restrict__ f2c, const double* __restrict__ Wc,
                                 const double* __restrict__ Wc0, double* __restrict__ Wf, double gamma, double relax,
                                 unsigned long long* skipped) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= ncf) return;
  double acc[5], sv = vol[i];
  {
    const int64_t c = f2c[i];
#pragma unroll
    for (int q = 0; q < 5; ++q) acc[q] = vol[i] * (Wc[q * ncc + c] - Wc0[q * ncc + c]);
  }
  for (int32_t k = ptr[i]; k < ptr[i + 1]; ++k) {
    const int64_t f = c2f[k];
    const int32_t a = fL[f], b = fR[f];
    if (b < 0 || a == b) continue;
    const int64_t j = a == i ? b : a;
    const int64_t c = f2c[j];
    const double v = vol[j];
#pragma unroll
    for (int q = 0; q < 5; ++q) acc[q] += v * (Wc[q * ncc + c] - Wc0[q * ncc + c]);
    sv += v;
  }
  double w[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) w[q] = Wf[q * ncf + i] + relax * (acc[q] / sv);
  const double p = (gamma - 1.0) * (w[4] - 0.5 * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]) / w[0]);
  if (w[0] > 0.0 && p > 0.0) {
#pragma unroll
    for (int q = 0; q < 5; ++q) Wf[q * ncf + i] = w[q];
  } else {
    atomicAdd(skipped, 1ULL);
  }
}

static cgks_status prolong(cgks_ctx* ctx, int lev_fine, const int32_t* f2c, int64_t ncc, const double* Wc,
                    const double* Wc0, double* Wf) {
  const Level& L = ctx->L[lev_fine];
  cudaStream_t st = ctx->stream;
  ProfScope ps(ctx, PK_PROLONG, (double)L.nc,
               L.nc * 84.0 + ncc * 80.0 +
                   (ctx->P.prolongation == 1 ? (L.nf + L.n_int + L.n_per) * 4.0 + L.nf * 8.0 + L.nc * 12.0 : 0.0));
  if (ctx->P.prolongation == 1)
    k_prolong_smooth<<<grid_for(L.nc, 256), 256, 0, st>>>(L.nc, ncc, L.c2f_ptr, L.c2f, L.fL, L.fR, L.vol, f2c, Wc, Wc0,
                                                           Wf, ctx->P.gamma, ctx->P.correction_relax,
                                                           (unsigned long long*)ctx->d_skipped);
  else
    CK(launch_overlapped(k_prolong, grid_for(L.nc, 256), 256, st, L.nc, ncc, f2c, Wc, Wc0, Wf,
                         ctx->P.gamma, ctx->P.correction_relax, (unsigned long long*)ctx->d_skipped));
  return CGKS_OK;
}

// sqrt(mean (res_rho / V)^2): per-block partial sums, then one warp adds them in a fixed order (lane l the
// partials l, l + 32, ..., then a tree): 2 us where one thread's chain of 304 loads and additions took 22
__global__ void k_norm_partial(int64_t n, const double* res, const double* __restrict__ vol, double* part) {
  __shared__ double s[256];
  wait_prior();
  double acc = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double x = res[i] / vol[i];
    acc += x * x;
  }
  s[threadIdx.x] = acc;
  __syncthreads();
  for (int k = blockDim.x / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) s[threadIdx.x] += s[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}

__global__ void __launch_bounds__(32) k_norm_final(int nparts, int64_t n, const double* part, double* out) {
  wait_prior();
  double s = 0.0;
  for (int k = threadIdx.x; k < nparts; k += 32) s += part[k];
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
  if (threadIdx.x == 0) *out = sqrt(s / (double)n);
}

cgks_status density_norm(cgks_ctx* ctx, const double* res, const double* vol, int64_t n, double* out_dev) {
  const int parts = 304;
  ProfScope ps(ctx, PK_NORM, (double)n, n * 16.0);
  CK(launch_overlapped(k_norm_partial, parts, 256, ctx->stream, n, res, vol, ctx->nrm_part));
  CK(launch_overlapped(k_norm_final, 1, 32, ctx->stream, parts, n, ctx->nrm_part, out_dev));
  CK(cudaGetLastError());
  return CGKS_OK;
}

cgks_status global_min_dt(cgks_ctx* ctx, double* dt, int64_t n);

// KFVS face fluxes of level `lev` (FP64)
static cgks_status kfvs_fluxes(cgks_ctx* ctx, int lev, const double* W) {
  const Level& L = ctx->L[lev];
  double* ff = lev == 0 ? ctx->ffl : ctx->C[lev].ff;
  ProfScope ps(ctx, PK_KFVS_FACES, (double)L.nf, L.nf * 84.0 + L.nc * 40.0);
  const int b = spread_block(L.nf, 256, ctx->n_sm);
  CK(launch_overlapped(k_kfvs_faces, grid_for(L.nf, b), b, ctx->stream, L.nf, L.fL, L.fR, L.ftag, L.nS, L.nc, W, ff,
                       make_phys(ctx->P), ctx->derr, ctx->tab));
  return CGKS_OK;
}

// their FP32 directional derivatives at W0
static cgks_status kfvs_jvp_fluxes(cgks_ctx* ctx, int lev, const double* W0, const double* X, int x_is_state) {
  const Level& L = ctx->L[lev];
  float* ff = lev == 0 ? ctx->ffl32 : ctx->C[lev].ff32;
  ProfScope ps(ctx, PK_KFVS_JVP, (double)L.nf, L.nf * 56.0 + L.nc * 80.0);
  CK(launch_overlapped(k_kfvs_jvp_faces, grid_for(L.nf, 256), 256,
                       ctx->stream, L.nf, L.fL, L.fR, L.ftag, L.Sn, L.nc, W0, X, x_is_state, ff,
                       make_phys(ctx->P), ctx->derr));
  return CGKS_OK;
}

template <typename T>
static cgks_status kfvs_gather(cgks_ctx* ctx, int lev, const T* ff, double* res) {
  const Level& L = ctx->L[lev];
  ProfScope ps(ctx, PK_KFVS_GATHER, (double)L.nc,
               L.nc * 44.0 + (L.nf + L.n_int + L.n_per) * 4.0 + L.nf * (8.0 + 5.0 * sizeof(T)));
  if (share_cells(L.nc, ctx->n_sm, GATHER_LANE_CELLS))
    CK(launch_overlapped(k_kfvs_gather<T, 8>, grid_for(8 * L.nc, 64), 64,
                         ctx->stream, L.nc, L.nf, L.c2f_ptr, L.c2f, L.fL, L.fR, ff, res));
  else
    CK(launch_overlapped(k_kfvs_gather<T, 1>, grid_for(L.nc, 256), 256,
                         ctx->stream, L.nc, L.nf, L.c2f_ptr, L.c2f, L.fL, L.fR, ff, res));
  return CGKS_OK;
}

// KFVS residual of level `lev` (FP64)
cgks_status kfvs_residual(cgks_ctx* ctx, int lev, const double* W, double* res) {
  CKS(kfvs_fluxes(ctx, lev, W));
  CKS(kfvs_gather<double>(ctx, lev, lev == 0 ? ctx->ffl : ctx->C[lev].ff, res));
  CK(cudaGetLastError());
  return CGKS_OK;
}

cgks_status kfvs_jvp(cgks_ctx* ctx, int lev, const double* W0, const double* X, int x_is_state, double* res) {
  CKS(kfvs_jvp_fluxes(ctx, lev, W0, X, x_is_state));
  CKS(kfvs_gather<float>(ctx, lev, lev == 0 ? ctx->ffl32 : ctx->C[lev].ff32, res));
  CK(cudaGetLastError());
  return CGKS_OK;
}

cgks_status coarse_dt(cgks_ctx* ctx, int lev, const double* W, double* dt) {
  const Level& L = ctx->L[lev];
  {
    ProfScope ps(ctx, PK_COARSE_DT, (double)L.nc, L.nc * 60.0 + (L.nf + L.n_int + L.n_per) * 4.0 + L.nf * 32.0);
    if (share_cells(L.nc, ctx->n_sm, DT_LANE_CELLS))
      CK(launch_overlapped(k_coarse_dt<8>, grid_for(8 * L.nc, 64), 64,
                           ctx->stream, L.nc, L.nf, L.c2f_ptr, L.c2f, L.nS, L.area, L.vol, W, dt, ctx->P.gamma,
                           ctx->P.cfl_coarse));
    else
      CK(launch_overlapped(k_coarse_dt<1>, grid_for(L.nc, 256), 256,
                           ctx->stream, L.nc, L.nf, L.c2f_ptr, L.c2f, L.nS, L.area, L.vol, W, dt, ctx->P.gamma,
                           ctx->P.cfl_coarse));
  }
  if (ctx->P.dt_mode == 1) CKS(global_min_dt(ctx, dt, L.nc));
  CK(cudaGetLastError());
  return CGKS_OK;
}

// coarse-level residual at the current state B.W into B.R, the defect being B.R + forcing:
// FP64 FAS: R = Res(W), forcing B.F = Res* - Res(W^0);  precision 1 (defect correction): R = J(W^0)
// (W - W^0) in FP32 forward mode, forcing Res*, so the defect is linear in the correction W - W^0 and
// FP32 only perturbs it relative to its own size
static cgks_status coarse_residual(cgks_ctx* ctx, int l) {
  CoarseBuf& B = ctx->C[l];
  if (ctx->P.precision == 1) return kfvs_jvp(ctx, l, B.W0, B.W, 1, B.R);
  return kfvs_residual(ctx, l, B.W, B.R);
}

// B.F = Res* - R, the forcing of the FAS equations
static cgks_status coarse_forcing(cgks_ctx* ctx, int l) {
  CoarseBuf& B = ctx->C[l];
  const int64_t n5 = 5 * ctx->L[l].nc;
  ProfScope ps(ctx, PK_FORCING, (double)ctx->L[l].nc, n5 * 24.0);
  CK(launch_overlapped(k_forcing, grid_for(n5, 256), 256, ctx->stream, n5, B.Rs, B.R, B.F));
  CK(cudaGetLastError());
  return CGKS_OK;
}

static double* forcing(cgks_ctx* ctx, CoarseBuf& B) { return ctx->P.precision == 1 ? B.Rs : B.F; }

// a smoothing step with the residual in B.R, in separate launches: the implicit smoother, and the
// forward Euler step with one global time step
static cgks_status smooth_from_residual(cgks_ctx* ctx, int l) {
  const Level& L = ctx->L[l];
  CoarseBuf& B = ctx->C[l];
  CKS(coarse_dt(ctx, l, B.W, B.dt));
  if (ctx->P.coarse_smoother == 1) return lusgs_step(ctx, l, forcing(ctx, B));
  {
    ProfScope ps(ctx, PK_FE_UPDATE, (double)L.nc, L.nc * 176.0);
    k_fe_update<<<grid_for(L.nc, 256), 256, 0, ctx->stream>>>(L.nc, B.dt, L.vol, B.R, forcing(ctx, B), B.W, ctx->P.gamma,
                                                               (unsigned long long*)ctx->d_skipped, ctx->derr);
  }
  CK(cudaGetLastError());
  return CGKS_OK;
}

template <typename T, bool GATHER>
static cgks_status coarse_step(cgks_ctx* ctx, int l, const T* ff, bool first) {
  const Level& L = ctx->L[l];
  CoarseBuf& B = ctx->C[l];
  const CoarseStep a{L.nc, L.nf, L.c2f_ptr, L.c2f, L.fL, L.fR, L.nS, L.area, B.Rs, forcing(ctx, B), B.W, ctx->P.gamma,
                     ctx->P.cfl_coarse, first, (unsigned long long*)ctx->d_skipped, ctx->derr};
  ProfScope ps(ctx, GATHER ? PK_KFVS_GATHER : PK_COARSE_DT, (double)L.nc,
               L.nc * (first && GATHER ? 164.0 : 124.0) + (L.nf + L.n_int + L.n_per) * 4.0 +
                   L.nf * (32.0 + (GATHER ? 8.0 + 5.0 * sizeof(T) : 0.0)));
  if (share_cells(L.nc, ctx->n_sm, STEP_LANE_CELLS))
    CK(launch_overlapped(k_coarse_step<T, 8, GATHER>, grid_for(8 * L.nc, 64), 64, ctx->stream, a, ff));
  else
    CK(launch_overlapped(k_coarse_step<T, 1, GATHER>, grid_for(L.nc, 128), 128, ctx->stream, a, ff));
  return CGKS_OK;
}

// one smoothing step of level l.  first: at W = W^0 with the restricted defect in B.Rs, which also fixes
// the forcing (the mixed cycle's first residual is zero)
static cgks_status coarse_smooth(cgks_ctx* ctx, int l, bool first) {
  const Level& L = ctx->L[l];
  CoarseBuf& B = ctx->C[l];
  const bool mixed = ctx->P.precision == 1;
  if (ctx->P.coarse_smoother == 0 && ctx->P.dt_mode == 0) {
    if (mixed && first) {
      CKS((coarse_step<float, false>(ctx, l, nullptr, true)));
    } else if (mixed) {
      CKS(kfvs_jvp_fluxes(ctx, l, B.W0, B.W, 1));
      CKS((coarse_step<float, true>(ctx, l, B.ff32, false)));
    } else {
      CKS(kfvs_fluxes(ctx, l, B.W));
      CKS((coarse_step<double, true>(ctx, l, B.ff, first)));
    }
    CK(cudaGetLastError());
    return CGKS_OK;
  }
  if (mixed && first) {
    CK(cudaMemsetAsync(B.R, 0, sizeof(double) * 5 * L.nc, ctx->stream));
  } else {
    CKS(coarse_residual(ctx, l));
    if (first) CKS(coarse_forcing(ctx, l));
  }
  return smooth_from_residual(ctx, l);
}

// coarse level l of the V-cycle, entered with W = W^0 (the restricted state) and Res* (the
// restricted defect)
static cgks_status coarse_cycle(cgks_ctx* ctx, int l) {
  const Level& L = ctx->L[l];
  CoarseBuf& B = ctx->C[l];
  if (ctx->P.coarse_steps == 0 && ctx->P.precision == 0) {  // the forcing alone
    CKS(coarse_residual(ctx, l));
    CKS(coarse_forcing(ctx, l));
  }
  for (int s = 0; s < ctx->P.coarse_steps; ++s) CKS(coarse_smooth(ctx, l, s == 0));
  if (l + 1 < (int)ctx->L.size()) {
    const Level& Cn = ctx->L[l + 1];
    CoarseBuf& N = ctx->C[l + 1];
    CKS(coarse_residual(ctx, l));
    CKS(restrict_to(ctx, l + 1, L.nc, L.vol, B.W, B.R, forcing(ctx, B)));
    CKS(coarse_cycle(ctx, l + 1));
    CKS(prolong(ctx, l, Cn.f2c, Cn.nc, N.W, N.W0, B.W));
    for (int s = 0; s < ctx->P.post; ++s) CKS(coarse_smooth(ctx, l, false));
  }
  CK(cudaGetLastError());
  return CGKS_OK;
}

// one explicit CGKS step of the fine level (Eq. smo); norm of the residual before the step
cgks_status step_once(cgks_ctx* ctx, double* norm_dev) {
  CKS(fine_fluxes(ctx, ctx->W, ctx->G, ctx->alpha));
  // the gather reads only the Gauss-point records, so W, gradW and alpha are updated in place
  return fine_gather(ctx, ctx->W, ctx->W, ctx->res, ctx->G, ctx->alpha, 1, norm_dev);
}

// one V-cycle (Sec. 4.2)
cgks_status vcycle_once(cgks_ctx* ctx, double* norm_dev) {
  const int pre = ctx->P.pre > 0 ? ctx->P.pre : 1;
  for (int s = 0; s < pre; ++s) CKS(step_once(ctx, s == 0 ? norm_dev : nullptr));
  if (ctx->L.size() <= 1) return CGKS_OK;
  const Fine& F = ctx->F;
  const Level& C1 = ctx->L[1];
  CoarseBuf& B1 = ctx->C[1];
  // defect at the smoothed state (the residual alone: no interface state, gradient or compression
  // factor is formed)
  CKS(fine_fluxes(ctx, ctx->W, ctx->G, ctx->alpha, false));
  CKS(fine_gather(ctx, ctx->W, nullptr, ctx->res, nullptr, nullptr, 0));
  CKS(restrict_to(ctx, 1, F.nc, ctx->L0c.vol, ctx->W, ctx->res, nullptr));
  CKS(coarse_cycle(ctx, 1));
  CKS(prolong(ctx, 0, C1.f2c, C1.nc, B1.W, B1.W0, ctx->W));
  for (int s = 0; s < ctx->P.post; ++s) CKS(step_once(ctx, nullptr));
  CK(cudaGetLastError());
  return CGKS_OK;
}
