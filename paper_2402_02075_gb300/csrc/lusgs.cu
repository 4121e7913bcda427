// Implicit coarse-level smoother of Sec. 4.3 (backward Euler with the first-order Lax-Friedrichs
// Jacobian splitting, matrix-free symmetric Gauss-Seidel: LU-SGS) on the agglomerated levels.
//
// One step solves, for the increments dU,
//   (|Omega_i|/dt_i + 1/2 sum_p lambda_p S_p) dU_i
//       + sum_p 1/2 [F_n(U_p + dU_p) - F_n(U_p) - lambda_p dU_p] S_p = Res_i + F_i
// (n out of cell i, F_n the Euler flux through the face, lambda_p = max(|U.n| + c) of the two cells,
// S_p the length of the face's summed area vector) with one forward and one backward Gauss-Seidel
// sweep.  The sweep order is colour-major: Jones-Plassmann rounds on priorities
// (splitmix64(id), id) give every cell a colour shared by none of its neighbours, so each colour is
// one parallel launch and the result equals the sequential sweep in (colour, id) order.  Ghost
// neighbours keep dU = 0, faces whose area vectors cancel and a cell's periodic face with itself are
// skipped, and an increment that would make rho or p non-positive is not applied (counted).
#include <algorithm>
#include <vector>

#include "fastmath.cuh"
#include "internal.cuh"

namespace {

__device__ __forceinline__ uint64_t mix64(uint64_t x) {  // splitmix64 (Steele, Lea, Flood 2014)
  uint64_t z = x + 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

__device__ __forceinline__ int64_t other_cell(const int32_t* fL, const int32_t* fR, int64_t f, int64_t i) {
  const int32_t a = fL[f], b = fR[f];
  if (b < 0 || a == b) return -1;
  return a == i ? b : a;
}

// an uncoloured cell whose priority beats every uncoloured neighbour's is selected this round
__global__ void k_jpl_select(int64_t nc, const int32_t* __restrict__ ptr, const int32_t* __restrict__ c2f,
                             const int32_t* __restrict__ fL, const int32_t* __restrict__ fR,
                             const int32_t* __restrict__ color, int8_t* __restrict__ sel) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  int8_t top = color[i] < 0;
  const uint64_t pi = mix64((uint64_t)i);
  for (int32_t k = ptr[i]; k < ptr[i + 1] && top; ++k) {
    const int64_t j = other_cell(fL, fR, c2f[k], i);
    if (j < 0 || color[j] >= 0) continue;
    const uint64_t pj = mix64((uint64_t)j);
    if (pj > pi || (pj == pi && j > i)) top = 0;
  }
  sel[i] = top;
}

// selected cells take the smallest colour none of their (earlier-coloured) neighbours has; two
// selected cells are never neighbours, so the assignments of one round are independent
__global__ void k_jpl_assign(int64_t nc, const int32_t* __restrict__ ptr, const int32_t* __restrict__ c2f,
                             const int32_t* __restrict__ fL, const int32_t* __restrict__ fR,
                             const int8_t* __restrict__ sel, int32_t* __restrict__ color,
                             unsigned long long* left) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  if (!sel[i]) {
    if (color[i] < 0) atomicAdd(left, 1ULL);
    return;
  }
  for (int32_t c = 0;; ++c) {
    bool used = false;
    for (int32_t k = ptr[i]; k < ptr[i + 1] && !used; ++k) {
      const int64_t j = other_cell(fL, fR, c2f[k], i);
      used = j >= 0 && color[j] == c;
    }
    if (!used) {
      color[i] = c;
      return;
    }
  }
}

// What a sweep reads of a neighbour, one 128-byte line: its state (density, velocity, total enthalpy per
// mass), the same of U + dU, p(U + dU) - p(U) and dU.  With it F_n(U + dU) - F_n(U) is 20 FP64
// instructions per face; formed from the conservative states at each of a cell's 10 to 40 faces it was 60.
// With that and lane_scatter a V-cycle of the 64x32x8 ramp takes 1.77 ms instead of 2.07.
struct SweepRecord {
  double rho, u[3], h, rho1, u1[3], h1, dp, dU[5];
};
static_assert(sizeof(SweepRecord) == 128, "one line per cell");

// velocity, pressure and enthalpy of a conservative state
__device__ __forceinline__ double sweep_state(const double w[5], double g, double u[3], double& h) {
  const double r = fast_rcp(w[0]);
#pragma unroll
  for (int d = 0; d < 3; ++d) u[d] = w[1 + d] * r;
  const double p = (g - 1.0) * (w[4] - 0.5 * w[0] * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]));
  h = (w[4] + p) * r;
  return p;
}

__device__ __forceinline__ double wave_speed(const double* W, int64_t nc, int64_t i, const double n[3], double g) {
  const double rho = W[i], r = fast_rcp(rho);
  const double u[3] = {W[nc + i] * r, W[2 * nc + i] * r, W[3 * nc + i] * r};
  const double p = (g - 1.0) * (W[4 * nc + i] - 0.5 * rho * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]));
  return fabs(u[0] * n[0] + u[1] * n[1] + u[2] * n[2]) + sqrt(g * p * r);
}

// lambda of every face: max over its cells of |U.n| + c (the cell's own on boundary faces); nS: unit
// normal and length of the face's summed area vector
__global__ void k_lusgs_lambda(int64_t nf, const int32_t* __restrict__ fL, const int32_t* __restrict__ fR,
                               const double* __restrict__ nS, int64_t nc, const double* W, double g, double* lam) {
  wait_prior();
  const int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (f >= nf) return;
  if (nS[3 * nf + f] == 0.0) {
    lam[f] = 0.0;
    return;
  }
  const double n[3] = {nS[f], nS[nf + f], nS[2 * nf + f]};
  const int32_t a = fL[f], b = fR[f];
  const double la = wave_speed(W, nc, a, n, g);
  lam[f] = b >= 0 ? fmax(la, wave_speed(W, nc, b, n, g)) : la;
}

// Threads per cell of the kernels below.  A colour of a level holds a few hundred to a few thousand
// cells of 10 to 40 faces, and each sweep waits for the one before it, so the time of a sweep is that
// of one cell: a thread that walks the faces alone takes 100 us (a warp's FP64 instruction takes 64
// clocks of its sub-partition, about 100 of them per face, and the loads are dependent).  LANES threads
// share the faces and add their parts in a fixed tree: a quarter warp, or a whole warp where the
// colour has so few cells that every sub-partition still gets at most two.  V-cycle of the 64x32x8 ramp
// (7,235 and 4,102 coarse cells, 18 and 20 sweeps per step): 2.3 ms against 9.7.  Two V-cycles by that rule,
// with a quarter warp always and with a whole one always, since their records and scattered sums: 64x32x8 ramp
// (colours of up to 1,613 cells) 3.50, 3.88 and 3.53 ms, 64x32x16 ramp (3,300) 5.82, 6.11 and 6.03, 96x4x69
// boundary layer (12,284) 9.68, 9.80 and 11.25.  The five sums of a cell end in five of its lanes, each of
// which then does one variable's division.
template <int LANES>
__device__ __forceinline__ double lane_sum(double v) {
#pragma unroll
  for (int d = LANES / 2; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// the sums over the LANES threads of v[0..4], added pairwise as lane_sum adds them, each left in the lanes
// whose sweep_variable says so: 6 additions for 8 lanes where five lane_sums take 15
template <int LANES>
__device__ __forceinline__ double lane_scatter(const double v[5], int sub) {
  constexpr unsigned ALL = 0xffffffffu;
  constexpr int d1 = LANES / 2, d2 = LANES / 4, d3 = LANES / 8;
  const bool h1 = sub & d1, h2 = sub & d2, h3 = sub & d3;
  double a = (h1 ? v[3] : v[0]) + __shfl_xor_sync(ALL, h1 ? v[0] : v[3], d1);
  double b = (h1 ? v[4] : v[1]) + __shfl_xor_sync(ALL, h1 ? v[1] : v[4], d1);
  double c = (h1 ? 0.0 : v[2]) + __shfl_xor_sync(ALL, h1 ? v[2] : 0.0, d1);
  a = (h2 ? b : a) + __shfl_xor_sync(ALL, h2 ? a : b, d2);
  c = (h2 ? 0.0 : c) + __shfl_xor_sync(ALL, h2 ? c : 0.0, d2);
  a = (h3 ? c : a) + __shfl_xor_sync(ALL, h3 ? a : c, d3);
#pragma unroll
  for (int d = d3 / 2; d > 0; d >>= 1) a += __shfl_xor_sync(ALL, a, d);
  return a;
}

// the variable whose sum lane_scatter leaves in lane sub (-1: none)
template <int LANES>
__device__ __forceinline__ int sweep_variable(int sub) {
  constexpr int d1 = LANES / 2, d2 = LANES / 4, d3 = LANES / 8;
  if (sub & d3) return sub & (d1 | d2) ? -1 : 2;
  return (sub & d1 ? 3 : 0) + (sub & d2 ? 1 : 0);
}

// the lane that holds variable q
template <int LANES>
__device__ __forceinline__ int sweep_lane(int q) {
  return q == 2 ? LANES / 8 : (q >= 3 ? LANES / 2 : 0) + (q == 1 || q == 4 ? LANES / 4 : 0);
}

// D_i = |Omega_i| / dt_i + 1/2 sum_p lambda_p S_p, and the cell's state in its sweep record
template <int LANES>
__global__ void k_lusgs_diag(int64_t nc, int64_t nf, const int32_t* __restrict__ ptr, const int32_t* __restrict__ c2f,
                             const int32_t* __restrict__ fL, const int32_t* __restrict__ fR,
                             const double* __restrict__ nS, const double* lam, const double* __restrict__ vol,
                             const double* dt, const double* W, double g, double* D, SweepRecord* rec) {
  wait_prior();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, i = t / LANES;
  const bool live = i < nc;
  double s = 0.0;
  const int32_t e = live ? ptr[i + 1] : 0;
  for (int32_t k = live ? ptr[i] + (int)(t % LANES) : 0; k < e; k += LANES) {
    const int64_t f = c2f[k];
    if (fL[f] == fR[f]) continue;
    s += lam[f] * nS[3 * nf + f];
  }
  s = lane_sum<LANES>(s);
  if (!live || t % LANES != 0) return;
  D[i] = vol[i] / dt[i] + 0.5 * s;
  double w[5], u[3], h;
#pragma unroll
  for (int q = 0; q < 5; ++q) w[q] = W[q * nc + i];
  sweep_state(w, g, u, h);
  rec[i].rho = w[0];
#pragma unroll
  for (int d = 0; d < 3; ++d) rec[i].u[d] = u[d];
  rec[i].h = h;
}

struct SweepArgs {
  int64_t nc, nf;
  const int32_t *ptr, *c2f, *fL, *fR, *color, *cells;
  const double *nS, *lam, *W, *R, *F, *D;
  SweepRecord* rec;
  double gamma;
};

// what a sweep needs of face entry e of cell i from the mesh alone: the neighbour (-1: nothing to add),
// the unit normal out of the cell and the summed area
struct SweepFace {
  int64_t f, j;
  double n[3], s;
};

template <bool FWD>
__device__ __forceinline__ SweepFace sweep_face(const SweepArgs& a, int64_t i, int32_t e, int32_t end, int32_t k) {
  SweepFace F;
  F.j = -1;
  if (e >= end) return F;
  F.f = a.c2f[e];
  const int64_t l = a.fL[F.f], r = a.fR[F.f], j = l == i ? r : l;
  if (r < 0 || l == r || (FWD ? a.color[j] >= k : a.color[j] <= k)) return F;
  F.s = a.nS[3 * a.nf + F.f];
  if (F.s == 0.0) return F;
  F.j = j;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double v = a.nS[d * a.nf + F.f];
    F.n[d] = l == i ? v : -v;
  }
  return F;
}

// forward (FWD) or backward sweep over the cells of colour k: neighbours of a lower (forward) or
// higher (backward) colour contribute 1/2 [F_n(U_j + dU_j) - F_n(U_j) - lambda dU_j] S
template <bool FWD, int LANES>
__global__ void k_lusgs_sweep(SweepArgs a, int64_t count, int32_t k) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, pos = t / LANES;
  const int64_t nc = a.nc;
  const bool live = pos < count;
  const int64_t i = live ? a.cells[pos] : 0;
  const int sub = (int)(t % LANES), var = sweep_variable<LANES>(sub), q = var < 0 ? 0 : var;
  const int32_t end = live ? a.ptr[i + 1] : 0;
  int32_t e = live ? a.ptr[i] + sub : 0;
  SweepFace F = sweep_face<FWD>(a, i, e, end, k);
  wait_prior();  // everything above is the mesh and its colours; all below may come from the kernel before
  const double w = a.W[q * nc + i], Di = a.D[i];
  const double rhs = !live ? 0.0 : FWD ? a.R[q * nc + i] + a.F[q * nc + i] : a.rec[i].dU[q];
  double acc[5] = {0, 0, 0, 0, 0};
  while (e < end) {
    e += LANES;
    const SweepFace next = sweep_face<FWD>(a, i, e, end, k);
    if (F.j >= 0) {
      double2 v[8];
      const double2* src = reinterpret_cast<const double2*>(a.rec + F.j);
#pragma unroll
      for (int m = 0; m < 8; ++m) v[m] = src[m];
      const double lam = a.lam[F.f], hs = 0.5 * F.s;
      const double u[3] = {v[0].y, v[1].x, v[1].y}, u1[3] = {v[3].x, v[3].y, v[4].x};
      const double dU[5] = {v[5].y, v[6].x, v[6].y, v[7].x, v[7].y}, dp = v[5].x;
      const double m0 = v[0].x * (u[0] * F.n[0] + u[1] * F.n[1] + u[2] * F.n[2]);
      const double m1 = v[2].y * (u1[0] * F.n[0] + u1[1] * F.n[1] + u1[2] * F.n[2]);
      acc[0] += (m1 - m0 - lam * dU[0]) * hs;
#pragma unroll
      for (int d = 0; d < 3; ++d) acc[1 + d] += (u1[d] * m1 - u[d] * m0 + dp * F.n[d] - lam * dU[1 + d]) * hs;
      acc[4] += (v[4].y * m1 - v[2].x * m0 - lam * dU[4]) * hs;
    }
    F = next;
  }
  const double sum = lane_scatter<LANES>(acc, sub);
  const double x = FWD ? (rhs - sum) / Di : rhs - sum / Di;  // this lane's variable of dU
  // the cell's lanes meet for the record of U + dU
  double w0[5], w1[5], dU[5], u[3], h;
  const int base = (threadIdx.x & 31) & ~(LANES - 1);
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    dU[m] = __shfl_sync(0xffffffffu, x, base + sweep_lane<LANES>(m));
    w0[m] = __shfl_sync(0xffffffffu, w, base + sweep_lane<LANES>(m));
    w1[m] = w0[m] + dU[m];
  }
  const double p1 = sweep_state(w1, a.gamma, u, h);
  if (!live || sub != 0) return;
  SweepRecord& r = a.rec[i];
  const double p0 =
      (a.gamma - 1.0) * (w0[4] - 0.5 * w0[0] * (r.u[0] * r.u[0] + r.u[1] * r.u[1] + r.u[2] * r.u[2]));
  r.rho1 = w1[0];
#pragma unroll
  for (int d = 0; d < 3; ++d) r.u1[d] = u[d];
  r.h1 = h;
  r.dp = p1 - p0;
#pragma unroll
  for (int m = 0; m < 5; ++m) r.dU[m] = dU[m];
}

template <bool FWD>
cudaError_t sweep(const SweepArgs& a, int64_t cnt, int32_t k, int n_sm, cudaStream_t st) {
  if (cnt <= (int64_t)n_sm * 4 * 2)
    return launch_overlapped(k_lusgs_sweep<FWD, 32>, grid_for(32 * cnt, 32), 32, st, a, cnt, k);
  return launch_overlapped(k_lusgs_sweep<FWD, 8>, grid_for(8 * cnt, 64), 64, st, a, cnt, k);
}

// W += dU, skipping (and counting) cells whose rho or p would not stay positive
__global__ void k_lusgs_apply(int64_t nc, const SweepRecord* rec, double* W, double g, unsigned long long* skipped,
                              DevErr* err) {
  wait_prior();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nc) return;
  double w[5];
  bool fin = true;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    w[q] = W[q * nc + i] + rec[i].dU[q];
    fin = fin && isfinite(w[q]);
  }
  if (!fin) {
    set_err(err, CGKS_ENAN, (int)i, 25);
    return;
  }
  const double p = (g - 1.0) * (w[4] - 0.5 * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]) / w[0]);
  if (w[0] > 0.0 && p > 0.0) {
#pragma unroll
    for (int q = 0; q < 5; ++q) W[q * nc + i] = w[q];
  } else {
    atomicAdd(skipped, 1ULL);
  }
}

}  // namespace

// colours and the colour-major cell order of level l (built once per mesh)
cgks_status lusgs_colors(cgks_ctx* ctx, int l) {
  CoarseBuf& B = ctx->C[l];
  if (B.color) return CGKS_OK;
  const Level& L = ctx->L[l];
  cudaStream_t st = ctx->stream;
  auto& M = ctx->mesh_allocs;
  int8_t* sel = nullptr;
  CKS(dalloc(ctx, M, &B.color, L.nc));
  CKS(dalloc(ctx, M, &B.order, L.nc));
  CKS(dalloc(ctx, M, &B.lam, L.nf));
  CKS(dalloc(ctx, M, &B.Dg, L.nc));
  CKS(dalloc(ctx, M, &B.sweep, sizeof(SweepRecord) / sizeof(double) * L.nc));
  std::vector<void*> tmp;
  const FreeList guard{ctx, tmp};
  CKS(dalloc(ctx, tmp, &sel, L.nc));
  std::vector<int32_t> minus1(L.nc, -1);
  cudaError_t e = cudaMemcpyAsync(B.color, minus1.data(), sizeof(int32_t) * L.nc, cudaMemcpyHostToDevice, st);
  // each round colours at least the uncoloured cell of highest priority, so nc rounds bound it
  int64_t left = L.nc;
  for (int64_t round = 0; e == cudaSuccess && left > 0 && round <= L.nc; ++round) {
    k_jpl_select<<<grid_for(L.nc, 256), 256, 0, st>>>(L.nc, L.c2f_ptr, L.c2f, L.fL, L.fR, B.color, sel);
    e = cudaMemsetAsync(ctx->d_count, 0, sizeof(int64_t), st);
    if (e != cudaSuccess) break;
    k_jpl_assign<<<grid_for(L.nc, 256), 256, 0, st>>>(L.nc, L.c2f_ptr, L.c2f, L.fL, L.fR, sel, B.color,
                                                      (unsigned long long*)ctx->d_count);
    e = cudaMemcpyAsync(ctx->h_count, ctx->d_count, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) left = *ctx->h_count;
  }
  CK(e);
  if (left > 0) return cgks_fail(ctx, CGKS_EINVAL, "LU-SGS colouring did not finish");
  // colour-major order, ascending cell id within a colour (counting sort on the host)
  std::vector<int32_t> col(L.nc), order(L.nc);
  CK(cudaMemcpyAsync(col.data(), B.color, sizeof(int32_t) * L.nc, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  int32_t ncol = 0;
  for (int32_t c : col) ncol = std::max(ncol, c + 1);
  B.coff.assign(ncol + 1, 0);
  for (int32_t c : col) ++B.coff[c + 1];
  for (int32_t c = 0; c < ncol; ++c) B.coff[c + 1] += B.coff[c];
  std::vector<int64_t> pos(B.coff.begin(), B.coff.end() - 1);
  for (int64_t i = 0; i < L.nc; ++i) order[pos[col[i]]++] = (int32_t)i;
  CK(cudaMemcpyAsync(B.order, order.data(), sizeof(int32_t) * L.nc, cudaMemcpyHostToDevice, st));
  CK(cudaStreamSynchronize(st));
  return CGKS_OK;
}

// one LU-SGS step on level l for the defect B.R + F with the time steps in B.dt
cgks_status lusgs_step(cgks_ctx* ctx, int l, const double* F) {
  CKS(lusgs_colors(ctx, l));
  const Level& L = ctx->L[l];
  CoarseBuf& B = ctx->C[l];
  cudaStream_t st = ctx->stream;
  const double g = ctx->P.gamma;
  SweepRecord* rec = reinterpret_cast<SweepRecord*>(B.sweep);
  CK(launch_overlapped(k_lusgs_lambda, grid_for(L.nf, 128), 128, st, L.nf, L.fL, L.fR, L.nS, L.nc, B.W, g, B.lam));
  CK(launch_overlapped(k_lusgs_diag<8>, grid_for(8 * L.nc, 128), 128, st, L.nc, L.nf, L.c2f_ptr, L.c2f, L.fL, L.fR,
                       L.nS, B.lam, L.vol, B.dt, B.W, g, B.Dg, rec));
  SweepArgs a{L.nc, L.nf, L.c2f_ptr, L.c2f, L.fL, L.fR, B.color, B.order, L.nS, B.lam, B.W, B.R, F, B.Dg, rec, g};
  const int32_t ncol = (int32_t)B.coff.size() - 1;
  for (int32_t k = 0; k < ncol; ++k) {
    a.cells = B.order + B.coff[k];
    CK(sweep<true>(a, B.coff[k + 1] - B.coff[k], k, ctx->n_sm, st));
  }
  for (int32_t k = ncol - 1; k >= 0; --k) {
    a.cells = B.order + B.coff[k];
    CK(sweep<false>(a, B.coff[k + 1] - B.coff[k], k, ctx->n_sm, st));
  }
  CK(launch_overlapped(k_lusgs_apply, grid_for(L.nc, 256), 256, st, L.nc, rec, B.W, g,
                       (unsigned long long*)ctx->d_skipped, ctx->derr));
  CK(cudaGetLastError());
  return CGKS_OK;
}

cgks_status lusgs_color_count(cgks_ctx* ctx, int l, int32_t* colors, int32_t* n_colors) {
  CKS(lusgs_colors(ctx, l));
  const CoarseBuf& B = ctx->C[l];
  if (colors)
    CK(cudaMemcpyAsync(colors, B.color, sizeof(int32_t) * ctx->L[l].nc, cudaMemcpyDefault, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  if (n_colors) *n_colors = (int32_t)B.coff.size() - 1;
  return CGKS_OK;
}
