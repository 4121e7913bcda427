// Kernels of the fine-level CGKS residual (bodies in fine.cuh) and their host launchers.
#include "fine.cuh"

// ---- reconstruction ------------------------------------------------------------------------------
//
// The FP64 pipe bounds it (about 310 FP64 instructions per cell and variable, most of them the operator
// product), and a sub-partition of an SM takes 64 clocks for one warp's FP64 instruction however many
// independent ones that warp has.  So a cell's five variables go to five warps and its time step to a
// sixth: they share the operator through L1, need no spills (one thread for all five variables took
// 128 registers and 872 bytes of stack), and a launch of few cells ends after the chain of one variable.
// The ghosts of boundary slots are formed once per block, one slot per warp, and passed through shared
// memory.  Measured (CUDA events, one thread per cell before): 1.51 M cells of the 96x64x69 boundary
// layer 4.19 ms against 4.81, 94,464 cells 0.31 ms against 0.42, 1,152 cells 23 us against 95.  One-warp
// blocks that form their own ghosts were slower at every size (5.30 ms, 0.37 ms, 25 us).
#define RECON_GROUP 192  // 6 warps: 5 variables and the time step

__global__ void __launch_bounds__(RECON_GROUP) k_reconstruct(ReconArgs a) {
  __shared__ double gs[20 * RECON_GROUP];  // ghost (W_c, gradient of W_c) of slot m: [4 c ..][32 m + lane]
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  const int64_t nc = a.nc, i = blockIdx.x * (int64_t)32 + lane;
  const bool ghost = i < nc && q < (a.ctype[i] == 7 ? 5 : a.ctype[i]) && recon_neighbour(i, q, a) < 0;
  wait_prior();
  if (ghost) {  // slot q of cell i
    double Wg[5], Gg[15];
    recon_ghost(i, q, a, Wg, Gg);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      gs[(4 * c) * RECON_GROUP + threadIdx.x] = Wg[c];
#pragma unroll
      for (int d = 0; d < 3; ++d) gs[(4 * c + 1 + d) * RECON_GROUP + threadIdx.x] = Gg[3 * c + d];
    }
  }
  __syncthreads();
  if (i >= nc) return;
  if (q == 5) {
    double Q0[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) Q0[c] = a.W[c * nc + i];
    a.dt[i] = time_step<double>(i, a, Q0);
    return;
  }
  double out[10];
  reconstruct_variable(i, q, a, [&](int m, double v[4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = gs[(4 * q + c) * RECON_GROUP + 32 * m + lane];
  }, out);
  double2* dst = reinterpret_cast<double2*>(a.rc + (int64_t)CGKS_RC * i + 10 * q);
#pragma unroll
  for (int k = 0; k < 5; ++k) dst[k] = make_double2(out[2 * k], out[2 * k + 1]);
}

template <bool STATE>
__global__ void __launch_bounds__(128) k_gks_points(PointArgs a) {
  wait_prior();
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g < a.ngp) gks_point_body<STATE>(g, a);
}

// ---- gather: per cell, fixed-order sums of its faces' Gauss-point records ----------------------
//
// One thread per cell, 32 cells per warp.  The records of a face are contiguous (3 or 4 records of
// 112 bytes), so for each local-face slot the warp copies the 32 faces' records into shared memory
// with 16-byte cp.async copies, lanes of one copy instruction covering one face's contiguous bytes
// (coalesced), and each thread then sums its own face from shared memory in ascending point order
// (gather_face, the same arithmetic and order as gather_body).  The copies of slot m + 1 are in
// flight while slot m is summed (two buffers per warp).  GRAD false (residual only): the first three
// chunks of each record (the flux) are copied.

#define GATHER_WARPS 2                      // warps per block
#define GATHER_FACE_DOUBLES (4 * CGKS_GPR)  // room for the records of one face: 448 bytes
#define GATHER_SMEM (GATHER_WARPS * 2 * 32 * GATHER_FACE_DOUBLES * (int)sizeof(double))

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_one() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

template <bool GRAD>
__global__ void __launch_bounds__(32 * GATHER_WARPS) k_gather(GatherArgs a) {
  constexpr int CH = GRAD ? CGKS_GPR / 2 : 3;  // 16-byte chunks copied per record
  extern __shared__ __align__(16) double gsm[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t nc = a.nc;
  const int64_t i = ((int64_t)blockIdx.x * GATHER_WARPS + w) * 32 + lane;
  const bool valid = i < nc;
  const int nt = valid ? (a.ctype[i] == 7 ? 5 : a.ctype[i]) : 0;  // pyramids (type 7) have 5 faces
  const int nmax = __reduce_max_sync(0xffffffffu, nt);
  double* const buf0 = gsm + (size_t)(2 * w) * 32 * GATHER_FACE_DOUBLES;  // buffers of slots 0, 2, 4
  double* const buf1 = buf0 + 32 * GATHER_FACE_DOUBLES;                    // and of slots 1, 3, 5
  // face slot m of this lane's cell: first record, number of records, side sign
  auto slot = [&](int m, int64_t& g0, int& ng, bool& sg) {
    g0 = 0;
    ng = 0;
    sg = false;
    if (m < nt) {
      const int64_t f = a.cf[(int64_t)m * nc + i];
      sg = a.cside[(int64_t)m * nc + i] != 0;
      g0 = a.gp_ptr[f];
      ng = (int)(a.gp_ptr[f + 1] - g0);
    }
  };
  // the 32 faces of one slot into buffer b: chunk c of record k of face j by lane k CH + c, each to
  // its offset within the face's records (lanes 0 .. CH ng - 1; CH ng <= 28)
  const int rk = lane / CH, rc = lane - rk * CH;
  const int off = CGKS_GPR * rk + 2 * rc;
  auto issue = [&](double* b, int64_t g0, int ng) {
    for (int j = 0; j < 32; ++j) {
      const int64_t gj = __shfl_sync(0xffffffffu, g0, j);
      const int nj = __shfl_sync(0xffffffffu, ng, j);
      if (rk < nj) cp_async16(b + j * GATHER_FACE_DOUBLES + off, a.gpr + CGKS_GPR * gj + off);
    }
    cp_async_commit();
  };
  GatherAcc c;
  gather_init(c);
  int64_t g0;
  int ng;
  bool sg;
  slot(0, g0, ng, sg);
  if (nmax > 0) issue(buf0, g0, ng);
  for (int m = 0; m < nmax; ++m) {
    int64_t g1 = 0;
    int n1 = 0;
    bool s1 = false;
    if (m + 1 < nmax) {
      slot(m + 1, g1, n1, s1);
      issue((m & 1) ? buf0 : buf1, g1, n1);
    } else {
      cp_async_commit();  // an empty group keeps "all but the newest group" meaning slot m
    }
    cp_async_wait_one();
    __syncwarp();
    if (ng > 0) gather_face<GRAD>(((m & 1) ? buf1 : buf0) + lane * GATHER_FACE_DOUBLES, ng, sg, c);
    __syncwarp();  // every lane is done with buffer m & 1 before slot m + 2 is copied into it
    g0 = g1;
    ng = n1;
    sg = s1;
  }
  if (valid) gather_store(i, a, c);
}

// The gather on a small mesh: a thread per cell and variable instead of one for all five, since there the
// time is that of one warp (540 FP64 instructions of 64 clocks each, one face after the other: 32 us).  A
// cell's five threads are neighbours, so that they read a record's flux and state as one segment from L2,
// without staging; the sums run in the same order.  With `norm` the density residual's norm is formed on
// the way, from per-block sums that the last block to finish adds in block order.  Up to half a warp of
// cells per sub-partition: 1,152 cells 20 us against 44 for gather and norm, 7,296 cells 21 against 38; at
// 18,432 cells both take 49.
#define GATHER_VARS 128                                   // threads: 4 warps of 6 cells
#define GATHER_VARS_CELLS (6 * GATHER_VARS / 32)

struct GatherNorm {
  double *part, *out;
  unsigned* done;
};

template <bool GRAD>
__global__ void __launch_bounds__(GATHER_VARS) k_gather_vars(GatherArgs a, GatherNorm norm) {
  __shared__ double ws[GATHER_VARS / 32];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = lane / 5, q = lane - 5 * c;
  const int64_t nc = a.nc, i = (int64_t)blockIdx.x * GATHER_VARS_CELLS + 6 * warp + c;
  const bool live = c < 6 && i < nc;
  const int nt = live ? (a.ctype[i] == 7 ? 5 : a.ctype[i]) : 0;
  double r = 0.0, gs[3] = {0.0, 0.0, 0.0}, al = 1.0;
  int64_t g0[6];
  int ng[6];
  uint64_t sg[6];
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    const int64_t f = m < nt ? a.cf[(int64_t)m * nc + i] : 0;
    g0[m] = a.gp_ptr[f];
    ng[m] = m < nt ? a.gp_ptr[f + 1] - (int)g0[m] : 0;
    sg[m] = m < nt && a.cside[(int64_t)m * nc + i] ? 0x8000000000000000ull : 0ull;
  }
  wait_prior();
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    double v[4][6];  // flux, state, area vector, factor of the face's points
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k >= ng[m]) continue;
      const double* rec = a.gpr + (int64_t)CGKS_GPR * (g0[m] + k);
      v[k][0] = rec[q];
      if (GRAD) {
        v[k][1] = rec[5 + q];
#pragma unroll
        for (int d = 0; d < 4; ++d) v[k][2 + d] = rec[10 + d];
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k >= ng[m]) continue;
      r -= xor_sign(v[k][0], sg[m]);
      if (GRAD) {
#pragma unroll
        for (int d = 0; d < 3; ++d) gs[d] += v[k][1] * xor_sign(v[k][2 + d], sg[m]);
        al *= v[k][5];
      }
    }
  }
  const double rv = live ? 1.0 / a.vol[i] : 0.0;
  double w = 0.0;
  if (live) {
    if (a.res) a.res[q * nc + i] = r;
    if (GRAD && a.G_out) {
      const double k = al * rv;
#pragma unroll
      for (int d = 0; d < 3; ++d) a.G_out[(3 * q + d) * nc + i] = k * gs[d];
    }
    if (GRAD && a.alpha_out && q == 0) a.alpha_out[i] = al;
    if (GRAD && a.update) a.W_out[q * nc + i] = w = a.W_in[q * nc + i] + a.dt[i] * rv * r;
  }
  if (GRAD && a.update) {  // the cell's five values meet in its first thread
    double u[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) u[k] = __shfl_sync(0xffffffffu, w, lane + k > 31 ? 31 : lane + k);
    const double p = (a.gamma - 1.0) * (u[4] - 0.5 * (u[1] * u[1] + u[2] * u[2] + u[3] * u[3]) / u[0]);
    if (live && q == 0 && (!(u[0] > 0.0) || !(p > 0.0) || !isfinite(p))) set_err(a.err, CGKS_ENAN, (int)i, 6);
  }
  if (!norm.out) return;
  const double x = live && q == 0 ? r / a.vol[i] : 0.0;
  double s = x * x;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
  if (lane == 0) ws[warp] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    s = ws[0];
    for (int k = 1; k < GATHER_VARS / 32; ++k) s += ws[k];
    norm.part[blockIdx.x] = s;
    __threadfence();
    last = atomicAdd(norm.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last || warp != 0) return;
  __threadfence();
  s = 0.0;
  for (unsigned k = lane; k < gridDim.x; k += 32) s += __ldcg(norm.part + k);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
  if (lane == 0) {
    *norm.out = sqrt(s / (double)nc);
    *norm.done = 0;  // for the next launch
  }
}

// global minimum time step (dt_mode 1): fixed-order two-stage reduction, then broadcast
__global__ void k_min_partial(int64_t n, const double* __restrict__ x, double* __restrict__ part) {
  __shared__ double s[256];
  double v = 1e300;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    v = fmin(v, x[i]);
  s[threadIdx.x] = v;
  __syncthreads();
  for (int k = blockDim.x / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) s[threadIdx.x] = fmin(s[threadIdx.x], s[threadIdx.x + k]);
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}

__global__ void k_min_broadcast(int64_t n, int nparts, const double* __restrict__ part, double* __restrict__ x) {
  __shared__ double mn;
  if (threadIdx.x == 0) {
    double v = 1e300;
    for (int k = 0; k < nparts; ++k) v = fmin(v, part[k]);
    mn = v;
  }
  __syncthreads();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) x[i] = mn;
}

cgks_status global_min_dt(cgks_ctx* ctx, double* dt, int64_t n) {
  const int parts = 304;
  k_min_partial<<<parts, 256, 0, ctx->stream>>>(n, dt, ctx->nrm_part);
  k_min_broadcast<<<parts, 256, 0, ctx->stream>>>(n, parts, ctx->nrm_part, dt);
  CK(cudaGetLastError());
  return CGKS_OK;
}

cgks_status fine_fluxes(cgks_ctx* ctx, const double* W, const double* G, const double* alpha, bool state) {
  const Fine& F = ctx->F;
  const Phys ph = make_phys(ctx->P);
  ReconArgs ra{F.nc, F.nf, F.ctype, F.cf, F.fL, F.fR, F.ftag, F.cside, F.fnrm, F.Kop, F.ggw, F.lsw, F.aux, F.dtw,
               F.vol, W, G, alpha, ctx->rc, ctx->dt, ph, ctx->derr, F.nbr};
  const double slots = (double)(F.nf + F.n_int + F.n_per);
  {
    ProfScope ps(ctx, PK_RECON, (double)F.nc, F.nc * (306.0 * 8 + 1 + 51.0 * 8) + slots * 5 + F.nf * 36.0);
    CK(launch_overlapped(k_reconstruct, grid_for(F.nc, 32), RECON_GROUP, ctx->stream, ra));
  }
  if (ctx->P.dt_mode == 1) CKS(global_min_dt(ctx, ctx->dt, F.nc));
  PointArgs pa{F.ngp, F.nf, F.nc, F.gp_face, F.fL, F.fR, F.ftag, F.gp_x, F.gp_A, F.fshift, F.ctr, ctx->rc,
               ctx->dt, ctx->gpr, ph, ctx->derr, ctx->tab};
  {
    ProfScope ps(ctx, state ? PK_POINTS : PK_POINTS_FLUX, (double)F.ngp,
                 F.ngp * (52.0 + (state ? 8.0 * CGKS_GPR : 40.0)) + F.nf * 36.0 + F.nc * 432.0);
    const int b = spread_block(F.ngp, 128, ctx->n_sm);
    if (state)
      CK(launch_overlapped(k_gks_points<true>, grid_for(F.ngp, b), b, ctx->stream, pa));
    else
      CK(launch_overlapped(k_gks_points<false>, grid_for(F.ngp, b), b, ctx->stream, pa));
  }
  CK(cudaGetLastError());
  return CGKS_OK;
}

cgks_status fine_gather(cgks_ctx* ctx, const double* W_in, double* W_out, double* res, double* G_out,
                        double* alpha_out, int update, double* norm_dev) {
  const Fine& F = ctx->F;
  GatherArgs ga{F.nc, F.ngp, F.ctype, F.cside, F.cf, F.gp_ptr, ctx->gpr, F.vol,
                ctx->dt, W_in, W_out, res, G_out, alpha_out, update, ctx->P.gamma, ctx->derr};
  // (the blocks' parts of the norm have to fit nrm_part)
  const unsigned vars_blocks = grid_for(F.nc, GATHER_VARS_CELLS);
  const bool small = F.nc <= (int64_t)ctx->n_sm * 4 * 16 && vars_blocks <= CGKS_NORM_PARTS;
  {
    // the residual alone (no gradient, compression factor or update): only the records' fluxes are read
    const bool grad = G_out || alpha_out || update;
    const double per_cell = 1 + 8 + (update ? 88 : 0) + (res ? 40 : 0) + (G_out ? 120 : 0) + (alpha_out ? 8 : 0);
    ProfScope ps(ctx, grad ? PK_GATHER : PK_GATHER_RES, (double)F.gp_sides,
                 F.nc * per_cell + (F.nf + F.n_int + F.n_per) * 5.0 + F.nf * 4.0 + F.ngp * (grad ? 8.0 * CGKS_GPR : 40.0));
    if (small) {
      const GatherNorm norm{ctx->nrm_part, norm_dev, ctx->nrm_done};
      if (grad)
        CK(launch_overlapped(k_gather_vars<true>, vars_blocks, GATHER_VARS, ctx->stream, ga, norm));
      else
        CK(launch_overlapped(k_gather_vars<false>, vars_blocks, GATHER_VARS, ctx->stream, ga, norm));
    } else {
      static bool smem_set = false;  // the kernel's dynamic shared memory exceeds the 48 KiB default
      if (!smem_set) {
        CK(cudaFuncSetAttribute(k_gather<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, GATHER_SMEM));
        CK(cudaFuncSetAttribute(k_gather<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, GATHER_SMEM));
        smem_set = true;
      }
      const int64_t per_block = 32 * GATHER_WARPS;
      const unsigned nb = (unsigned)((F.nc + per_block - 1) / per_block);
      if (grad)
        k_gather<true><<<nb, 32 * GATHER_WARPS, GATHER_SMEM, ctx->stream>>>(ga);
      else
        k_gather<false><<<nb, 32 * GATHER_WARPS, GATHER_SMEM, ctx->stream>>>(ga);
    }
  }
  CK(cudaGetLastError());
  return norm_dev && !small ? density_norm(ctx, res, F.vol, F.nc, norm_dev) : CGKS_OK;
}
