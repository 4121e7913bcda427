"""The FP64 flux that the kernels run (gks_flux) against the generic point flux in extended precision
(point_flux<long double>) on the host, over states, options and sides of the face, and the table behind
its half-space moments.

Tolerances: the flux takes about 1,300 FP64 operations per point; a conservative flux or interface
state is compared with 1e-12 of the size of the terms it sums (as in the other parity tests: the larger
side's state, for the flux times |u| + c and the weight): several hundred rounding errors of that scale,
amplified by the cancellation in the pressure at Mach 8 (gamma (gamma - 1)/2 M^2 = 18).  The flux-only
variant is the same arithmetic: equal bits."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2402_02075_gb300", "csrc")

HARNESS = r'''
#include "fine.cuh"

typedef long double LD;
HD LD rsqrt_hd(LD x) { return 1.0L / sqrtl(x); }
template <> HD LD tsqrt<LD>(LD x) { return sqrtl(x); }
template <> HD LD tpow<LD>(LD x, LD y) { return powl(x, y); }

// p = (gamma, mu, prandtl, sutherland, cf); out: gks_flux F, Wg, alpha; flux-only F; point_flux F, Wg, alpha
extern "C" int both(const double* p, int bnd, int tag, const double* WL, const double* GL, const double* WR,
                    const double* GR, const double* n, double weight, double dt, double* out) {
  Phys ph{};
  ph.gamma = p[0];
  ph.K = (5.0 - 3.0 * p[0]) / (p[0] - 1.0);
  ph.mu = p[1];
  ph.viscous = p[1] >= 0.0;
  ph.prandtl = p[2];
  ph.suth = p[3];
  ph.cf = (int)p[4];
  ph.eps_inviscid = 0.01;
  ph.c_press = 1.0;
  ph.Winf[0] = 1.0; ph.Winf[1] = 0.5; ph.Winf[4] = 1.0 / p[0] / (p[0] - 1.0) + 0.125;
  DevErr err{};
  double Wr[5], Gr[15];
  for (int q = 0; q < 5; ++q) Wr[q] = WR[q];
  for (int j = 0; j < 15; ++j) Gr[j] = GR[j];
  if (bnd) bc_ghost<double>(tag, n, WL, GL, Wr, Gr, ph.gamma, ph.Winf);
  double scratch[5], al;
  const int a = gks_flux<true>(n, weight, bnd, WL, GL, Wr, Gr, dt, ph, nullptr, out, out + 5, out[10]);
  const int b = gks_flux<false>(n, weight, bnd, WL, GL, Wr, Gr, dt, ph, nullptr, out + 11, scratch, al);
  LD wl[5], gl[15], wr[5], gr[15], Fl[5], Wl[5], all;
  for (int q = 0; q < 5; ++q) wl[q] = WL[q], wr[q] = WR[q];
  for (int j = 0; j < 15; ++j) gl[j] = GL[j], gr[j] = GR[j];
  point_flux<LD>(n, 1.0 / weight, bnd, tag, wl, gl, wr, gr, (LD)dt, ph, Fl, Wl, all, &err, 0);
  for (int q = 0; q < 5; ++q) out[16 + q] = (double)Fl[q], out[21 + q] = (double)Wl[q];
  out[26] = (double)all;
  return a != b || a != err.detail;
}

// the 41 x 10 linearisation of a point by point_jacobian_body, and by point_flux on dual numbers, input by input
extern "C" int jacobians(const double* p, int bnd, int tag, const double* WL, const double* GL, const double* WR,
                         const double* GR, const double* A, double dt, double* Jn, double* Jo) {
  PointArgs a{};
  const int32_t face = 0, fL = 0, fR = bnd ? -1 : 1, ftag = bnd ? tag : -1;
  const double x[3] = {0, 0, 0}, shift[3] = {0, 0, 0}, ctr[6] = {0, 0, 0, 0, 0, 0}, dts[2] = {dt, dt * 1.5};
  alignas(16) double rc[100];
  for (int s = 0; s < 2; ++s)
    for (int q = 0; q < 5; ++q)
      for (int k = 0; k < 10; ++k)
        rc[50 * s + 10 * q + k] = k == 0 ? (s ? WR : WL)[q] : (k < 4 ? (s ? GR : GL)[3 * q + k - 1] : 0.0);
  DevErr err{};
  a.ngp = 1; a.nf = 1; a.nc = 2;
  a.gp_face = &face; a.fL = &fL; a.fR = &fR; a.ftag = &ftag;
  a.gp_x = x; a.gp_A = A; a.fshift = shift; a.ctr = ctr; a.rc = rc; a.dt = dts; a.err = &err;
  Phys& ph = a.ph;
  ph.gamma = p[0];
  ph.K = (5.0 - 3.0 * p[0]) / (p[0] - 1.0);
  ph.mu = p[1];
  ph.viscous = p[1] >= 0.0;
  ph.prandtl = p[2];
  ph.suth = p[3];
  ph.eps_inviscid = 0.01;
  ph.c_press = 1.0;
  ph.Winf[0] = 1.0; ph.Winf[1] = 0.5; ph.Winf[4] = 1.0 / p[0] / (p[0] - 1.0) + 0.125;
  point_jacobian_body(0, a, Jn);
  PointIn in;
  point_inputs(0, a, in);
  for (int k = 0; k < 41; ++k) {
    DualD wl[5], gl[15], wr[5], gr[15], F[5], W[5], al;
    for (int q = 0; q < 5; ++q) wl[q] = DualD(WL[q], k == q), wr[q] = DualD(WR[q], k == 20 + q);
    for (int j = 0; j < 15; ++j) gl[j] = DualD(GL[j], k == 5 + j), gr[j] = DualD(GR[j], k == 25 + j);
    point_flux<DualD>(in.n, in.iw, bnd, tag, wl, gl, wr, gr, DualD(dt, k == 40), ph, F, W, al, &err, 0);
    for (int o = 0; o < 5; ++o) Jo[10 * k + o] = F[o].d, Jo[10 * k + 5 + o] = W[o].d;
    if (bnd && k >= 20 && k < 40)
      for (int o = 0; o < 10; ++o) Jo[10 * k + o] = 0.0;
  }
  return err.code;
}

// largest relative error of the table's erfc(a)/2 over na points of [0, 6], and of its powers of two
extern "C" double table_error(int na) {
  static double t[HALF_TABLE];
  half_table_fill(t);
  double worst = 0.0;
  for (int i = 0; i <= na; ++i) {
    const long double a = 6.0L * i / na;
    const int j = (int)roundl(a * HALF_STEPS);
    const double* c = t + j * HALF_ROW;
    const double d = (double)(a - c[0]);
    long double q = c[9];
    for (int k = 8; k >= 1; --k) q = q * d + c[k];
    const long double ref = 0.5L * erfcl(c[0] + (long double)d) * expl((c[0] + (long double)d) * (c[0] + (long double)d));
    worst = fmax(worst, (double)fabsl(q / ref - 1.0L));
  }
  for (int i = 0; i < 64; ++i) worst = fmax(worst, (double)fabsl(t[HALF_EXP + i] * exp2l(i / 64.0L) - 1.0L));
  return worst;
}
'''


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("host_flux")
    (d / "h.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-fPIC", "-shared", "--expt-relaxed-constexpr",
                    "-I" + os.path.join(ROOT, "include"), "-I" + CSRC, "-o", str(d / "h.so"), str(d / "h.cu")], check=True)
    L = C.CDLL(str(d / "h.so"))
    L.both.argtypes = [C.c_void_p, C.c_int, C.c_int] + [C.c_void_p] * 5 + [C.c_double] * 2 + [C.c_void_p]
    L.table_error.restype = C.c_double
    L.jacobians.argtypes = [C.c_void_p, C.c_int, C.c_int] + [C.c_void_p] * 5 + [C.c_double] + [C.c_void_p] * 2
    return L


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


@pytest.mark.parametrize("gamma", [1.4, 5.0 / 3.0, 1.2])
@pytest.mark.parametrize("mu,prandtl,suth", [(-1.0, 1.0, 0.0), (1e-3, 0.72, 0.0), (1e-3, 1.0, 0.383), (0.0, 0.72, 0.0)])
@pytest.mark.parametrize("bnd,tag", [(0, -1), (1, 1), (1, 2), (1, 3), (1, 4), (1, 5)])
def test_flux_matches_the_generic_point_flux(host, gamma, mu, prandtl, suth, bnd, tag):
    rng = np.random.default_rng(17)
    for k in range(24):
        mach = [0.0, 0.3, 3.0, 8.0][k % 4]
        jump = [0.0, 0.05, 0.8][k % 3]
        axis = np.eye(3)[k % 3] if k < 6 else rng.normal(size=3)
        n = axis / np.linalg.norm(axis)
        base = rng.normal(size=3)
        base *= mach / np.linalg.norm(base)

        def state():
            rho, p = np.exp(jump * rng.normal()), np.exp(jump * rng.normal()) / gamma
            u = base + jump * rng.normal(size=3)
            return np.array([rho, *(rho * u), p / (gamma - 1.0) + 0.5 * rho * u @ u])
        WL, WR = state(), state()
        GL, GR = rng.normal(size=15) * 0.3, rng.normal(size=15) * 0.3
        out = np.zeros(27)
        prm = np.array([gamma, mu, prandtl, suth, 1.0])
        assert host.both(_p(prm), bnd, tag, _p(WL), _p(GL), _p(WR), _p(GR), _p(n), 0.37, [1e-6, 0.01, 0.2][k % 3], _p(out)) == 0
        F, W, al, F0, Fp, Wp, alp = out[:5], out[5:10], out[10], out[11:16], out[16:21], out[21:26], out[26]
        assert np.isfinite(Fp).all()
        sides = [WL] if bnd else [WL, WR]
        sw = max(np.abs(w).max() for w in sides)
        speed = max(np.linalg.norm(w[1:4]) / w[0] + np.sqrt(gamma * (gamma - 1.0) * w[4] / w[0]) for w in sides)
        assert np.abs(F - Fp).max() <= 1e-12 * 0.37 * sw * speed, (k, F, Fp)
        assert np.abs(W - Wp).max() <= 1e-12 * sw, (k, W, Wp)
        assert abs(al - alp) <= 1e-12, (k, al, alp)
        assert np.array_equal(F, F0)


@pytest.mark.parametrize("mu,prandtl,suth", [(-1.0, 1.0, 0.0), (1e-3, 0.72, 0.383), (1e-3, 1.0, 0.0)])
@pytest.mark.parametrize("bnd,tag", [(0, -1), (1, 1), (1, 2), (1, 3), (1, 4), (1, 5)])
def test_point_linearisation_matches_duals_input_by_input(host, mu, prandtl, suth, bnd, tag):
    """Rank-one gradient columns, one-sided state columns (the right ones by symmetry) and the time
    step's against 41 dual evaluations of the generic flux.  Both are exact derivatives in FP64 of some
    3,000 operations; a column is compared with 1e-10 of the largest entry of its kind (state, gradient,
    time step) in the flux rows and in the state rows (the conservative-to-primitive cancellation at Mach 3
    squared, gamma (gamma - 1)/2 M^2 = 2.5, on 1e-12; a column itself can be the small difference of a
    side's and its mirror image's at a wall)."""
    rng = np.random.default_rng(23)
    for k in range(12):
        mach, jump = [0.3, 1.2, 3.0][k % 3], [0.02, 0.2][k % 2]
        base = rng.normal(size=3)
        base *= mach / np.linalg.norm(base)

        def state():
            rho, p = np.exp(jump * rng.normal()), np.exp(jump * rng.normal()) / 1.4
            u = base + jump * rng.normal(size=3)
            return np.array([rho, *(rho * u), p / 0.4 + 0.5 * rho * u @ u])
        WL, WR = state(), state()
        GL, GR = rng.normal(size=15) * 0.3, rng.normal(size=15) * 0.3
        A = rng.normal(size=3) * 0.2
        Jn, Jo = np.zeros((41, 10)), np.zeros((41, 10))
        prm = np.array([1.4, mu, prandtl, suth])
        assert host.jacobians(_p(prm), bnd, tag, _p(WL), _p(GL), _p(WR), _p(GR), _p(A), [0.003, 0.05][k % 2], _p(Jn), _p(Jo)) == 0
        for rows in (slice(0, 5), slice(5, 10)):
            scale = np.abs(Jo[:, rows]).max(axis=1, keepdims=True)
            states, grads = np.r_[0:5, 20:25], np.r_[5:20, 25:40]
            scale[states], scale[grads] = scale[states].max(), scale[grads].max()
            assert (np.abs(Jn[:, rows] - Jo[:, rows]) <= 1e-10 * scale).all(), \
                (k, (np.abs(Jn[:, rows] - Jo[:, rows]).max(axis=1) / np.maximum(scale[:, 0], 1e-300)).max())


def test_half_space_table(host):
    """Rows are rounded once (2^-53 = 1.1e-16) and the polynomial's remainder is below 2^-58."""
    assert host.table_error(20011) <= 2.3e-16
