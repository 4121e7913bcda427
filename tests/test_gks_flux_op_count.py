"""Source-level operation counts of the flux that the kernels run (gks_flux_t, csrc/flux.cuh) per interior Gauss
point, with and without the interface state, on the counting scalar of test_flux_op_count.py: an accidental
change of its arithmetic shows up here, and the FP64 operations that bench.py states for the kernels are tied
to it."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

import bench
from test_flux_op_count import CSRC, HARNESS, ROOT, _p

MORE = r'''
static long g_half = 0;
CD Cnt fast_rcp(Cnt x) { CNT(g_div); return Cnt(1.0 / x.v); }
CD Cnt fast_rsqrt(Cnt x) { CNT(g_sqrt); return Cnt(1.0 / sqrt(x.v)); }
CD Cnt exp_neg(Cnt x, const double*) { CNT(g_trans); return Cnt(exp(-x.v)); }
CD bool positive(Cnt x) { return x.v > 0.0; }
CD void half_gauss(Cnt y, const double*, Cnt& m0, Cnt& e) {
  CNT(g_half);
  m0 = Cnt(0.5 * erfc(y.v));
  e = Cnt(exp(-y.v * y.v));
}
extern "C" void count_gks(int state, int viscous, double prandtl, const double* WL, const double* GL, const double* WR,
                          const double* GR, const double* n, double dt, long* out) {
  Phys ph{};
  ph.gamma = 1.4;
  ph.K = 2.0;
  ph.mu = viscous ? 1e-3 : 0.0;
  ph.prandtl = prandtl;
  ph.eps_inviscid = 0.01;
  ph.c_press = 1.0;
  ph.viscous = viscous;
  ph.cf = 1;
  Cnt wl[5], wr[5], F[5], Wt[5], al;
  for (int q = 0; q < 5; ++q) { wl[q] = WL[q]; wr[q] = WR[q]; }
  g_flop = g_div = g_sqrt = g_trans = g_half = 0;
  const int bad = state ? gks_flux_t<true, Cnt, Cnt, Cnt, Cnt>(n, 1.0, false, wl, GL, wr, GR, Cnt(dt), ph, nullptr, F, Wt, al)
                        : gks_flux_t<false, Cnt, Cnt, Cnt, Cnt>(n, 1.0, false, wl, GL, wr, GR, Cnt(dt), ph, nullptr, F, Wt, al);
  out[0] = g_flop; out[1] = g_div; out[2] = g_sqrt; out[3] = g_trans; out[4] = g_half; out[5] = bad;
}
'''


@pytest.fixture(scope="module")
def counter(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("gks_op_count")
    (d / "count.cu").write_text(HARNESS + MORE)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-Xcompiler", "-fPIC", "-shared", "--expt-relaxed-constexpr",
                    "-I" + os.path.join(ROOT, "include"), "-I" + CSRC, "-o", str(d / "count.so"), str(d / "count.cu")],
                   check=True)
    lib = C.CDLL(str(d / "count.so"))
    lib.count_gks.argtypes = [C.c_int, C.c_int, C.c_double] + [C.c_void_p] * 5 + [C.c_double, C.c_void_p]
    return lib


# FP64 operations (2 per multiply-add) of a reciprocal, of CUDA's rsqrt, of exp_neg and of half_gauss as their device
# code has them, and of the rest of a point's body: both sides' polynomials (30 per variable, 9 per side) and
# the unit normal (8 and an rsqrt)
RCP, RSQRT, EXP, HALF = 6, 9, 16, 35
BODY = 2 * (5 * 30 + 9) + 8 + RSQRT


@pytest.mark.parametrize("state,viscous,prandtl,expect", [
    (1, 0, 1.0, (1425, 7)), (1, 1, 0.72, (1540, 8)), (0, 0, 1.0, (1209, 6)), (0, 1, 0.72, (1324, 7))])
def test_flux_operation_count_per_gauss_point(counter, state, viscous, prandtl, expect):
    rng = np.random.default_rng(51)
    WL = np.array([1.0, 0.5, 0.1, 0.0, 2.0])
    WR = np.array([1.1, 0.4, 0.0, 0.1, 2.1])
    GL, GR = rng.normal(size=15) * 0.1, rng.normal(size=15) * 0.1
    n = np.array([0.6, 0.8, 0.0])
    out = np.zeros(6, np.int64)
    counter.count_gks(state, viscous, prandtl, _p(WL), _p(GL), _p(WR), _p(GR), _p(n), 0.01, out.ctypes.data_as(C.c_void_p))
    flop, rcp, rsqrt, exp, half, bad = (int(x) for x in out)
    assert not bad and (rcp, rsqrt, exp, half) == (expect[1], 2, 1, 2), out
    assert abs(flop - expect[0]) <= 0.01 * expect[0], out
    if viscous:  # the bench's case: the counters of the kernels agree with what the source has
        total = flop + RCP * rcp + RSQRT * rsqrt + EXP * exp + HALF * half + BODY
        stated = bench.FLOP_PER_GP if state else bench.FLOP_PER_GP_FLUX
        assert abs(total - stated) <= 0.02 * stated, (total, stated)
