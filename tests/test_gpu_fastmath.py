"""The elementary functions of csrc/fastmath.cuh on the device against long double, over their ranges, the edges
of their tables and the inputs where their integer comparisons and FP32 parts could go wrong.

Bounds, in units of u = 2^-53 (half an ulp at 1):
 fast_rcp    the approximation takes and gives 20 mantissa bits, so |e| <= 2^-18.5 and e^3 <= 2^-55.5 = 0.18 u; the
             last multiply-add rounds by u: 1.2 u
 fast_rsqrt  an ulp: 2 u
 exp_neg     the power's and the polynomial's rounding u each, the product's u, the reduced argument's and the
             polynomial's remainder (|r|^6/720, |r| <= 1.03 ln 2/128: 0.3 u) and lower steps below 0.5 u: 3.6 u
 half_gauss  exp as above; erfc/2 the exp, c_0, the last step and the product u each, the lower steps (|d| <= 1/64
             times |c_1/c_0| <= 1.2) and the remainder below 0.4 u: 7 u; for y < 0 the same of a part below 1/2, and
             u of the difference of which is at least 1/2: 5 u"""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U = 2.0 ** -53

SRC = r"""
#include "fastmath.cuh"
__global__ void k_eval(int which, int n, const double* x, const double* y, const double* tab, double* o0, double* o1) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  o1[i] = 0.0;
  if (which == 0) o0[i] = fast_rcp(x[i]);
  if (which == 1) o0[i] = fast_rsqrt(x[i]);
  if (which == 2) o0[i] = exp_neg(x[i], tab);
  if (which == 3) half_gauss(x[i], tab, o0[i], o1[i]);
  if (which == 4) o0[i] = positive(x[i]);
  if (which == 5) o0[i] = min_positive(x[i], y[i]);
}
extern "C" int table_size() { return HALF_TABLE; }
extern "C" void table(double* t) { half_table_fill(t); }
extern "C" int eval(int which, int n, const double* x, const double* y, const double* tab, double* o0, double* o1) {
  k_eval<<<(n + 127) / 128, 128>>>(which, n, x, y, tab, o0, o1);
  return cudaDeviceSynchronize();
}
// relative errors of the results r0 (and r1) of function `which` in long double
extern "C" void errors(int which, int n, const double* x, const double* r0, const double* r1, double* e0, double* e1) {
  for (int i = 0; i < n; ++i) {
    const long double a = x[i];
    long double v0 = 0, v1 = 1;
    if (which == 0) v0 = 1 / a;
    if (which == 1) v0 = 1 / sqrtl(a);
    if (which == 2) v0 = expl(-a);
    if (which == 3) v0 = 0.5L * erfcl(a), v1 = expl(-a * a);
    e0[i] = (double)fabsl((r0[i] - v0) / v0);
    e1[i] = which == 3 ? (double)fabsl((r1[i] - v1) / v1) : 0.0;
  }
}
"""


@pytest.fixture(scope="module")
def fm(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_02075_gb300 import build
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("fastmath")
    (d / "f.cu").write_text(SRC)
    subprocess.run([nvcc, *build.GENCODE, *build.FLAGS, "-shared", "-o", str(d / "f.so"), str(d / "f.cu")], check=True)
    lib = C.CDLL(str(d / "f.so"))
    tab = np.zeros(lib.table_size())
    lib.table(tab.ctypes.data_as(C.c_void_p))
    tab = torch.from_numpy(tab).cuda()

    def p(t):
        return C.c_void_p(t.data_ptr())

    def run(which, x, y=None):
        x = torch.from_numpy(np.array(x, dtype=np.float64))
        g, h = x.cuda(), (x if y is None else torch.from_numpy(np.array(y, dtype=np.float64))).cuda()
        o0, o1 = torch.empty_like(g), torch.empty_like(g)
        torch.cuda.synchronize()
        assert lib.eval(which, len(x), p(g), p(h), p(tab), p(o0), p(o1)) == 0
        r0, r1 = o0.cpu(), o1.cpu()
        e0, e1 = torch.empty_like(x), torch.empty_like(x)
        lib.errors(which, len(x), p(x), p(r0), p(r1), p(e0), p(e1))
        return r0.numpy(), r1.numpy(), e0.numpy(), e1.numpy()
    return run


def _near(x):
    """the values with their neighbours"""
    x = np.asarray(x, dtype=np.float64)
    return np.concatenate([np.nextafter(x, -np.inf), x, np.nextafter(x, np.inf)])


NANS = np.array([0x7FF8000000000000, 0xFFF8000000000000, 0x7FFFFFFFFFFFFFFF, 0xFFFFFFFFFFFFFFFF, 0x7FF8000000000001],
                dtype=np.uint64).view(np.float64)


def _wide(rng, n, lo, hi):
    return np.exp2(rng.uniform(lo, hi, n)) * rng.uniform(1.0, 2.0, n)


def test_reciprocal(fm):
    rng = np.random.default_rng(1)
    x = np.concatenate([rng.uniform(1.0, 2.0, 200_000), _wide(rng, 100_000, -1020, 1019), _near(np.exp2(np.arange(-1020, 1020))),
                        _near(1.0 + np.arange(1 << 12) / (1 << 12))])
    for s in (1.0, -1.0):
        assert fm(0, s * x)[2].max() <= 1.2 * U
    bad = fm(0, np.concatenate([[0.0, -0.0, np.inf, -np.inf, 5e-324, -5e-324], NANS]))[0]
    assert not np.isfinite(bad[[0, 1, 4, 5]]).any() and np.isnan(bad[6:]).all()
    assert not (np.abs(bad[2:4]) > 0).any()  # of an infinity: zero or not a number


def test_reciprocal_square_root(fm):
    rng = np.random.default_rng(2)
    x = np.concatenate([rng.uniform(1.0, 4.0, 200_000), _wide(rng, 100_000, -1020, 1019), _near(np.exp2(np.arange(-1020, 1020)))])
    assert fm(1, x)[2].max() <= 2.0 * U
    assert not np.isfinite(fm(1, np.concatenate([[0.0, -0.0, -1.0, -np.inf], NANS]))[0]).any()


def test_exponential(fm):
    rng = np.random.default_rng(3)
    ties = (np.arange(0, 64 * 1000) + 0.5) * np.log(2.0) / 64.0  # where n changes
    x = np.concatenate([rng.uniform(0.0, 700.0, 200_000), _wide(rng, 50_000, -60, 0), _near(ties[ties < 699.9]), [0.0, 699.9]])
    x = x[x >= 0.0]
    assert fm(2, x)[2].max() <= 3.6 * U
    r = fm(2, np.concatenate([[-0.0, 700.5, 745.0, 1e4, 1e300, np.inf], NANS]))[0]
    assert r[0] == 1.0 and (r[1:6] == 0.0).all() and np.isnan(r[6:]).all()


def test_half_space_pair(fm):
    rng = np.random.default_rng(4)
    j = (np.arange(0, 6 * 32) + 0.5) / 32.0  # where the row changes
    n = np.sqrt((np.arange(0, 36 * 92) + 0.5) * np.log(2.0) / 64.0)
    a = np.concatenate([rng.uniform(0.0, 6.0, 300_000), _near(j), _near(n[n < 5.999]), _wide(rng, 20_000, -70, 0),
                        np.nextafter(6.0, 0.0) - np.arange(2000) * 1e-5, np.arange(0, 6 * 32) / 32.0])
    a = a[(a >= 0.0) & (a < 6.0)]
    m0, e, em, ee = fm(3, a)
    assert ee.max() <= 3.6 * U and em.max() <= 7.0 * U
    m0, e, em, ee = fm(3, -a)
    assert ee.max() <= 3.6 * U and em.max() <= 5.0 * U
    # beyond the table CUDA's erfc (5 ulp) and exp (an ulp) of the rounded square (y^2 u relative)
    b = np.concatenate([[6.0, np.nextafter(6.0, 7.0)], rng.uniform(6.0, 20.0, 20_000)])
    m0, e, em, ee = fm(3, b)
    assert (ee <= (b * b + 3.0) * U).all() and em.max() <= 11.0 * U
    m0, e, em, ee = fm(3, -b)
    assert (ee <= (b * b + 3.0) * U).all() and em.max() <= 11.0 * U
    m0, e, _, _ = fm(3, np.concatenate([[0.0, -0.0, 40.0, -40.0, np.inf, -np.inf], NANS]))
    assert list(m0[:6]) == [0.5, 0.5, 0.0, 1.0, 0.0, 1.0] and list(e[:6]) == [1.0, 1.0, 0.0, 0.0, 0.0, 0.0]
    assert np.isnan(m0[6:]).all() and np.isnan(e[6:]).all()


def test_comparisons(fm):
    tiny, big = 2.0 ** -1022, np.finfo(np.float64).max
    yes = [2.0 ** -1042, np.nextafter(tiny, 0.0), tiny, 1e-300, 1.0, big, np.inf]
    no = [0.0, -0.0, 5e-324, np.nextafter(2.0 ** -1042, 0.0), -5e-324, -tiny, -1.0, -big, -np.inf, *NANS]
    assert (fm(4, yes)[0] == 1.0).all() and (fm(4, no)[0] == 0.0).all()
    # the smaller of two numbers that are not negative; a NaN of either sign loses on either side, as with fmin
    v = np.array([0.0, 5e-324, tiny, 1e-40, 1.0, np.nextafter(1.0, 2.0), 3.0, big, np.inf])
    x, y = (a.ravel() for a in np.meshgrid(v, v))
    assert np.array_equal(fm(5, x, y)[0], np.minimum(x, y))
    x, y = (a.ravel() for a in np.meshgrid(v, NANS))
    assert np.array_equal(fm(5, x, y)[0], x) and np.array_equal(fm(5, y, x)[0], x)
    x, y = (a.ravel() for a in np.meshgrid(NANS, NANS))
    assert np.isnan(fm(5, x, y)[0]).all()
