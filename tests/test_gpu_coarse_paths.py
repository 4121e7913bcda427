"""Coarse-level paths that sizes and options choose, against the oracle: the forward Euler step with one and
with eight threads per cell in both precisions, the FP32 directional derivative's sums, and cycles without
coarse steps.

The mixed cycle's first step of a level takes the restricted defect alone, which is what the FP64 cycle's
residual and forcing add up to there: with one step on one coarse level, and with none, the two cycles are
the same up to rounding, and are compared within the tolerance of the other solver tests.  With more steps
the bounds are those of the mixed cycle's own tests (the operators differ at second order)."""
import numpy as np
import pytest

import meshgen as mg
from parity import assert_normwise
from test_gpu_mixed import _flux_scale

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LINE = 96 * 152  # cells: one thread per cell above, eight below


@pytest.fixture(scope="module")
def cg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2402_02075_gb300 as cg
    from paper_2402_02075_gb300 import build
    build.build()
    return cg


@pytest.fixture(scope="module")
def box(orc):
    mesh = mg.periodic_box(28)
    return mesh, orc.Mesh(mesh), *mg.density_wave_state(mesh)


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _cycle(cg, orc, box, n, opts, **prm):
    """(W of the library, W of the oracle's FP64 cycle, the start), the levels' cells"""
    mesh, om, W, G = box
    prm = dict(mach=0.2, **prm)
    ctx = cg.upload_mesh(mesh, cg.default_params(**prm, **opts))
    levels = [ctx.level_info(k)[0] for k in range(1, prm["n_levels"])]
    ctx.state_init(_t(W), _t(G))
    h = ctx.vcycle(n)
    Wg = ctx.state_get()[0].cpu().numpy()
    ctx.close()
    os_ = orc.Solver(om, orc.params(**prm))
    os_.set_state(W, G)
    ho = os_.run(n, multigrid=True)
    np.testing.assert_allclose(h[0], ho[0], rtol=1e-9)
    return Wg, os_.state()[0], W, levels


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("levels,steps,post", [(2, 1, 0), (3, 0, 0), (3, 0, 1)])
def test_cycles_that_both_precisions_share(cg, orc, box, precision, levels, steps, post):
    Wg, Wo, W, n = _cycle(cg, orc, box, 1, dict(precision=precision), n_levels=levels, coarse_steps=steps, post=post)
    assert n[0] > LINE and (levels == 2 or n[1] < LINE), n
    assert np.abs(Wg - Wo).max() <= 1e-11 * np.abs(Wo).max()


@pytest.mark.parametrize("precision", [0, 1])
def test_cycle_with_more_steps(cg, orc, box, precision):
    Wg, Wo, W, n = _cycle(cg, orc, box, 2, dict(precision=precision), n_levels=3, coarse_steps=2, post=1)
    assert n[0] > LINE > n[1], n
    change = np.abs(Wo - W).max()
    assert np.abs(Wg - Wo).max() <= (0.05 * change if precision else 1e-11 * np.abs(Wo).max())


def test_directional_derivative_with_one_thread_per_cell(cg, orc):
    mesh = mg.periodic_box(34)
    prm = dict(mach=0.6, n_levels=2)
    ctx = cg.upload_mesh(mesh, cg.default_params(precision=1, **prm))
    os_ = orc.Solver(orc.Mesh(mesh), orc.params(**prm))
    rng = np.random.default_rng(5)
    n = ctx.level_info(1)[0]
    assert n > 128 * 152, n
    W0, _ = mg.uniform_state(n, mach=0.6)
    W0 = W0 * (1 + 0.03 * rng.standard_normal(W0.shape))
    sw = np.abs(W0).max(axis=1)
    sw[1:4] = sw[1:4].max()
    dW = 0.01 * sw[:, None] * rng.standard_normal(W0.shape)
    h = 1e-4
    got = ctx.kfvs_jvp(1, _t(W0), _t(dW)).cpu().numpy()
    ref = (os_.kfvs_residual(1, W0 + h * dW) - os_.kfvs_residual(1, W0 - h * dW)) / (2 * h)
    rel = (np.abs(dW) / sw[:, None]).max()
    assert_normwise(got, ref, 1e-5, "KFVS JVP", scale=_flux_scale(os_.level(1), W0) * rel)
    ctx.close()
