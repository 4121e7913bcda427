"""The paths that sizes choose between, against the oracle: one and eight threads per coarse cell (levels
above and below a warp of cells per sub-partition), eight and 32 per cell of an LU-SGS colour; and a
context that uploads one mesh after another into the memory of the one before.  Tolerances as in the
other solver tests."""
import numpy as np
import pytest

import meshgen as mg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2402_02075_gb300 as cg
    from paper_2402_02075_gb300 import build
    build.build()
    return cg


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("extra", [dict(), dict(coarse_smoother=1), dict(dt_mode=1)])
def test_vcycle_on_levels_on_both_sides_of_the_lane_rules(cg, orc, extra):
    mesh = mg.periodic_box(34)  # 66 k cells; levels of about 31 k and 18 k, LU-SGS colours of 1 k to 4 k
    W, G = mg.density_wave_state(mesh)
    prm = dict(mach=0.2, n_levels=3, **extra)
    ctx = cg.upload_mesh(mesh, cg.default_params(**prm))
    n = [ctx.level_info(k)[0] for k in (1, 2)]
    assert n[0] > 4 * 32 * 152 > n[1], n
    ctx.state_init(_t(W), _t(G))
    om = orc.Mesh(mesh)
    os_ = orc.Solver(om, orc.params(**prm))
    os_.set_state(W, G)
    np.testing.assert_allclose(ctx.vcycle(1), os_.run(1, multigrid=True), rtol=1e-9)
    Wg, Wo = ctx.state_get()[0].cpu().numpy(), os_.state()[0]
    assert np.abs(Wg - Wo).max() <= 1e-11 * np.abs(Wo).max()
    ctx.close()


def test_uploads_into_the_memory_of_earlier_meshes(cg):
    """Larger, smaller and larger again, with the adjoint's arrays in between: the same bits as fresh
    contexts."""
    makers = [lambda: mg.periodic_box(8), lambda: mg.pyramid_box(6), lambda: mg.ramp_box(24, 12, 8, n_prism=3),
              lambda: mg.periodic_box(8)]
    prm = dict(mach=0.5, n_levels=3, compression_factor=0)
    kept = cg.Context(cg.default_params(**prm))
    rng = np.random.default_rng(3)
    for mk in makers:
        mesh = mk()
        n = len(mesh["cell_type"])
        W, G = mg.uniform_state(n, mach=0.5)
        W = W * (1.0 + 0.01 * rng.standard_normal(W.shape))
        w = rng.standard_normal((20, n))
        outs = []
        for ctx in (kept, cg.Context(cg.default_params(**prm))):
            ctx.mesh_upload(mesh)
            ctx.state_init(_t(W), _t(G))
            ctx.linearize()
            got = [*ctx.residual_vjp(_t(w[:5]), _t(w[5:]))]
            h = ctx.vcycle(2)
            got += [*ctx.state_get(), torch.from_numpy(h), ctx.coarse_map(1), ctx.level_geometry(2)["Sn"]]
            outs.append([x.cpu().numpy() for x in got])
        for a, b in zip(*outs):
            assert np.array_equal(a, b)
    kept.close()
