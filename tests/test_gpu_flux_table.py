"""The flux at the end of its table of half-space moments, |U_n| sqrt(rho / 2p) = 6: a flow along a mesh
direction, just inside the table and across its end, against the oracle's residual.

Tolerance: as the other parity tests, 1e-11 of the summed flux magnitudes; the compression factor takes
the relative pressure jump, whose rounding grows with the kinetic part of the energy: times 1 + M^2."""
import numpy as np
import pytest

import meshgen as mg
from parity import assert_normwise, grad_scale

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mach,inside", [(6.95, True), (7.17, False)])
@pytest.mark.parametrize("phys", [dict(), dict(viscous=1, reynolds=500.0, prandtl=0.72),
                                  dict(viscous=1, reynolds=500.0, prandtl=1.0, compression_factor=0)])
def test_residual_at_the_end_of_the_table(orc, mach, inside, phys):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2402_02075_gb300 as cg
    from paper_2402_02075_gb300 import build
    build.build()
    om = orc.Mesh(mg.periodic_box(6))
    prm = dict(mach=mach, n_levels=1, **phys)
    rng = np.random.default_rng(8)
    amp = 0.02 / (1.0 + mach ** 2)
    W, G = mg.uniform_state(om.nc, mach=mach)
    W = W * (1.0 + amp * rng.standard_normal(W.shape))
    G = amp * rng.standard_normal(G.shape)
    ctx = cg.upload_mesh(mg.periodic_box(6), cg.default_params(**prm))
    ctx.state_init(torch.from_numpy(W).cuda(), torch.from_numpy(G).cuda())
    os_ = orc.Solver(om, orc.params(**prm))
    os_.set_state(W, G)
    # the argument at the faces, from their cells' averages (the points' differ by the amplitude)
    g = {k: v.cpu().numpy() for k, v in ctx.level_geometry(0).items()}
    n = g["Sn"] / np.linalg.norm(g["Sn"], axis=0)
    y = []
    for side in (g["fL"], g["fR"]):
        w = W[:, side]
        p = 0.4 * (w[4] - 0.5 * (w[1] ** 2 + w[2] ** 2 + w[3] ** 2) / w[0])
        y.append(np.abs((w[1:4] * n).sum(axis=0)) / w[0] * np.sqrt(0.5 * w[0] / p))
    y = np.concatenate(y)
    if inside:
        assert 5.9 < y.max() < 5.99, y.max()
    else:
        assert (y > 6.01).sum() > 50 and ((y > 5.0) & (y < 5.99)).sum() > 50, y.max()
    r, ro = ctx.residual(order=3), os_.residual()
    assert_normwise(r["res"].cpu().numpy(), ro["res"], 1e-11, "residual", scale=ro["fscale"])
    assert_normwise(r["grad"].cpu().numpy(), ro["grad"], 1e-11, "gradients", scale=grad_scale(ro["gscale"]))
    assert_normwise(r["alpha"].cpu().numpy()[None], ro["alpha"][None], 1e-11 * (1.0 + mach ** 2), "compression factor")
    ctx.close()
