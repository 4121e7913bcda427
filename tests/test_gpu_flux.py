"""The flux kernels' half-space moments on the device at normal velocities over and beyond their table
(normal Mach numbers 0 to 20; the table ends at 7), against the oracle's residual.

Tolerance: as the other parity tests, 1e-11 of the summed flux magnitudes; the compression factor takes
the relative pressure jump, whose rounding grows with the kinetic part of the energy: times 1 + M^2."""
import numpy as np
import pytest

import meshgen as mg
from parity import assert_normwise, grad_scale

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mach", [0.0, 0.7, 6.9, 7.1, 20.0])
@pytest.mark.parametrize("phys", [dict(), dict(viscous=1, reynolds=500.0, prandtl=0.72),
                                  dict(viscous=1, reynolds=500.0, prandtl=1.0, compression_factor=0)])
def test_residual_over_the_table_of_the_half_space_moments(orc, mach, phys):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2402_02075_gb300 as cg
    from paper_2402_02075_gb300 import build
    build.build()
    mesh = mg.periodic_box(6)
    om = orc.Mesh(mesh)
    prm = dict(mach=mach, aoa=(20.0, 10.0), n_levels=1, **phys)
    rng = np.random.default_rng(8)
    amp = 0.02 / (1.0 + mach ** 2)
    W, G = mg.uniform_state(om.nc, mach=mach, aoa=(20.0, 10.0))
    W = W * (1.0 + amp * rng.standard_normal(W.shape))
    G = amp * rng.standard_normal(G.shape)
    ctx = cg.upload_mesh(mesh, cg.default_params(**prm))
    ctx.state_init(torch.from_numpy(W).cuda(), torch.from_numpy(G).cuda())
    os_ = orc.Solver(om, orc.params(**prm))
    os_.set_state(W, G)
    r, ro = ctx.residual(order=3), os_.residual()
    assert_normwise(r["res"].cpu().numpy(), ro["res"], 1e-11, "residual", scale=ro["fscale"])
    assert_normwise(r["grad"].cpu().numpy(), ro["grad"], 1e-11, "gradients", scale=grad_scale(ro["gscale"]))
    assert_normwise(r["alpha"].cpu().numpy()[None], ro["alpha"][None], 1e-11 * (1.0 + mach ** 2), "compression factor")
