"""Device memory of a context as other users of the GPU see it: what it holds beyond a context that has only
ever had its present mesh stays within the 256 MiB that it may keep (csrc/device_pool.h), also after a larger
mesh with the adjoint's arrays and after an upload that fails."""
import numpy as np
import pytest

import meshgen as mg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# the 256 MiB, and 32 MiB for the granularity of the device's allocations (2 MiB; arrays below 1 MiB share one)
KEEP = (256 + 32) << 20


@pytest.fixture(scope="module")
def cg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2402_02075_gb300 as cg
    from paper_2402_02075_gb300 import build
    build.build()
    torch.zeros(1, device="cuda")
    cg.upload_mesh(mg.periodic_box(6), cg.default_params()).close()  # module and context memory
    return cg


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _broken(mesh):
    """a cell given twice: its faces have three cells"""
    m = dict(mesh)
    n = mesh["cell_ptr"][1]
    m["cell_type"] = np.concatenate([mesh["cell_type"], mesh["cell_type"][:1]])
    m["cell_ptr"] = np.concatenate([mesh["cell_ptr"], mesh["cell_ptr"][-1:] + n])
    m["cell_nodes"] = np.concatenate([mesh["cell_nodes"], mesh["cell_nodes"][:n]])
    return m


def test_memory_after_a_larger_mesh_and_after_a_failed_upload(cg):
    prm = cg.default_params(mach=3.0, n_levels=3, compression_factor=0)
    small, large = mg.ramp_box(128, 64, 9), mg.ramp_box(128, 64, 16)
    empty = _free()
    needs = []
    for mesh in (small, large):
        fresh = cg.Context(prm)
        fresh.mesh_upload(mesh)
        needs.append(empty - _free())
        fresh.close()
        assert empty - _free() <= 4 << 20
    need, need_large = needs
    ctx = cg.Context(prm)
    ctx.mesh_upload(large)
    W, G = mg.uniform_state(ctx.nc, mach=3.0)
    ctx.state_init(torch.from_numpy(W).cuda(), torch.from_numpy(G).cuda())
    ctx.linearize()
    assert empty - _free() > 4 * (need + KEEP)  # the adjoint's arrays
    ctx.mesh_upload(large)
    assert empty - _free() <= need_large + KEEP
    ctx.mesh_upload(small)
    assert empty - _free() <= need + KEEP
    for mesh in (large, small):
        ctx.mesh_upload(mesh)
        with pytest.raises(cg.CgksError):
            ctx.mesh_upload(_broken(mesh))
        assert empty - _free() <= KEEP
    ctx.mesh_upload(small)  # and works on
    assert ctx.nc == len(small["cell_type"]) and empty - _free() <= need + KEEP
    ctx.close()
    assert empty - _free() <= 4 << 20
