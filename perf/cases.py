"""The work that a user of the library has it do, as cases to be timed and compared.

Each case is one call sequence through the public binding (paper_2402_02075_gb300.Context) on a
synthetic mixed-element mesh: residuals, explicit steps, V-cycles in the three coarse smoothers, a
steady solve, the adjoint's linearisation and transposed product, a mesh upload.  Meshes are boxes
split into hexahedra, prisms, Kuhn tetrahedra and pyramids (the layouts of the tests and the
benchmark); states are a free stream with smooth perturbations and a little noise, with the matching
gradients.  `exact` evaluates the same scheme in plain 64-bit torch: Householder least squares,
full monomial moments of the Maxwellians, automatic differentiation for the transposed products.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2402_02075_gb300 as cg

F64 = torch.float64


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


# ---- the cases -----------------------------------------------------------------------------------

VISCOUS = dict(mach=0.5, viscous=1, reynolds=1e4, prandtl=0.72)


def listed():
    return [
        # a residual evaluation inside a user's own time integrator, all four split kinds, periodic
        dict(name="residual-periodic", call="residual", mesh="periodic", nx=16, ny=16, nz=16, mach=0.2),
        # a residual evaluation on a million cells (viscous, temperature-dependent viscosity)
        dict(name="residual-million", call="residual", mesh="scale", nx=84, ny=84, nz=84, sutherland=0.383, **VISCOUS),
        # single-grid steps on the smallest ramp that the convergence runs use: launches and latency
        dict(name="steps-ramp-small", call="step", count=10, mesh="ramp", nx=32, ny=16, nz=2, mach=3.0),
        # one single-grid step on a slab of the benchmark's boundary layer
        dict(name="step-slab", call="step", count=1, mesh="wall", nx=96, ny=4, nz=69, **VISCOUS),
        # one V-cycle on the smallest boundary layer: the smallest call of the multigrid path
        dict(name="vcycle-smallest", call="vcycle", count=1, mesh="wall", nx=12, ny=2, nz=12, precision=0, smoother=0,
             **VISCOUS),
        # the benchmark's step: one FP64 V-cycle on the 1.5 million cell boundary layer
        dict(name="vcycle-boundary-layer", call="vcycle", count=1, mesh="wall", nx=96, ny=64, nz=69, precision=0,
             smoother=0, **VISCOUS),
        # mixed-precision V-cycles on the slab that is driven to convergence
        dict(name="vcycle-mixed-slab", call="vcycle", count=2, mesh="wall", nx=96, ny=4, nz=69, precision=1, smoother=0,
             **VISCOUS),
        # V-cycles with the implicit coarse smoother on the supersonic ramp
        dict(name="vcycle-lusgs-ramp", call="vcycle", count=2, mesh="ramp", nx=64, ny=32, nz=8, precision=0, smoother=1,
             mach=3.0),
        # a stretch of the steady solve on a boundary layer
        dict(name="steady-boundary-layer", call="steady", count=50, mesh="wall", nx=24, ny=4, nz=24, precision=0,
             smoother=0, **VISCOUS),
        # forming the adjoint's linearisation and one product with it (a new design point)
        dict(name="linearize-ramp", call="linearize", recompute=0, mesh="ramp", nx=64, ny=32, nz=8, mach=3.0),
        # the transposed product that the adjoint solve repeats thousands of times
        dict(name="product-ramp", call="product", recompute=0, mesh="ramp", nx=128, ny=64, nz=16, mach=3.0),
        # uploading a mesh: faces, operators and the coarse levels (each design point of a shape study)
        dict(name="upload-box", call="upload", mesh="scale", nx=40, ny=40, nz=40, mach=0.5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["residual", "residual", "step", "vcycle", "vcycle", "vcycle", "steady", "linearize", "product",
                       "upload"])
    most = dict(residual=250_000, step=250_000, vcycle=200_000, steady=3_000, linearize=12_000, product=60_000,
                upload=60_000)[call]
    if call in ("linearize", "product"):
        mesh = rng.choice(["ramp", "ramp", "periodic", "pyramid"])
    elif call in ("step", "vcycle", "steady"):
        mesh = rng.choice(["wall", "wall", "ramp"])
    else:
        mesh = rng.choice(["periodic", "scale", "ramp", "wall", "pyramid"])
    n = _log_int(rng, 300 if call in ("step", "vcycle", "steady") else 600, most)  # grid cells before the split
    c = dict(call=call, mesh=mesh)
    if mesh in ("periodic", "scale", "pyramid"):
        s = max(6, int(round(n ** (1.0 / 3.0))))
        c.update(nx=s, ny=s, nz=s)
    elif mesh == "wall":
        nz = rng.randint(10, 16) if n < 1000 else rng.randint(20, 32) if n < 20_000 else rng.randint(48, 69)
        ny = rng.randint(2, 5) if n < 50_000 else rng.randint(4, 24)
        c.update(nx=max(8, n // (nz * ny)), ny=ny, nz=nz)
    else:
        nz = rng.randint(2, 4) if n < 5000 else rng.randint(5, 17)
        ny = max(8, int(round(math.sqrt(n / nz / 2.0))))
        c.update(nx=max(10, n // (nz * ny)), ny=ny, nz=nz)
    if mesh == "ramp":
        c.update(mach=3.0)
    elif mesh == "wall" or (mesh == "scale" and call != "upload"):
        c.update(**VISCOUS, sutherland=rng.choice([0.0, 0.383]))
    else:
        c.update(mach=rng.choice([0.2, 0.5]))
    if call in ("step", "vcycle"):
        c["count"] = rng.randint(1, 5) if n < 50_000 else 1
    if call == "steady":
        c["count"] = rng.choice([30, 40, 50])
    if call in ("vcycle", "steady"):
        c["precision"] = rng.choice([0, 0, 1])
        c["smoother"] = 1 if c["precision"] == 0 and n < 10_000 and rng.random() < 0.3 else 0
    if call in ("linearize", "product"):
        c["recompute"] = rng.choice([0, 0, 1])
    return c


def _params(case):
    adjoint = case["call"] in ("linearize", "product")
    p = dict(mach=case["mach"], viscous=case.get("viscous", 0), sutherland=case.get("sutherland", 0.0),
             precision=case.get("precision", 0), coarse_smoother=case.get("smoother", 0),
             compression_factor=0 if adjoint else 1, adjoint_recompute=case.get("recompute", 0),
             n_levels=1 if adjoint or case["call"] in ("residual", "step") else 3)
    if p["viscous"]:
        p.update(reynolds=case["reynolds"], prandtl=case["prandtl"])
    return p


def prepare(case, seed):
    call = case["call"]
    m = _mesh(case["mesh"], case["nx"], case["ny"], case["nz"], _scale(call, seed))
    ctx = cg.Context(cg.default_params(**_params(case)))
    state = dict(case=dict(case), ctx=ctx)
    if call == "upload":
        state["mesh"] = m["host"]
        return state
    ctx.mesh_upload(m["host"])
    state["W"], state["G"] = _state(case, seed)
    if call in ("linearize", "product"):
        state["rbar"], state["gbar"] = _cotangents(case, seed)
    if call == "product":
        ctx.state_init(state["W"], state["G"])
        ctx.linearize()
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    call = case["call"]
    if call == "upload":
        ctx.mesh_upload(state["mesh"])
        out = dict(levels=[list(ctx.level_info(k)) for k in range(3)], m2=ctx.fine_moments())
        out["geometry"] = [ctx.level_geometry(k) for k in range(3)]
        out["maps"] = [ctx.coarse_map(k) for k in (1, 2)]
        return out
    if call == "product":
        return ctx.residual_vjp(state["rbar"], state["gbar"])
    ctx.state_init(state["W"], state["G"])
    if call == "residual":
        return ctx.residual(order=3)
    if call == "linearize":
        ctx.linearize()
        return ctx.residual_vjp(state["rbar"], state["gbar"])
    if call == "step":
        h = ctx.step(case["count"])
    elif call == "vcycle":
        h = ctx.vcycle(case["count"])
    else:
        r = ctx.steady_solve(multigrid=True, drop=1e-12, max_iters=case["count"], raise_on_notconv=False)
        h = np.array([r["drop"], float(r["iters"])])
    return [h, *ctx.state_get()]


def work(case):
    """Compulsory traffic (state, operators and outputs once per evaluation) and the operations of the
    scheme: about 1,500 per Gauss point of a full flux, 12 per entry of a cell's 9 x 4 N_f operator,
    160 per face of a first-order coarse flux."""
    m = _mesh(case["mesh"], case["nx"], case["ny"], case["nz"])
    nc, links, sides = m["nc"], m["n_links"], m["gp_sides"]
    points = (sides + m["gp_boundary"]) // 2
    faces = links // 2
    fine_bytes = nc * (42.0 * 8) + links * 36.0 * 8 + points * 24.0
    fine_flops = points * 1500.0 + links * 36.0 * 12.0 + nc * 600.0
    call, count = case["call"], case.get("count", 1)
    if call == "upload":
        return dict(bytes=nc * 400.0 + links * 350.0, flops=links * 4000.0)
    if call in ("residual", "step"):
        return dict(bytes=count * fine_bytes, flops=count * fine_flops)
    if call in ("vcycle", "steady"):
        return dict(bytes=count * (2 * fine_bytes + faces * 4 * 120.0), flops=count * (2 * fine_flops + faces * 4 * 160.0))
    product = points * 410.0 * 8 + (0 if case["recompute"] else (nc * 1020.0 + links * 200.0) * 8) + nc * 320.0
    if call == "product":
        return dict(bytes=product, flops=product / 4)
    return dict(bytes=2 * product + fine_bytes, flops=points * 30 * 700.0 + points * 11 * 3000.0 + product / 4)


# ---- inputs --------------------------------------------------------------------------------------

HEX, PRZ, PRX, TET, PYR = range(5)
# corners of a grid cell as (i, j, k) bits, in the order of a hexahedron's nodes
CORNERS = [(0, 0, 0), (1, 0, 0), (1, 1, 0), (0, 1, 0), (0, 0, 1), (1, 0, 1), (1, 1, 1), (0, 1, 1)]
# the cells of a split grid cell: nodes as corner numbers (8: the node mean of a pyramid split)
SPLITS = {HEX: [[0, 1, 2, 3, 4, 5, 6, 7]],
          PRZ: [[0, 1, 2, 4, 5, 6], [0, 2, 3, 4, 6, 7]],
          PRX: [[0, 3, 7, 1, 2, 6], [0, 7, 4, 1, 6, 5]],
          TET: [[0, 1, 2, 6], [0, 5, 1, 6], [0, 2, 3, 6], [0, 3, 7, 6], [0, 4, 5, 6], [0, 7, 4, 6]],
          PYR: [[1, 2, 3, 0, 8], [7, 6, 5, 4, 8], [4, 5, 1, 0, 8], [5, 6, 2, 1, 8], [6, 7, 3, 2, 8], [7, 4, 0, 3, 8]]}
TYPE_OF = {4: 4, 6: 5, 8: 6, 5: 7}  # number of nodes -> cell type of the interface
# outward faces of each cell type
FACES = {4: [[0, 2, 1], [0, 1, 3], [1, 2, 3], [0, 3, 2]],
         5: [[0, 2, 1], [3, 4, 5], [0, 1, 4, 3], [1, 2, 5, 4], [2, 0, 3, 5]],
         6: [[0, 3, 2, 1], [4, 5, 6, 7], [0, 1, 5, 4], [1, 2, 6, 5], [2, 3, 7, 6], [3, 0, 4, 7]],
         7: [[0, 3, 2, 1], [0, 1, 4], [1, 2, 4], [2, 3, 4], [3, 0, 4]]}


def _layout(mesh, nx, ny, nz):
    """(grid lines, split kind per grid cell (i, j, k), periodic axes, tag per side, jitter, mapping)"""
    x, y, z = (np.linspace(0.0, 1.0, n + 1) for n in (nx, ny, nz))
    i, j, k = np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij")
    quadrant = np.where(i < (3 * nx) // 4, np.where(k < (3 * nx) // 4, HEX, PRX), np.where(k < (3 * nx) // 4, PRZ, TET))
    if mesh == "periodic":
        return (x, y, z), quadrant, (True, True, True), {}, 0.05, None
    if mesh == "scale":
        return (x, y, z), quadrant, (False, True, False), {0: 3, 1: 3, 4: 2, 5: 3}, 0.05, None
    if mesh == "pyramid":
        lo, hi = nx // 3, nx - nx // 3
        inside = (i >= lo) & (i < hi) & (j >= lo) & (j < hi) & (k >= lo) & (k < hi)
        return (x, y, z), np.where(inside, PYR, HEX), (True, True, True), {}, 0.05, None
    if mesh == "wall":  # prisms while the wall-normal spacing is below half of dx, tetrahedra up to twice
        first, ratio = (2e-3, 1.3) if nz < 18 else (1e-3, 1.2) if nz < 40 else (1e-4, 1.1)
        dz = np.minimum(first * ratio ** np.arange(nz), 2.0 / nx)
        prisms = int(np.argmax(dz >= 0.5 / nx)) if (dz >= 0.5 / nx).any() else nz
        z = np.concatenate([[0.0], np.cumsum(dz)])
        return (x, np.arange(ny + 1) / nx, z), np.where(k < prisms, PRZ, TET), (False, True, False), \
            {0: 3, 1: 5, 4: 2, 5: 3}, 0.0, None
    # compression ramp: 15 degrees from x = 0
    t = math.tan(math.radians(15.0))
    layers = max(1, ny // 8)
    return (np.linspace(-0.5, 1.5, nx + 1), y, np.arange(nz + 1) * (2.0 / nx)), np.where(j < layers, PRZ, HEX), \
        (False, False, True), {0: 4, 1: 5, 2: 1, 3: 5}, 0.0, lambda p: p[:, 1] + p[:, 0].clamp(min=0.0) * t


@functools.lru_cache(maxsize=6)
def _mesh(mesh, nx, ny, nz, scale=1.0):
    """Host arrays of cgks_mesh_upload, the face topology that `exact` uses, and sizes.  Cells are
    numbered by grid cell with i running fastest."""
    lines, kind, periodic, tags, jitter, mapping = _layout(mesh, nx, ny, nz)
    d_, dims = _dev(), (nx, ny, nz)

    def grid(n):  # (i, j, k) of every node or grid cell, i running fastest
        k, j, i = torch.meshgrid(*(torch.arange(m, device=d_) for m in reversed(n)), indexing="ij")
        return torch.stack([i.reshape(-1), j.reshape(-1), k.reshape(-1)], 1)

    def node(i, j, k):
        return i + (nx + 1) * (j + (ny + 1) * k)
    lines = [torch.from_numpy(np.asarray(a)).to(d_) for a in lines]
    size = torch.tensor(dims, device=d_)
    ijk = grid([n + 1 for n in dims])
    xyz = torch.stack([lines[d][ijk[:, d]] for d in range(3)], 1)
    wrapped = torch.where(torch.tensor(periodic, device=d_) & (ijk == size), 0, ijk)
    wid = node(*wrapped.unbind(1))
    if jitter:
        r = torch.from_numpy(np.random.default_rng(2402).uniform(-jitter, jitter, xyz.shape)).to(d_)[wid] / size
        free = torch.tensor(periodic, device=d_) | ((ijk > 0) & (ijk < size))
        if mesh == "scale":
            free &= ijk[:, 2:] > 1
        xyz += torch.where(free, r, 0.0)
    if mapping is not None:
        xyz[:, 1] = mapping(xyz)
    xyz = scale * xyz
    g = grid(dims)
    kind = torch.from_numpy(np.ascontiguousarray(kind.transpose(2, 1, 0))).to(d_).reshape(-1)
    corner = torch.stack([node(g[:, 0] + a, g[:, 1] + b, g[:, 2] + c) for a, b, c in CORNERS], 1)
    pyr = torch.nonzero(kind == PYR)[:, 0]
    apex = torch.zeros_like(kind)
    apex[pyr] = len(xyz) + torch.arange(len(pyr), device=d_)
    xyz = torch.cat([xyz, xyz[corner[pyr]].mean(1)])
    wid = torch.cat([wid, apex[pyr]])
    ijk = torch.cat([ijk, torch.full((len(pyr), 3), -1, device=d_)])
    corner = torch.cat([corner, apex[:, None]], 1)
    parts = torch.tensor([len(SPLITS[q]) for q in range(5)], device=d_)[kind]
    first = torch.cumsum(parts, 0) - parts
    nc = int(parts.sum())
    ctype, nodes = torch.empty(nc, dtype=torch.int8, device=d_), torch.full((nc, 8), -1, device=d_)
    for q, subs in SPLITS.items():
        sel = torch.nonzero(kind == q)[:, 0]
        for s, nd in enumerate(subs):
            ctype[first[sel] + s] = TYPE_OF[len(nd)]
            nodes[first[sel] + s, :len(nd)] = corner[sel][:, nd]
    # the faces of every cell, slot by slot: node ids (-1 for the fourth of a triangle)
    fn = torch.full((nc, 6, 4), -1, device=d_)
    for t, faces in FACES.items():
        sel = torch.nonzero(ctype == t)[:, 0]
        for s, f in enumerate(faces):
            fn[sel, s, :len(f)] = nodes[sel][:, f]
    cell, slot = torch.nonzero(fn[:, :, 0] >= 0, as_tuple=True)
    flat = fn[cell, slot]
    big = 1 << 20

    def face_key(f, ids=None):  # the three smallest node ids name a face
        v = torch.where(f < 0, big, f if ids is None else ids[f.clamp(min=0)]).sort(1).values
        return (v[:, 0] * big + v[:, 1]) * big + v[:, 2]
    key = face_key(flat)
    order = torch.argsort(key, stable=True)
    same = key[order][1:] == key[order][:-1]
    mate = torch.full_like(key, -1)
    mate[order[:-1][same]], mate[order[1:][same]] = order[1:][same], order[:-1][same]
    bnd = torch.nonzero(mate < 0)[:, 0]
    tag = torch.full_like(key, -1)
    at = ijk[torch.where(flat[bnd] < 0, flat[bnd][:, :1], flat[bnd])]
    for d in range(3):
        for hi in (0, 1):
            on = (at[:, :, d] == (dims[d] if hi else 0)).all(1)
            tag[bnd[on]] = 100 + 2 * d + hi if periodic[d] else tags[2 * d + hi]
    # periodic partners: the same wrapped nodes on the opposite side
    pairs, shift = [torch.zeros(0, 2, dtype=torch.long, device=d_)], torch.zeros(len(key), 3, dtype=F64, device=d_)
    for d in range(3):
        if periodic[d]:
            lo, hi = (bnd[tag[bnd] == 100 + 2 * d + s] for s in (0, 1))
            lo, hi = (b[torch.argsort(face_key(flat[b], wid))] for b in (lo, hi))
            mate[lo], mate[hi] = hi, lo
            length = scale * (lines[d][-1] - lines[d][0])
            shift[lo, d], shift[hi, d] = -length, length
            pairs.append(torch.stack([lo, hi], 1))
    number = torch.full_like(key, -1)
    number[bnd] = torch.arange(len(bnd), device=d_)
    nn, nv = (nodes >= 0).sum(1), (flat >= 0).sum(1)

    def offsets(n):
        return torch.cat([torch.zeros(1, dtype=torch.long, device=d_), torch.cumsum(n, 0)])
    host = dict(xyz=xyz, cell_type=ctype, cell_ptr=offsets(nn), cell_nodes=nodes[nodes >= 0].int(),
                bface_ptr=offsets(nv[bnd]), bface_nodes=flat[bnd][flat[bnd] >= 0].int(), bface_tag=tag[bnd].int(),
                periodic_pairs=number[torch.cat(pairs)].int())
    host = {k: np.ascontiguousarray(v.cpu().numpy()) for k, v in host.items()}
    centre = torch.where((nodes >= 0)[:, :, None], xyz[nodes.clamp(min=0)], 0.0).sum(1) / nn[:, None]
    topo = dict(xyz=xyz, nodes=nodes, ctype=ctype, cell=cell, slot=slot, flat=flat, mate=mate, tag=tag, shift=shift)
    return dict(host=host, topo=topo, centre=centre, nc=nc, n_links=len(key), gp_sides=int(nv.sum()),
                gp_boundary=int(nv[mate < 0].sum()))


def _scale(call, seed):
    """An uploaded mesh is the box in a size of its own: other coordinates, the same coarse cells."""
    return 1.0 + 0.001 * (seed % 997) if call == "upload" else 1.0


def _free_stream(mach):
    return [1.0, mach, 0.0, 0.0, 1.0 / 1.4 / 0.4 + 0.5 * mach * mach]


def _state(case, seed):
    """Free stream times (1 + smooth waves + noise) and the waves' gradient (with noise)."""
    m = _mesh(case["mesh"], case["nx"], case["ny"], case["nz"])
    d = _dev()
    g = torch.Generator(device=d)
    g.manual_seed(int(seed))
    x = m["centre"].T
    amp = 0.01 if case["mach"] < 1.0 else 0.002
    W0 = torch.tensor(_free_stream(case["mach"]), dtype=F64, device=d)
    scale = W0.abs()
    scale[2:4] = scale[1]
    W, G = W0[:, None].repeat(1, m["nc"]), torch.zeros(5, 3, m["nc"], dtype=F64, device=d)
    k = 2.0 * math.pi * torch.randint(1, 3, (5, 3, 3), generator=g, device=d).to(F64)
    phase = 2.0 * math.pi * torch.rand(5, 3, generator=g, device=d, dtype=F64)
    for q in range(5):
        for s in range(3):
            a = k[q, s] @ x + phase[q, s]
            W[q] += amp / 3.0 * scale[q] * torch.sin(a)
            G[q] += amp / 3.0 * scale[q] * torch.cos(a) * k[q, s][:, None]
    W += 0.02 * amp * scale[:, None] * torch.randn(W.shape, generator=g, device=d, dtype=F64)
    G += 0.02 * amp * scale[:, None, None] * torch.randn(G.shape, generator=g, device=d, dtype=F64)
    return W.contiguous(), G.reshape(15, -1).contiguous()


def _cotangents(case, seed):
    d = _dev()
    n = _mesh(case["mesh"], case["nx"], case["ny"], case["nz"])["nc"]
    g = torch.Generator(device=d)
    g.manual_seed(int(seed) + 1)
    return (torch.randn(5, n, generator=g, device=d, dtype=F64), torch.randn(15, n, generator=g, device=d, dtype=F64))


# ---- the scheme in plain 64-bit torch ------------------------------------------------------------

def exact(case, seed):
    call = case["call"]
    if call in ("vcycle", "steady"):
        return None  # agglomeration is a sequential pass: minutes in plain Python on these meshes
    m = _mesh(case["mesh"], case["nx"], case["ny"], case["nz"], _scale(call, seed))
    geo = _Geometry(m)
    if call == "upload":
        return dict(levels=None, m2=geo.m2.T.contiguous(), maps=None,
                    geometry=[dict(vol=geo.vol, ctr=geo.ctr.T.contiguous()), None, None])
    p = _params(case)
    geo.operators()
    W, G = _state(case, seed)
    alpha = torch.ones(m["nc"], dtype=F64, device=W.device)
    if call == "residual":
        r = _residual(geo, p, W, G, alpha)
        return dict(r, norm=float(((r["res"][0] / geo.vol) ** 2).mean().sqrt()))
    if call == "step":
        h = []
        for _ in range(case["count"]):
            r = _residual(geo, p, W, G, alpha)
            h.append(float(((r["res"][0] / geo.vol) ** 2).mean().sqrt()))
            W, G, alpha = W + r["dt"] / geo.vol * r["res"], r["grad"], r["alpha"]
        return [np.array(h), W, G, alpha]
    rbar, gbar = _cotangents(case, seed)
    W.requires_grad_(True)
    G.requires_grad_(True)
    r = _residual(geo, p, W, G, alpha)
    return torch.autograd.grad((r["res"] * rbar).sum() + (r["grad"] * gbar).sum(), (W, G))


class _Geometry:
    """Gauss points, volume moments and reconstruction operators of a mesh."""

    def __init__(self, m):
        t, self.nc = m["topo"], m["nc"]
        self.t = t
        self.moments()
        # one record per face: the side with the lower cell is the left one
        cell, mate = t["cell"], t["mate"]
        link = torch.arange(len(cell), device=cell.device)
        left = (mate < 0) | (cell < cell[mate.clamp(min=0)]) | ((cell == cell[mate.clamp(min=0)]) & (link < mate))
        self.face = link[left]                                # its link in the left cell
        self.L, self.R = cell[self.face], torch.where(mate[self.face] < 0, -1, cell[mate[self.face].clamp(min=0)])
        self.tag, self.shift = t["tag"][self.face], t["shift"][self.face]
        self.points()

    def moments(self):
        t, nc = self.t, self.nc
        X = t["xyz"][t["nodes"].clamp(min=0)]
        q = math.sqrt(0.6)
        gp = [(s, w) for s, w in ((-q, 5 / 9), (0.0, 8 / 9), (q, 5 / 9))]
        xs, ws = [], []
        hexa, tet, pri = ((t["ctype"] == 6) | (t["ctype"] == 7)), t["ctype"] == 4, t["ctype"] == 5
        Xh = X.clone()
        Xh[t["ctype"] == 7, 5:] = X[t["ctype"] == 7, 4:5]     # a pyramid: the top face collapsed onto the apex
        for a, wa in gp:
            for b, wb in gp:
                for c, wc in gp:
                    N, D = torch.zeros(nc, 8, dtype=F64, device=X.device), torch.zeros(nc, 8, 3, dtype=F64, device=X.device)
                    jac = torch.zeros(nc, dtype=F64, device=X.device)
                    for n, (i, j, k) in enumerate(CORNERS):
                        f = [(1 + (2 * s - 1) * v) / 2 for s, v in ((i, a), (j, b), (k, c))]
                        g = [(2 * s - 1) / 2 for s in (i, j, k)]
                        N[hexa, n] = f[0] * f[1] * f[2]
                        for d, v in enumerate((g[0] * f[1] * f[2], f[0] * g[1] * f[2], f[0] * f[1] * g[2])):
                            D[hexa, n, d] = v
                    jac[hexa] = 1.0
                    u, v, w = (1 + a) / 2, (1 + b) / 2, (1 + c) / 2
                    r, s = u, v * (1 - u)
                    for n, (f, g) in enumerate(((1 - r - s, (-1, -1)), (r, (1, 0)), (s, (0, 1)))):
                        for top in (0, 1):
                            h = (1 + c) / 2 if top else (1 - c) / 2
                            N[pri, n + 3 * top] = f * h
                            for d, val in enumerate((g[0] * h, g[1] * h, f * (0.5 if top else -0.5))):
                                D[pri, n + 3 * top, d] = val
                    jac[pri] = (1 - u) / 4
                    tt = w * (1 - u) * (1 - v)
                    for n, (f, g) in enumerate(((1 - r - s - tt, (-1, -1, -1)), (r, (1, 0, 0)), (s, (0, 1, 0)), (tt, (0, 0, 1)))):
                        N[tet, n] = f
                        for d in range(3):
                            D[tet, n, d] = g[d]
                    jac[tet] = (1 - u) ** 2 * (1 - v) / 8
                    Y = torch.where((hexa[:, None, None]), Xh, X)
                    xs.append(torch.einsum("cn,cnd->cd", N, Y))
                    ws.append(wa * wb * wc * jac * torch.linalg.det(torch.einsum("cnk,cnd->ckd", D, Y)))
        x, w = torch.stack(xs), torch.stack(ws)
        self.vol = w.sum(0)
        self.ctr = (w[:, :, None] * x).sum(0) / self.vol[:, None]
        y = x - self.ctr
        pair = ((0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2))
        self.m2 = torch.stack([(w * y[..., a] * y[..., b]).sum(0) for a, b in pair], 1) / self.vol[:, None]

    def points(self):
        """Gauss points of every face (3 or 4), their area vectors outward of the left cell."""
        nodes = self.t["flat"][self.face]
        P = self.t["xyz"][nodes.clamp(min=0)]
        tri = nodes[:, 3] < 0
        g = 1.0 / math.sqrt(3.0)
        xs, As = [], []
        area3 = torch.linalg.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]) / 6.0
        for k, (s, t) in enumerate(((-g, -g), (g, -g), (g, g), (-g, g))):
            N = [(1 - s) * (1 - t) / 4, (1 + s) * (1 - t) / 4, (1 + s) * (1 + t) / 4, (1 - s) * (1 + t) / 4]
            ds = ((1 - t) * (P[:, 1] - P[:, 0]) + (1 + t) * (P[:, 2] - P[:, 3])) / 4
            dt = ((1 - s) * (P[:, 3] - P[:, 0]) + (1 + s) * (P[:, 2] - P[:, 1])) / 4
            x4 = sum(N[i] * P[:, i] for i in range(4))
            x3 = (4.0 * P[:, k % 3] + P[:, (k + 1) % 3] + P[:, (k + 2) % 3]) / 6.0
            xs.append(torch.where(tri[:, None], x3, x4))
            As.append(torch.where(tri[:, None], area3, torch.linalg.cross(ds, dt)))
        x, A = torch.stack(xs, 1), torch.stack(As, 1)
        live = torch.ones(len(P), 4, dtype=torch.bool, device=P.device)
        live[:, 3] = ~tri
        size = torch.where(live, A.norm(dim=2), 0.0)
        self.area = size.sum(1)
        self.S = torch.where(live[:, :, None], A, 0.0).sum(1)
        self.fctr = (size[:, :, None] * x).sum(1) / self.area[:, None]
        self.pf = torch.nonzero(live)[:, 0]                   # face of every point
        self.px, self.pA = x[live], A[live]

    def operators(self):
        """Stencils and the least-squares maps of every cell, by number of faces."""
        t, nc = self.t, self.nc
        face_of = torch.empty(len(t["cell"]), dtype=torch.long, device=self.vol.device)
        face_of[self.face] = torch.arange(len(self.face), device=face_of.device)
        inner = self.R >= 0
        face_of[t["mate"][self.face[inner]]] = torch.nonzero(inner)[:, 0]
        is_left = torch.zeros(len(t["cell"]), dtype=torch.bool, device=face_of.device)
        is_left[self.face] = True
        of = torch.full((nc, 6), -1, dtype=torch.long, device=face_of.device)
        of[t["cell"], t["slot"]] = torch.arange(len(t["cell"]), device=face_of.device)
        self.groups = []
        for nt in (4, 5, 6):
            cells = torch.nonzero((of >= 0).sum(1) == nt)[:, 0]
            if not len(cells):
                continue
            link = of[cells][:, :nt]
            f, left, mate = face_of[link], is_left[link], t["mate"][link]
            bnd = mate < 0
            nb = torch.where(bnd, cells[:, None], t["cell"][mate.clamp(min=0)])
            sg = torch.where(left, 1.0, -1.0).to(F64)
            S = sg[..., None] * self.S[f]
            n = self.S[f] / self.S[f].norm(dim=2, keepdim=True)
            c0 = self.ctr[cells][:, None]
            off = self.ctr[nb] + t["shift"][link] - c0
            off = torch.where(bnd[..., None], -2.0 * ((c0 - self.fctr[f]) * n).sum(2, keepdim=True) * n, off)
            sym = torch.tensor([[0, 3, 5], [3, 1, 4], [5, 4, 2]], device=f.device)
            refl = torch.eye(3, dtype=F64, device=f.device) - 2.0 * n[..., :, None] * n[..., None, :]
            M = self.m2[nb][..., sym]
            M = torch.where(bnd[..., None, None], refl @ M @ refl, M)
            x, y, z = off.unbind(2)
            m0 = self.m2[cells][:, None]
            quad = torch.stack([M[..., a, b] + off[..., a] * off[..., b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2))], 2)
            C = torch.cat([off, quad - m0], 2)                # nt x 9
            o, e = torch.zeros_like(x), torch.ones_like(x)
            B = torch.stack([torch.stack([e, o, o, 2 * x, o, o, y, o, z], 2), torch.stack([o, e, o, o, 2 * y, o, x, z, o], 2),
                             torch.stack([o, o, e, o, o, 2 * z, o, y, x], 2)], 2).reshape(len(cells), 3 * nt, 9)
            Q, Rc = _householder(C.transpose(1, 2))
            Q1, Q2 = Q[:, :, :nt], Q[:, :, nt:]
            A1 = _right_solve(Q1, Rc)
            Kg = Q2 @ _pinv(B @ Q2)
            self.groups.append(dict(cells=cells, f=f, left=left, bnd=bnd, nb=nb, n=n, tag=self.tag[f], S=S,
                                    Sdt=S * (self.area[f] / S.norm(dim=2))[..., None], area=self.area[f],
                                    Kq=A1 - Kg @ (B @ A1), Kg=Kg, lsq=_pinv(off)))


def _householder(A):
    """Q (m x m) and R (n x n) of a batch of m x n matrices."""
    b, m, n = A.shape
    R, Q = A.clone(), torch.eye(m, dtype=F64, device=A.device).repeat(b, 1, 1)
    for k in range(n):
        v = torch.zeros(b, m, dtype=F64, device=A.device)
        v[:, k:] = R[:, k:, k]
        v[:, k] += torch.where(v[:, k] >= 0, 1.0, -1.0) * v.norm(dim=1)
        v = v / v.norm(dim=1, keepdim=True)
        R = R - 2.0 * v[:, :, None] * (v[:, None] @ R)
        Q = Q - 2.0 * (Q @ v[:, :, None]) * v[:, None]
    return Q, R[:, :n]


def _right_solve(Q1, R):
    """X with X R^T = Q1, R upper triangular."""
    n = R.shape[1]
    X = [None] * n
    for k in range(n - 1, -1, -1):
        s = Q1[:, :, k]
        for j in range(k + 1, n):
            s = s - R[:, k, j, None] * X[j]
        X[k] = s / R[:, k, k, None]
    return torch.stack(X, 2)


def _pinv(A):
    """Pseudo-inverse of full-column-rank matrices (R^-1 Q^T)."""
    n = A.shape[2]
    Q, R = _householder(A)
    y, X = Q[:, :, :n].transpose(1, 2), [None] * n
    for k in range(n - 1, -1, -1):
        s = y[:, k]
        for j in range(k + 1, n):
            s = s - R[:, k, j, None] * X[j]
        X[k] = s / R[:, k, k, None]
    return torch.stack(X, 1)


def _viscosity(p, t):
    mu, s = p["mach"] / p["reynolds"], p["sutherland"]
    return mu * torch.ones_like(t) if s == 0.0 else mu * t ** 1.5 * (1.0 + s) / (t + s)


def _ghost(p, tag, n, W, G):
    """Ghost state and gradient behind boundary faces with outward normal n; W [k, 5], G [k, 5, 3]."""
    Wi = torch.tensor(_free_stream(p["mach"]), dtype=F64, device=W.device)
    refl = torch.eye(3, dtype=F64, device=W.device) - 2.0 * n[:, :, None] * n[:, None, :]
    Gr = G @ refl
    one, end = slice(0, 1), slice(4, 5)
    slip = torch.cat([W[:, one], (refl @ W[:, 1:4, None])[..., 0], W[:, end]], 1)
    gslip = torch.cat([Gr[:, one], refl @ Gr[:, 1:4], Gr[:, end]], 1)
    wall = torch.cat([W[:, one], -W[:, 1:4], W[:, end]], 1)
    gwall = torch.cat([Gr[:, one], -Gr[:, 1:4], Gr[:, end]], 1)
    rho, u = W[:, 0], W[:, 1:4] / W[:, :1]
    pr = 0.4 * (W[:, 4] - 0.5 * rho * (u * u).sum(1))
    ui, pi = Wi[1:4], 1.0 / 1.4
    c, ci = torch.sqrt(1.4 * pr / rho), 1.0
    un, uni = (u * n).sum(1), (ui * n).sum(1)
    rp, rm = un + 5.0 * c, uni - 5.0 * ci
    ub, cb = 0.5 * (rp + rm), 0.1 * (rp - rm)
    out = ub > 0
    s = torch.where(out, pr / rho ** 1.4, torch.full_like(pr, pi))
    ut = torch.where(out[:, None], u - un[:, None] * n, ui - uni[:, None] * n)
    rb = (cb * cb / (1.4 * s)) ** 2.5
    v = ut + ub[:, None] * n
    far = torch.cat([rb[:, None], rb[:, None] * v, (rb * cb * cb / 1.4 / 0.4 + 0.5 * rb * (v * v).sum(1))[:, None]], 1)
    far = torch.where((un >= c)[:, None], W, torch.where((un <= -c)[:, None], Wi[None], far))
    k = tag[:, None]
    Wg = torch.where(k == 1, slip, torch.where(k == 2, wall, torch.where(k == 3, far, torch.where(k == 4, Wi[None], W))))
    k = k[..., None]
    zero = torch.zeros_like(G)
    return Wg, torch.where(k == 1, gslip, torch.where(k == 2, gwall, torch.where(k == 5, G, zero)))


def _reconstruct(geo, p, W, G, alpha):
    """Coefficients of 1, X, Y, Z, X^2, Y^2, Z^2, XY, YZ, XZ per cell and variable, and time steps."""
    Wc, Gc = W.T, G.T.reshape(-1, 5, 3)
    coef, step = [], []
    for g in geo.groups:
        cells = g["cells"]
        Q0, V = Wc[cells], geo.vol[cells]
        Qn, Gn = Wc[g["nb"]], Gc[g["nb"]]
        if bool(g["bnd"].any()):
            at = torch.nonzero(g["bnd"])
            gw, gg = _ghost(p, g["tag"][g["bnd"]], g["n"][g["bnd"]], Q0[at[:, 0]], Gc[cells][at[:, 0]])
            Qn = Qn.index_put((at[:, 0], at[:, 1]), gw)
            Gn = Gn.index_put((at[:, 0], at[:, 1]), gg)
        dQ = Qn - Q0[:, None]
        b = g["Kq"] @ dQ + g["Kg"] @ Gn.permute(0, 1, 3, 2).reshape(len(cells), -1, 5)   # 9 x 5
        p1 = alpha[cells, None, None] * torch.einsum("kmd,kmq->kdq", g["S"], Qn + Q0[:, None]) / (2.0 * V[:, None, None])
        ls = g["lsq"] @ dQ
        v23, v43 = V[:, None] ** (2.0 / 3.0), V[:, None] ** (4.0 / 3.0)
        beta1 = torch.minimum(v23 * (p1 ** 2).sum(1), v23 * (ls ** 2).sum(1))
        m2 = geo.m2[cells]
        sym = torch.tensor([[0, 3, 5], [3, 1, 4], [5, 4, 2]], device=W.device)
        M = m2[:, sym]
        H = b[:, 3:][:, sym] * torch.where(torch.eye(3, device=W.device).bool(), 2.0, 1.0)[None, :, :, None]  # k 3 3 q
        first = (b[:, :3] ** 2).sum(1) + torch.einsum("kdaq,kab,kdbq->kq", H, M, H)
        second = 4.0 * (b[:, 3:6] ** 2).sum(1) + (b[:, 6:] ** 2).sum(1)
        beta2 = v23 * first + v43 * second
        den = Q0 ** 2 + beta1 + 1e-40
        t1, t2 = beta1 / den, beta2 / den
        sig = (t2 - t1).abs()
        w1, w2 = (0.5 * (1.0 + (sig / (1e-5 + t)) ** 2) for t in (t1, t2))
        w1, w2 = w1 / (w1 + w2), w2 / (w1 + w2)
        c2, c1 = 2.0 * w2, w1 - w2
        a0 = Q0 - (b[:, 3:] * m2[:, :, None]).sum(1)
        coef.append(torch.cat([(c2 * a0 + c1 * Q0)[:, None], c2[:, None] * b[:, :3] + c1[:, None] * p1, c2[:, None] * b[:, 3:]], 1))
        rho, u = Q0[:, 0], Q0[:, 1:4] / Q0[:, :1]
        pr = 0.4 * (Q0[:, 4] - 0.5 * rho * (u * u).sum(1))
        c = torch.sqrt(1.4 * pr / rho)
        s = torch.einsum("kmd,kd->km", g["Sdt"], u).abs() + g["area"] * c[:, None]
        if p["viscous"]:
            s = s + 2.0 * (_viscosity(p, 1.4 * pr / rho) / rho / V)[:, None] * g["area"] ** 2
        step.append(0.5 * V / s.sum(1))
    order = torch.argsort(torch.cat([g["cells"] for g in geo.groups]))
    return torch.cat(coef)[order], torch.cat(step)[order]


def _evaluate(c, X):
    """Values [k, 5] and gradients [k, 5, 3] of the polynomials c [k, 10, 5] at offsets X [k, 3]."""
    x, y, z = (X[:, d:d + 1] for d in range(3))
    w = c[:, 0] + c[:, 1] * x + c[:, 2] * y + c[:, 3] * z + c[:, 4] * x * x + c[:, 5] * y * y + c[:, 6] * z * z + \
        c[:, 7] * x * y + c[:, 8] * y * z + c[:, 9] * x * z
    g = [c[:, 1] + 2 * c[:, 4] * x + c[:, 7] * y + c[:, 9] * z, c[:, 2] + 2 * c[:, 5] * y + c[:, 7] * x + c[:, 8] * z,
         c[:, 3] + 2 * c[:, 6] * z + c[:, 8] * y + c[:, 9] * x]
    return w, torch.stack(g, 2)


class _Maxwellian:
    """Moments of g / rho: powers of u over u > 0, u < 0 or all u, of v and w, of the internal
    velocity (K = 2 degrees for gamma = 1.4)."""

    def __init__(self, W, side):
        self.rho = W[0]
        self.U = [W[1] / W[0], W[2] / W[0], W[3] / W[0]]
        self.p = 0.4 * (W[4] - 0.5 * (W[1] * self.U[0] + W[2] * self.U[1] + W[3] * self.U[2]))
        h = self.h = self.p / W[0]
        lam = 0.5 / h
        if side:
            m0 = 0.5 * torch.erfc(-side * torch.sqrt(lam) * self.U[0])
            m1 = self.U[0] * m0 + side * 0.5 * torch.exp(-lam * self.U[0] ** 2) / torch.sqrt(math.pi * lam)
        else:
            m0, m1 = torch.ones_like(h), self.U[0]
        self.M = [self.powers(m0, m1, 0, 8)] + [self.powers(torch.ones_like(h), self.U[d], d, 6) for d in (1, 2)]
        self.x2, self.x4 = 2.0 * h, 8.0 * h * h

    def powers(self, m0, m1, d, n):
        M = [m0, m1]
        while len(M) < n:
            M.append(self.U[d] * M[-1] + (len(M) - 1) * self.h * M[-2])
        return M

    def one(self, i, j, k):
        return self.M[0][i] * self.M[1][j] * self.M[2][k]

    def psi(self, i, j, k, x=0):
        """< u^i v^j w^k (xi^2)^x psi >"""
        f, f2 = ((1.0, self.x2), (self.x2, self.x4))[x]
        e = 0.5 * (f * (self.one(i + 2, j, k) + self.one(i, j + 2, k) + self.one(i, j, k + 2)) + f2 * self.one(i, j, k))
        return [f * self.one(i, j, k), f * self.one(i + 1, j, k), f * self.one(i, j + 1, k), f * self.one(i, j, k + 1), e]

    def apsi(self, a, i, j, k):
        """< u^i v^j w^k (a . psi) psi >"""
        t = [self.psi(*ix) for ix in ((i, j, k), (i + 1, j, k), (i, j + 1, k), (i, j, k + 1), (i + 2, j, k), (i, j + 2, k),
                                      (i, j, k + 2))] + [self.psi(i, j, k, 1)]
        return [a[0] * t[0][q] + a[1] * t[1][q] + a[2] * t[2][q] + a[3] * t[3][q]
                + 0.5 * a[4] * (t[4][q] + t[5][q] + t[6][q] + t[7][q]) for q in range(5)]

    def slope(self, dW):
        """a with < a . psi psi > = dW / rho over all velocities"""
        d = [x / self.rho for x in dW]
        U, h = self.U, self.h
        r = [d[1 + i] - U[i] * d[0] for i in range(3)]
        r4 = 2.0 * d[4] - (U[0] ** 2 + U[1] ** 2 + U[2] ** 2 + 5.0 * h) * d[0]
        a4 = (r4 - 2.0 * (U[0] * r[0] + U[1] * r[1] + U[2] * r[2])) / (5.0 * h * h)
        a = [r[i] / h - U[i] * a4 for i in range(3)]
        a0 = d[0] - U[0] * a[0] - U[1] * a[1] - U[2] * a[2] - 0.5 * a4 * (U[0] ** 2 + U[1] ** 2 + U[2] ** 2 + 5.0 * h)
        return [a0, *a, a4]


def _moving(g, a, i):
    """rho < u^i (a . velocity) psi >"""
    t = [g.apsi(a[0], i + 1, 0, 0), g.apsi(a[1], i, 1, 0), g.apsi(a[2], i, 0, 1)]
    return [g.rho * (t[0][q] + t[1][q] + t[2][q]) for q in range(5)]


def _flux(p, n, bnd, WL, GL, WR, GR, dt):
    """Time-averaged flux, interface state at dt and compression factor per point; W [k, 5], G [k, 5, 3]."""
    sign = torch.where(n[:, 2] >= 0, 1.0, -1.0).to(F64)
    a = -1.0 / (sign + n[:, 2])
    b = n[:, 0] * n[:, 1] * a
    E = torch.stack([n, torch.stack([1.0 + sign * n[:, 0] ** 2 * a, sign * b, -sign * n[:, 0]], 1),
                     torch.stack([b, sign + n[:, 1] ** 2 * a, -n[:, 1]], 1)], 1)         # rows n, t1, t2

    def turn(W):
        return [W[:, 0], *(E @ W[:, 1:4, None])[..., 0].unbind(1), W[:, 4]]

    def turn_gradient(G):
        D = (G @ E.transpose(1, 2)).permute(0, 2, 1)                                      # k, direction, variable
        v = torch.einsum("kij,kdj->kdi", E, D[:, :, 1:4])
        return [[D[:, d, 0], v[:, d, 0], v[:, d, 1], v[:, d, 2], D[:, d, 4]] for d in range(3)]
    gl, gr = _Maxwellian(turn(WL), 1.0), _Maxwellian(turn(WR), -1.0)
    Wc = [gl.rho * x + gr.rho * y for x, y in zip(gl.psi(0, 0, 0), gr.psi(0, 0, 0))]
    gc = _Maxwellian(Wc, 0)
    jump = ((gl.p - gr.p) / (gl.p + gr.p)).abs()
    if p["viscous"]:
        tau = _viscosity(p, 1.4 * gc.h) / gc.p
        tn = tau + jump * dt
    else:
        tau = tn = (0.01 + jump) * dt
    e = torch.exp(-dt / tn)
    om = 1.0 - e
    q1 = dt - tn * om
    q2 = (tn * tn + tau * tn) * om - tn * dt * e - tau * dt
    q3 = 0.5 * dt * dt - tau * dt + tau * tn * om
    q4 = tn * om
    q5 = (tau * tn + tn * tn) * om - tn * dt * e
    F, I, S = ([0.0] * 5 for _ in range(3))
    dWc = [[0.0] * 5 for _ in range(3)]
    for g, grad in ((gl, turn_gradient(GL)), (gr, turn_gradient(GR))):
        s = [g.slope(d) for d in grad]
        full = _Maxwellian([g.rho, g.rho * g.U[0], g.rho * g.U[1], g.rho * g.U[2],
                            2.5 * g.p + 0.5 * g.rho * (g.U[0] ** 2 + g.U[1] ** 2 + g.U[2] ** 2)], 0)
        A = g.slope([-x for x in _moving(full, s, 0)])
        for d in range(3):
            t = g.apsi(s[d], 0, 0, 0)
            dWc[d] = [dWc[d][q] + g.rho * t[q] for q in range(5)]
        v0, f0, va, fa = g.psi(0, 0, 0), g.psi(1, 0, 0), _moving(g, s, 0), _moving(g, s, 1)
        vA, fA = g.apsi(A, 0, 0, 0), g.apsi(A, 1, 0, 0)
        F = [F[q] + q4 * g.rho * f0[q] - q5 * fa[q] - tau * q4 * g.rho * fA[q] for q in range(5)]
        I = [I[q] + q4 * g.rho * v0[q] - q5 * va[q] - tau * q4 * g.rho * vA[q] for q in range(5)]
        S = [S[q] + e * (g.rho * v0[q] - (tau + dt) * va[q] - tau * g.rho * vA[q]) for q in range(5)]
    s = [gc.slope(d) for d in dWc]
    va, fa, f0 = _moving(gc, s, 0), _moving(gc, s, 1), gc.psi(1, 0, 0)
    A = gc.slope([-x for x in va])
    fA = gc.apsi(A, 1, 0, 0)
    F = [F[q] + gc.rho * (q1 * f0[q] + q3 * fA[q]) + q2 * fa[q] for q in range(5)]
    I = [I[q] + q1 * Wc[q] + (q2 - q3) * va[q] for q in range(5)]
    S = [S[q] + om * (Wc[q] - dt * va[q]) for q in range(5)]
    if p["viscous"] and p["prandtl"] != 1.0:
        U = gc.U

        def about(X):
            return X[4] - U[0] * X[1] - U[1] * X[2] - U[2] * X[3] + 0.5 * (U[0] ** 2 + U[1] ** 2 + U[2] ** 2) * X[0]
        F[4] = F[4] + (1.0 / p["prandtl"] - 1.0) * (about(F) - U[0] * about(I))
    mach = [[g.U[d] / torch.sqrt(1.4 * g.h) for d in range(3)] for g in (gl, gr)]
    dp, dm = (gl.p - gr.p).abs(), [mach[0][d] - mach[1][d] for d in range(3)]
    A = dp / gl.p + dp / gr.p + dm[0] ** 2 + dm[1] ** 2 + dm[2] ** 2
    factor = torch.where(bnd, torch.ones_like(A), 1.0 / (1.0 + A * A)) if p["compression_factor"] else torch.ones_like(A)

    def back(X):
        v = (E.transpose(1, 2) @ torch.stack(X[1:4], 1)[..., None])[..., 0]
        return torch.cat([X[0][:, None], v, X[4][:, None]], 1)
    return back([x / dt for x in F]), back(S), factor


def _residual(geo, p, W, G, alpha):
    coef, dt = _reconstruct(geo, p, W, G, alpha)
    f = geo.pf
    L, R = geo.L[f], geo.R[f]
    bnd = R < 0
    Rc = torch.where(bnd, L, R)
    WL, GL = _evaluate(coef[L], geo.px - geo.ctr[L])
    # the right cell seen from the left side of the face: shifted by the period
    WR, GR = _evaluate(coef[Rc], geo.px - geo.shift[f] - geo.ctr[Rc])
    area = geo.pA.norm(dim=1)
    n = geo.pA / area[:, None]
    if bool(bnd.any()):
        at = torch.nonzero(bnd)[:, 0]
        gw, gg = _ghost(p, geo.tag[f][at], n[at], WL[at], GL[at])
        WR, GR = WR.index_put((at,), gw), GR.index_put((at,), gg)
    F, S, factor = _flux(p, n, bnd, WL, GL, WR, GR, torch.minimum(dt[L], dt[Rc]))
    F = F * area[:, None]
    SA = (S[:, :, None] * geo.pA[:, None]).reshape(len(f), 15)
    both = torch.nonzero(~bnd)[:, 0]
    res = torch.zeros(geo.nc, 5, dtype=F64, device=W.device).index_add(0, L, -F).index_add(0, R[both], F[both])
    grad = torch.zeros(geo.nc, 15, dtype=F64, device=W.device).index_add(0, L, SA).index_add(0, R[both], -SA[both])
    log = torch.zeros(geo.nc, dtype=F64, device=W.device)
    lf = torch.log(factor)
    new = torch.exp(log.index_add(0, L, lf).index_add(0, R[both], lf[both]))
    grad = grad * (new / geo.vol)[:, None]
    return dict(res=res.T.contiguous(), grad=grad.T.contiguous(), alpha=new, dt=dt)
