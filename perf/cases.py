"""The work that programs give this solver, as cases that can be timed and
compared.

One Newton step of the segregated predictor multi-corrector asks for the
set-up and the solve of a velocity-pressure block system and for a mesh
motion solve; the cases run these whole calls over the range of meshes that
the generator's presets and the tests span (a few thousand to 2.5 million
unknowns, straight, stenosed and bifurcating vessels, odd section and layer
counts), in FP64 and in the mixed precision form, with a new Jacobian per
call or one kept set-up, one or eight right-hand sides, one system or a batch
of them, and the Newton corrector with its element loops.

The block systems are Jacobians of the generator: the tangent at a state
between two assembled ones (inflow peaks 20 and 40 cm/s, other perturbations),
the place between them drawn from the seed.  Right-hand sides are calA x* for
a drawn, smooth x* of a Newton increment's size (velocity rates about 3e3,
pressure rates about 1e7, as the presets' own solutions have them; the
velocity close to divergence-free, zero on Dirichlet nodes), so that x* is
what an exact solve returns.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import fsi_inputs as F
import paper_2206_06996_gb300 as pkg


# --------------------------------------------------------------------- cases
def _tube(name, what, n_circ, n_rad_f, n_rad_s, n_ax, precision="fp64", kind=0, **more):
    return dict(name=name, what=what, kind=kind, n_circ=n_circ, n_rad_f=n_rad_f, n_rad_s=n_rad_s, n_ax=n_ax,
                precision=precision, **more)


def listed():
    return [
        # a kept set-up and one more right-hand side on the smallest vessel
        # (preset tube_mini): the modified Newton iteration of a quick study,
        # nothing but launches and waits
        _tube("solve tiny vessel fp64", "solve", 12, 3, 2, 12),
        # one Newton step on the small preset (tube_small): set-up, solve,
        # mesh set-up, mesh solve
        _tube("step small vessel fp64", "step", 24, 4, 2, 40),
        # the same with odd counts everywhere, in mixed precision
        _tube("step odd vessel mixed", "step", 37, 5, 3, 61, "mixed"),
        # SIMPLE instead of Schur complement reduction, kept set-up
        _tube("simple medium vessel mixed", "solve", 48, 8, 4, 75, "mixed", precond="simple"),
        # a bifurcation with a kept set-up (modified Newton), FP64
        _tube("solve bifurcation fp64", "solve", 24, 11, 3, 48, kind=2),
        # a stenosed vessel of the wide section (preset stenosis, shortened)
        _tube("step stenosis mixed", "step", 160, 13, 7, 30, "mixed", kind=1),
        # many vessels of uneven size as one block-diagonal solve
        dict(name="batch of vessels fp64", what="batch", members=8, first=0, precision="fp64"),
        # Newton corrector with the mesh moving inside: element loops,
        # numeric re-set-up, block solves, mesh solves
        _tube("newton ale vessel fp64", "newton", 48, 7, 3, 80, n_iter=2),
        # eight inflow peaks on one Jacobian as one block solve
        _tube("eight rhs vessel mixed", "multi", 96, 11, 5, 80, "mixed"),
        # mesh motion alone, kept set-up, on the bench section
        _tube("mesh motion large fp64", "mesh", 96, 11, 5, 200),
        # one Newton step on half of the bench tube in FP64: HBM and the FP64 pipe
        _tube("step half bench tube fp64", "step", 96, 11, 5, 200),
        # the bench tube (preset tube_large, 2.5 million unknowns) in mixed precision
        _tube("step bench tube mixed", "step", 96, 11, 5, 400, "mixed"),
    ]


def draw(rng):
    """Vessels with the presets' proportions from about 800 to 300k nodes,
    every size drawn on a logarithmic scale and every count by itself."""
    what = rng.choice(["step", "step", "solve", "multi", "mesh", "newton", "batch"])
    precision = rng.choice(["fp64", "mixed"])
    if what == "batch":
        return dict(what="batch", members=rng.randint(2, 7), first=rng.randint(0, 50), precision=precision)
    # eight columns on a very coarse vessel share one Krylov space for
    # thousands of steps: not what the block form is for
    low, top = {"newton": (800.0, 4e4), "multi": (4e3, 2.5e4)}.get(what, (800.0, 3e5))
    nodes = math.exp(rng.uniform(math.log(low), math.log(top)))
    kind = rng.choice([0, 0, 1])
    # sections of the presets: 61 nodes (12 x 5 rings) to 1537 (96 x 16)
    section = min(1600.0, max(55.0, nodes ** 0.6 * 0.85)) * math.exp(rng.uniform(-0.25, 0.25))
    n_circ = max(8, int(round(math.sqrt(section * 5.0) * math.exp(rng.uniform(-0.15, 0.15)))))
    rings = max(4, int(round(section / n_circ)))
    n_rad_s = max(1, int(round(rings * rng.uniform(0.25, 0.4))))
    n_rad_f = max(2, rings - n_rad_s)
    n_ax = max(8, int(round(nodes / (1 + n_circ * (n_rad_f + n_rad_s)))) - 1)
    c = dict(what=what, kind=kind, n_circ=n_circ, n_rad_f=n_rad_f, n_rad_s=n_rad_s, n_ax=n_ax, precision=precision)
    if what == "newton":
        c["n_iter"] = rng.randint(1, 2)
    if what == "mesh":
        c["precision"] = "fp64"  # the mesh solve has one precision
    return c


def _geometry(case):
    """Generator parameters of a vessel (the bifurcation's radius, wall and
    branch length are the presets')."""
    g = {k: case[k] for k in ("kind", "n_circ", "n_rad_f", "n_rad_s", "n_ax")}
    if case["kind"] == 2:
        g.update(R=0.5, wall=0.06, L=4.0)
    return g


# -------------------------------------------------------------------- systems
_base = {}  # the last vessels' two assembled states on the device, by geometry


def _assembled(geometry, keep=2):
    """Two Jacobians of one mesh (inflow peaks 20 and 40 cm/s): the first
    one's values, the difference to the second, patterns and mesh."""
    key = tuple(sorted(geometry.items()))
    if key not in _base:
        while len(_base) >= keep:
            _base.pop(next(iter(_base)))
        one = F.tube_system("vessel", keep_mesh=True, u_max=20.0, seed=2206, **geometry)
        two = F.tube_system("vessel", u_max=40.0, seed=4412, **geometry)
        dev = {}
        for n in "ABCD":
            M, N = getattr(one, n), getattr(two, n)
            v = torch.as_tensor(M.val, device="cuda")
            dev[n] = (M.br, M.bc, M.nb_rows, M.nb_cols, torch.as_tensor(M.row_ptr, device="cuda"),
                      torch.as_tensor(M.col, device="cuda"), v, torch.as_tensor(N.val, device="cuda") - v)
        L = one.L
        dev["L"] = (1, 1, L.nb_rows, L.nb_cols, torch.as_tensor(L.row_ptr, device="cuda"),
                    torch.as_tensor(L.col, device="cuda"), torch.as_tensor(L.val, device="cuda"), None)
        _base[key] = dev, one.mesh, one.params
    return _base[key]


def _matrix(entry, w):
    br, bc, nr, nc, rp, col, v, d = entry
    val = v.clone() if d is None else torch.add(v, d, alpha=w)
    return pkg.DeviceBSR(br, bc, nr, nc, rp.clone(), col.clone(), val)


def _times(M, x):
    """M x for a device matrix, in torch (x: nb_cols * bc entries, or that by
    the number of columns)."""
    k = x.numel() // (M.nb_cols * M.bc)
    xb = x.reshape(M.nb_cols, M.bc, k)[M.col.long()]
    y = torch.matmul(M.val.reshape(-1, M.br, M.bc), xb).reshape(M.nnzb, M.br * k)
    lengths = (M.row_ptr[1:] - M.row_ptr[:-1]).long()
    return torch.segment_reduce(y, "sum", lengths=lengths, axis=0, unsafe=True).reshape(-1)


def _increment(mesh, seed):
    """A drawn smooth Newton increment x*: swirl and axial stretch that
    vanish at both ends (divergence-free) with a small general part, zero on
    the Dirichlet nodes, and smooth pressures."""
    g = np.random.default_rng(seed)
    xyz = torch.as_tensor(mesh.xyz, device="cuda")
    lo, hi = xyz.amin(0), xyz.amax(0)
    z = (xyz[:, 2] - lo[2]) / (hi[2] - lo[2])
    a = 0.5 * (hi[0] - lo[0])
    x, y = xyz[:, 0] / a, xyz[:, 1] / a
    swirl, h, dh = torch.zeros_like(z), torch.zeros_like(z), torch.zeros_like(z)
    length = float((hi[2] - lo[2]) / a)
    for k in range(1, 4):
        ak, bk = g.standard_normal(2) / k
        swirl += ak * torch.sin(k * math.pi * z)
        h += bk * (1.0 - torch.cos(2.0 * k * math.pi * z))
        dh += bk * 2.0 * k * math.pi / length * torch.sin(2.0 * k * math.pi * z)
    v = torch.stack([-y * swirl - 0.5 * x * dh, x * swirl - 0.5 * y * dh, h], 1)
    for c in range(3):
        e = g.standard_normal(4)
        v[:, c] += 0.02 * (e[0] + e[1] * x + e[2] * y + e[3] * x * y) * torch.sin(math.pi * z)
    v *= 3e3
    v[torch.as_tensor(mesh.dir_v, device="cuda")] = 0.0
    p = torch.zeros_like(z)
    for k in range(3):
        e = g.standard_normal(3)
        p += (e[0] + 0.3 * e[1] * x + 0.3 * e[2] * y) * torch.cos(k * math.pi * z) / (1 + k)
    p *= 1e7
    # node pressures, then the interface's second ones
    extra = np.flatnonzero(mesh.iface_of >= 0)
    extra = extra[np.argsort(mesh.iface_of[extra])]
    return torch.cat([v.reshape(-1), p, p[torch.as_tensor(extra, device="cuda")]])


def _mesh_displacement(mesh, seed):
    """A drawn smooth mesh displacement of the fluid nodes (three
    interleaved components)."""
    g = np.random.default_rng(seed + 1)
    nodes = np.flatnonzero(mesh.fluid_id >= 0)
    nodes = nodes[np.argsort(mesh.fluid_id[nodes])]
    xyz = torch.as_tensor(mesh.xyz[nodes], device="cuda")
    z = xyz[:, 2] / xyz[:, 2].amax()
    u = torch.zeros_like(xyz)
    for c in range(3):
        for k in range(1, 4):
            e = g.standard_normal(3)
            u[:, c] += 1e-3 / k * (e[0] + e[1] * xyz[:, 0] + e[2] * xyz[:, 1]) * torch.sin(k * math.pi * z)
    return u.reshape(-1)


def _weight(seed):
    return float(np.random.default_rng(seed + 2).uniform(0.1, 0.9))


def _blocks(geometry, seed):
    dev, mesh, params = _assembled(geometry)
    w = _weight(seed)
    return [_matrix(dev[n], w) for n in "ABCD"], dev, mesh, params


def _rhs(mats, x):
    A, B, C, D = mats
    xv, xp = x[: 3 * A.nb_rows], x[3 * A.nb_rows :]
    return torch.cat([_times(A, xv) + _times(B, xp), _times(C, xv) + _times(D, xp)])


def _solver(case, **more):
    opts = dict(precision=pkg.SCR_MIXED if case["precision"] == "mixed" else pkg.SCR_FP64)
    if case.get("precond") == "simple":
        opts["precond"] = pkg.SCR_PC_SIMPLE
    return pkg.BlockSolver(**opts, **more)


PEAKS = 8  # right-hand sides of a "multi" case: inflow peaks up to 60 cm/s


def _columns(mesh, seed):
    peaks = np.random.default_rng(seed + 3).uniform(2.0, 60.0, PEAKS) / 30.0
    return [float(s) * _increment(mesh, 100 * seed + c) for c, s in enumerate(peaks)]


def _members(case):
    """Parameters of the batch: consecutive members of the generator's
    uneven set, at half their length (the seed moves their states)."""
    out = []
    for i in range(case["members"]):
        p = F.batch_member_params(case["first"] + i)
        p["n_ax"] = max(8, p["n_ax"] // 2)
        out.append(p)
    return out


# ---------------------------------------------------------------------- a case
def prepare(case, seed):
    what = case["what"]
    if what == "batch":
        systems, bs = [], []
        for i, p in enumerate(_members(case)):
            dev, mesh, _ = _assembled({k: v for k, v in p.items() if k != "seed"}, keep=16)
            mats = [_matrix(dev[n], _weight(seed + i)) for n in "ABCD"]
            systems.append(tuple(mats))
            bs.append(_rhs(mats, _increment(mesh, seed + 10 * i)))
        return dict(what=what, sol=_solver(case), systems=systems, bs=bs)
    geometry = _geometry(case)
    if what == "mesh":
        dev, mesh, _ = _assembled(geometry)
        L = _matrix(dev["L"], 0.0)
        g = _times(L, _mesh_displacement(mesh, seed))
        return dict(what=what, sol=_solver(case).mesh_setup(L), g=g)
    mats, dev, mesh, params = _blocks(geometry, seed)
    if what == "multi":
        return dict(what=what, sol=_solver(case, nrhs=PEAKS), mats=mats,
                    bs=[_rhs(mats, x) for x in _columns(mesh, seed)])
    if what == "solve":
        return dict(what=what, sol=_solver(case).setup(*mats), b=_rhs(mats, _increment(mesh, seed)))
    if what == "step":
        L = _matrix(dev["L"], 0.0)
        return dict(what=what, sol=_solver(case), mats=mats, L=L, b=_rhs(mats, _increment(mesh, seed)),
                    g=_times(L, _mesh_displacement(mesh, seed)))
    # newton: the state of a time step's predictor, rates zero
    asm = F.Assembler(F.make_params(u_max=20.0 + 20.0 * _weight(seed), seed=seed % 100003, **geometry))
    v, p = asm.initial_state()
    lap = asm.mesh_laplacian()
    asm.close()
    sol = _solver(case, newton=1).setup(*mats)
    sol.assembly_setup(mesh, params)
    sol.mesh_setup(_matrix(dev["L"], 0.0))
    sol.mesh_coupling(lap, mesh.fluid_id, mesh.dir_m, F.interface_follow(mesh))
    zero = torch.zeros(v.size, dtype=torch.float64, device="cuda")
    return dict(what=what, sol=sol, v=torch.as_tensor(v, device="cuda"), p=torch.as_tensor(p, device="cuda"),
                zero=zero, uhat=torch.zeros(3 * mesh.n_fluid, dtype=torch.float64, device="cuda"),
                n_iter=case["n_iter"])


def run(state):
    what, sol = state["what"], state["sol"]
    if what == "solve":
        return {"x": sol.solve(state["b"])}
    if what == "step":
        sol.setup(*state["mats"])
        x = sol.solve(state["b"])
        sol.mesh_setup(state["L"])
        return {"x": x, "u": sol.mesh_solve(state["g"])}
    if what == "mesh":
        return {"u": sol.mesh_solve(state["g"])}
    if what == "multi":
        sol.setup(*state["mats"])
        return {"x": sol.solve_multi(state["bs"])[0]}
    if what == "batch":
        sol.setup_batch(state["systems"])
        return {"x": sol.solve_batch(state["bs"])}
    # the corrector updates its state in place: it starts from the predictor's copy
    v, p = state["v"].clone(), state["p"].clone()
    vdot, u = state["zero"].clone(), state["zero"].clone()
    norms, uhat = sol.corrector_ale(v, p, vdot, u, state["uhat"], state["n_iter"])
    return {"v": v, "p": p, "vdot": vdot, "u": u, "uhat": uhat, "first_norm": float(norms[0])}


def _sizes(geometry):
    """(velocity nodes, pressures, fluid nodes, stored blocks per node) of a
    vessel, from its counts."""
    if geometry["kind"] == 2:
        # an O-grid: core cells and four arcs of rings, about
        c, f, s, n = (geometry[k] for k in ("n_circ", "n_rad_f", "n_rad_s", "n_ax"))
        section, fluid = (c + 1) ** 2 + 4 * c * (f + s), (c + 1) ** 2 + 4 * c * f
    else:
        c, f, s, n = (geometry[k] for k in ("n_circ", "n_rad_f", "n_rad_s", "n_ax"))
        section, fluid = 1 + c * (f + s), 1 + c * f
    nv = section * (n + 1)
    return nv, nv + c * (n + 1), fluid * (n + 1), 14.5


def work(case):
    """What a pass cannot do without: the system's matrices read once (a
    kept set-up is read once by its solve too), right-hand sides read and
    solutions written, and two operations per stored value for one product
    with the whole system."""
    what = case["what"]
    if what == "batch":
        sizes = [_sizes(p) for p in _members(case)]
    else:
        sizes = [_sizes(_geometry(case))]
    nbytes = flops = 0.0
    for nv, np_, nf, k in sizes:
        block = k * (nv * (9 * 8 + 4) + 2 * np_ * (3 * 8 + 4) + np_ * (8 + 4))
        mesh = 14.0 * nf * (8 + 4)
        vec = 8.0 * (3 * nv + np_)
        values = k * (9 * nv + 6 * np_ + np_)
        cols = PEAKS if what == "multi" else 1
        if what != "mesh":
            nbytes += block + 2 * cols * vec
            flops += 2.0 * cols * values * case.get("n_iter", 1)
        if what in ("step", "mesh", "newton"):
            nbytes += mesh + 2 * 24.0 * nf
            flops += 6.0 * 14.0 * nf
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    """The solutions that the right-hand sides were made from; the
    corrector's nonlinear iteration has none at hand."""
    what = case["what"]
    if what == "batch":
        out = []
        for i, p in enumerate(_members(case)):
            mesh = F.build_mesh(F.make_params(**{k: v for k, v in p.items() if k != "seed"}))
            out.append(_increment(mesh, seed + 10 * i))
        return {"x": out}
    if what == "newton":
        return None
    mesh = F.build_mesh(F.make_params(**_geometry(case)))
    if what == "solve":
        return {"x": _increment(mesh, seed)}
    if what == "step":
        return {"x": _increment(mesh, seed), "u": _mesh_displacement(mesh, seed)}
    if what == "mesh":
        return {"u": _mesh_displacement(mesh, seed)}
    return {"x": _columns(mesh, seed)}
