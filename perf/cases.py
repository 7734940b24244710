"""Performance cases of the finite-volume library: what its users run, through its public
entry points (the C ABI binding ``capi`` and ``DeviceMesh``).

Meshes are the repository's own recipes (jittered triangles of the unit square, jittered
Kuhn tetrahedra of the unit cube), their cells sorted along the Morton curve beforehand, so
that the library's internal cell order is the caller's. A mesh is uploaded once and kept, as
a program that advances a solution in time keeps it; the fields are made from the seed.

The exact values are plain FP64 torch, written here from the method's definitions.
"""
from __future__ import annotations

import collections
import math

import numpy as np
import torch

from paper_2203_00925_gb300 import capi, device
from synth.meshgen import jittered_cube, jittered_square
from synth.workloads import E_CHARGE, EPS0, StreamerCase

E_OVER_EPS0 = E_CHARGE / EPS0
CASE = StreamerCase()               # coefficients of the streamer workloads
WALLS = {t: ("wall", 0.0) for t in (1, 2, 3, 4)}
HIDDEN, HOPS, BOX_SLOTS = 64, 2, 6  # the warm-start network
F64 = torch.float64


def listed():
    return [
        # the 2D scalar advection-diffusion run: 5,000 triangles, 200 Euler steps in one call
        {"name": "advect2d_5k_f64", "kind": "transport", "dim": 2, "n": 50, "prec": "fp64", "recon": 0,
         "stages": 1, "steps": 200, "field": False, "src": False, "bc": "walls"},
        # one transport step of the coupled workload on the largest mesh: cell velocities,
        # source, the three stages of eq. 6, single precision
        {"name": "transport_f32_6m", "kind": "transport", "dim": 3, "n": 100, "prec": "mixed", "recon": 0,
         "stages": 3, "steps": 1, "field": True, "src": True, "bc": "streamer"},
        # second-order transport in double precision on a medium mesh
        {"name": "muscl_f64_162k", "kind": "transport", "dim": 3, "n": 30, "prec": "fp64", "recon": 1,
         "stages": 3, "steps": 2, "field": True, "src": True, "bc": "streamer"},
        # the field of the double-precision streamer: the least-squares gradient of the potential
        {"name": "gradient_f64_750k", "kind": "gradient", "dim": 3, "n": 50, "prec": "fp64", "bc": "streamer"},
        # the same in single precision on the largest mesh (the mixed-precision streamer)
        {"name": "gradient_f32_6m", "kind": "gradient", "dim": 3, "n": 100, "prec": "mixed", "bc": "streamer"},
        # a Poisson solve of test size (the sample mesh of the CPU comparison): launches and
        # grid-wide waits
        {"name": "poisson_f64_10k", "kind": "poisson", "n": 12, "prec": "fp64", "inner": 0, "inner_rtol": 0.5},
        # the double-precision solve of the 750,000-cell workload
        {"name": "poisson_f64_750k", "kind": "poisson", "n": 50, "prec": "fp64", "inner": 0, "inner_rtol": 0.5},
        # the mixed-precision solve of the 6,000,000-cell workload
        {"name": "poisson_mixed_6m", "kind": "poisson", "n": 100, "prec": "mixed", "inner": 0, "inner_rtol": 0.5},
        # a whole step of the fastest configuration: multigrid inner solve, mixed precision,
        # captured as one graph
        {"name": "streamer_mixed_6m", "kind": "streamer", "n": 100, "prec": "mixed", "inner": 2, "inner_rtol": 0.5,
         "graph": True, "recon": 0, "parts": 1, "steps": 1},
        # a batch of independent meshes of uneven sizes (20k to 200k cells), one graph step
        {"name": "ensemble_mixed_16", "kind": "streamer", "n": 32, "prec": "mixed", "inner": 0, "inner_rtol": 0.2,
         "graph": True, "recon": 0, "parts": 16, "steps": 1},
        # the learned start: a prediction by the multilevel network
        {"name": "predict_750k", "kind": "predict", "n": 50, "multilevel": True},
        # its training: loss gradient of one sample (forward and backward)
        {"name": "train_162k", "kind": "train", "n": 30, "multilevel": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["transport", "transport", "gradient", "gradient", "poisson", "poisson", "streamer", "predict", "train"])
    prec = rng.choice(["fp64", "mixed"])
    if kind == "transport":
        recon, stages = rng.choice([0, 1]), rng.choice([1, 3])
        if rng.random() < 0.4:
            n, steps = _log_int(rng, 50, 900), rng.choice([1, 10, 50])
            return {"kind": kind, "dim": 2, "n": n, "prec": prec, "recon": recon, "stages": stages,
                    "steps": max(1, min(steps, 4_000_000 // (n * n * stages))), "field": rng.random() < 0.5,
                    "src": rng.random() < 0.5, "bc": "walls"}
        return {"kind": kind, "dim": 3, "n": _log_int(rng, 10, 100), "prec": prec, "recon": recon, "stages": stages,
                "steps": 1, "field": rng.random() < 0.7, "src": rng.random() < 0.5, "bc": "streamer"}
    if kind == "gradient":
        if rng.random() < 0.2:
            return {"kind": kind, "dim": 2, "n": _log_int(rng, 50, 900), "prec": prec, "bc": "walls"}
        return {"kind": kind, "dim": 3, "n": _log_int(rng, 10, 100), "prec": prec, "bc": "streamer"}
    if kind == "poisson":
        return {"kind": kind, "n": _log_int(rng, 10, 64 if prec == "fp64" else 90), "prec": prec, "inner": rng.choice([0, 0, 2]),
                "inner_rtol": rng.choice([0.1, 0.5])}
    if kind == "streamer":
        return {"kind": kind, "n": _log_int(rng, 12, 64), "prec": prec, "inner": rng.choice([0, 2]), "inner_rtol": 0.5,
                "graph": rng.random() < 0.5, "recon": rng.choice([0, 1]), "parts": 1, "steps": rng.choice([1, 2])}
    return {"kind": kind, "n": _log_int(rng, 12, 64 if kind == "predict" else 40), "multilevel": rng.random() < 0.5}


# ---- meshes -----------------------------------------------------------------------------------
def _spread(v, dim):
    v = v.astype(np.uint64)
    steps = (((32, 0x1f00000000ffff), (16, 0x1f0000ff0000ff), (8, 0x100f00f00f00f00f), (4, 0x10c30c30c30c30c3),
              (2, 0x1249249249249249)) if dim == 3 else
             ((16, 0x0000ffff0000ffff), (8, 0x00ff00ff00ff00ff), (4, 0x0f0f0f0f0f0f0f0f), (2, 0x3333333333333333),
              (1, 0x5555555555555555)))
    for s, m in steps:
        v = (v | (v << np.uint64(s))) & np.uint64(m)
    return v


def _morton(mesh):
    """The mesh with its cells sorted along the Morton curve of their centres."""
    x = mesh.xyz
    cen = x[mesh.cells[:, 0]].copy()
    for k in range(1, mesh.dim + 1):
        cen += x[mesh.cells[:, k]]
    cen /= mesh.dim + 1
    lo, span = cen.min(axis=0), np.ptp(cen, axis=0)
    q = np.rint((cen - lo) / span * (2097151.0 if mesh.dim == 3 else 4294967295.0))
    key = np.zeros(cen.shape[0], dtype=np.uint64)
    for a in range(mesh.dim):
        key |= _spread(q[:, a], mesh.dim) << np.uint64(a)
    mesh.cells = np.ascontiguousarray(mesh.cells[np.argsort(key, kind="stable")])
    return mesh


def _part_sizes(case):
    """Cube resolutions of a batch: log-uniform cell counts up to 6 n^3 (a tenth at least)."""
    rng = np.random.default_rng(5000 + case["n"])
    top = 6.0 * case["n"] ** 3
    return [max(2, round((t / 6.0) ** (1 / 3))) for t in np.exp(rng.uniform(math.log(top / 10), math.log(top), case["parts"]))]


def _host_meshes(case):
    n = case["n"]
    if case.get("dim", 3) == 2:
        return [_morton(jittered_square(n))]
    if case.get("parts", 1) > 1:
        return [_morton(jittered_cube(k, seed=5000 + i)) for i, k in enumerate(_part_sizes(case))]
    return [_morton(jittered_cube(n, seed={100: 301}.get(n, 201)))]


def _bcs(case):
    """Boundary-condition sets: transport first, then (3D) the potential's."""
    if case.get("bc") == "walls":
        return [WALLS]
    return [CASE.bc_ne(), CASE.bc_phi()]


class _Mesh:
    def __init__(self, case):
        self.host = _host_meshes(case)
        many = len(self.host) > 1
        self.dm = device.DeviceMesh(self.host if many else self.host[0], [_bcs(case)] * len(self.host) if many else _bcs(case),
                                    prec=case.get("prec", "mixed"), ensemble=many)
        self.nets = {}
        self.work = None

    def __del__(self):
        for net in self.nets.values():
            capi.fvgb_mpnn_free(net)


_meshes = collections.OrderedDict()


def _mesh(case):
    key = (case.get("dim", 3), case["n"], case.get("prec", "mixed"), case.get("parts", 1), case.get("bc", "streamer"))
    if key not in _meshes:
        while len(_meshes) >= 20:
            _meshes.popitem(last=False)
        _meshes[key] = _Mesh(case)
    _meshes.move_to_end(key)
    return _meshes[key]


def _volumes(mesh):
    x = torch.as_tensor(mesh.xyz, device="cuda")[torch.as_tensor(mesh.cells, device="cuda").long()]
    return torch.linalg.det(x[:, 1:] - x[:, :1]) / math.factorial(mesh.dim)


# ---- inputs from the seed -----------------------------------------------------------------------
def _centres(hosts):
    out = []
    for m in hosts:
        x = torch.as_tensor(m.xyz, device="cuda")
        out.append(x[torch.as_tensor(m.cells, device="cuda").long()].mean(dim=1))
    return out


def _waves(c, g, count=6, top=3.0):
    """A smooth field of order one: a few random plane waves."""
    f = torch.zeros(c.shape[0], dtype=F64, device="cuda")
    for _ in range(count):
        k = (torch.rand(c.shape[1], generator=g, dtype=F64) * 2 - 1).to("cuda") * (2 * math.pi * top)
        f += float(torch.randn(1, generator=g)) / math.sqrt(count) * torch.cos(c @ k + 6.28 * float(torch.rand(1, generator=g)))
    return f


def _seeds(c, g, sigma, count=3):
    """Gaussian electron seeds (height about one) at random places."""
    f = torch.zeros(c.shape[0], dtype=F64, device="cuda")
    for _ in range(count):
        x = (0.2 + 0.7 * torch.rand(c.shape[1], generator=g, dtype=F64)).to("cuda")
        f += (0.3 + 0.7 * float(torch.rand(1, generator=g))) * torch.exp(-((c - x) ** 2).sum(dim=1) / sigma ** 2)
    return f


def _inputs(case, hosts, seed):
    """The case's fields in FP64, from the seed alone (rounded to the mesh's type by the caller)."""
    g = torch.Generator().manual_seed(seed)
    parts = _centres(hosts)
    c = torch.cat(parts)
    kind, h = case["kind"], min(m.h for m in hosts)
    if kind == "transport":
        v = torch.stack([0.6 + 0.4 * _waves(c, g) for _ in range(case["dim"])])
        # a stable step: outflow and two-point diffusion rates of a jittered simplex
        dt = 0.1 / (8.0 / h + 40.0 * 0.01 / h ** 2) if case["dim"] == 3 else 0.1 / (6.0 / h + 16.0 * 0.01 / h ** 2)
        return {"u": _seeds(c, g, 0.1) + 0.05, "vel": v, "src": 0.1 * _waves(c, g), "dt": dt}
    z = torch.cat([p[:, -1] for p in parts])
    if kind == "poisson":       # the previous step's potential, some volts off
        return {"f": -E_OVER_EPS0 * 2e13 * (_seeds(c, g, 0.03) - _seeds(c, g, 0.03)),
                "phi": CASE.V * z + 2.0 * _waves(c, g) * z * (1 - z)}
    if kind == "streamer":
        ne = torch.cat([CASE.peak * _seeds(p, g, 0.02) + CASE.background for p in parts])
        return {"ne": ne, "ni": ne * (1.0 + 0.001 * torch.cos(9.0 * z)),
                "phi": CASE.V * z + 2.0 * _waves(c, g) * z * (1 - z)}
    phi = CASE.V * z + 200.0 * _waves(c, g) * z * (1 - z)
    if kind == "gradient":
        return {"u": phi}
    dq = 1e13 * (_seeds(c, g, 0.05) - _seeds(c, g, 0.05))
    return {"dq": dq, "phi": phi, "dphi": 5.0 * _waves(c, g) * z * (1 - z)}


def _network(hosts):
    """The network a program holds: its parameters (as it is initialised) and its scales, the
    RMS of the inputs and of the target over a sample."""
    g = torch.Generator().manual_seed(11)
    theta = torch.cat([(torch.rand(o * (i + 1), generator=g) * 2 - 1) / math.sqrt(i)
                       for i, o in [(2, HIDDEN)] + 3 * [(2 * HIDDEN, HIDDEN)] + [(HIDDEN, 1)]]).float()
    x = _inputs({"kind": "train"}, hosts, 11)
    rms = lambda t: float(t.square().mean().sqrt())  # noqa: E731
    size = hosts[0].n_cell ** (-2 / 3)               # about the square of a cell's length
    return theta, [CASE.V, rms(E_OVER_EPS0 * x["dq"] * size) / CASE.V, rms(x["phi"]) / CASE.V, rms(x["dphi"]) / CASE.V]


def prepare(case, seed):
    m = _mesh(case)
    dm, x = m.dm, _inputs(case, m.host, seed)
    s = {"kind": case["kind"], "m": m, "dm": dm, "case": case}
    kind = case["kind"]
    if kind == "transport":
        s |= {"u0": x["u"].to(dm.real), "u": dm.empty(dm.n_cell), "dt": x["dt"]}
        s["tc"] = capi.tcoef(vel=x["vel"].to(dm.real).contiguous() if case["field"] else None,
                             vel_const=(1.0, 0.5, 0.25)[:case["dim"]], diff=0.01,
                             src=x["src"].to(dm.real) if case["src"] else None, recon=case["recon"])
        s["alpha"] = [0.5, 0.5, 1.0] if case["stages"] == 3 else None
    elif kind == "gradient":
        s |= {"u": x["u"].to(dm.real), "grad": dm.empty(dm.dim, dm.n_cell), "set": 0 if case["bc"] == "walls" else 1}
    elif kind in ("poisson", "streamer"):
        so = capi.solve_opts(rtol=1e-8, inner_rtol=case["inner_rtol"], inner=case["inner"],
                             prec=capi.FVGB_FP64 if case["prec"] == "fp64" else capi.FVGB_FP32)
        if kind == "poisson":
            s |= {"f": x["f"], "phi0": x["phi"], "phi": torch.empty_like(x["phi"]), "opts": so}
        else:
            capi.fvgb_set_graph_mode(dm.handle, case["graph"])
            s |= {"ne": x["ne"].to(dm.real), "ni": x["ni"].to(dm.real), "phi": x["phi"]}
            s["sp"] = capi.streamer_params(mu=CASE.mu, A=CASE.A, B=CASE.B, De=CASE.De, recon=case["recon"], solve=so,
                                           dt=CASE.dt(min(h.h for h in m.host)))
            if m.work is None:      # one set of arrays that the time loop advances
                m.work = [torch.empty_like(s["ne"]), torch.empty_like(s["ni"]), torch.empty_like(s["phi"]),
                          dm.empty(dm.dim, dm.n_cell)]
    else:
        if case["multilevel"] not in m.nets:
            theta, scales = _network(m.host)
            net = m.nets[case["multilevel"]] = capi.fvgb_mpnn_create(dm.handle, 1, multilevel=case["multilevel"])
            capi.fvgb_mpnn_set_params(net, theta.numpy())
            capi.fvgb_mpnn_set_scales(net, *scales)
        s |= {"net": m.nets[case["multilevel"]], "out": torch.empty_like(x["phi"]), **x}
    return s


def run(s):
    kind, h = s["kind"], s["dm"].handle
    if kind == "transport":
        s["u"].copy_(s["u0"])
        capi.fvgb_fv_step(h, s["tc"], s["u"], s["dt"], s["case"]["steps"], s["alpha"])
        return s["u"]
    if kind == "gradient":
        capi.fvgb_gradient(h, s["set"], s["u"], s["grad"])
        return s["grad"]
    if kind == "poisson":
        s["phi"].copy_(s["phi0"])
        capi.fvgb_poisson_solve(h, 1, s["f"], s["phi"], s["opts"])
        return s["phi"]
    if kind == "streamer":
        ne, ni, phi, E = s["m"].work
        ne.copy_(s["ne"])
        ni.copy_(s["ni"])
        phi.copy_(s["phi"])
        capi.fvgb_streamer_step(h, s["sp"], ne, ni, phi, E, s["case"]["steps"])
        return {"ne": ne, "ni": ni, "phi": phi, "E": E}
    net = s["net"]
    if kind == "predict":
        capi.fvgb_mpnn_predict(net, s["dq"], s["phi"], s["out"])
        return s["out"]
    loss, grad = capi.fvgb_mpnn_loss_grad(net, s["dq"], s["phi"], s["dphi"])
    return {"loss": loss, "grad": grad}


def work(case):
    """Bytes: fields in and out once, with the mesh that defines them (cell vertices and
    coordinates) for each operator evaluation; a solve: each conjugate-gradient iteration's
    vectors (r, p, q, x) and operator (four indices, four coefficients) once. Flops: the
    method's own multiply-adds."""
    dim, kind = case.get("dim", 3), case["kind"]
    sizes = _part_sizes(case) if case.get("parts", 1) > 1 else [case["n"]]
    N = sum(6 * k ** 3 if dim == 3 else 2 * k * k for k in sizes)
    V = sum((k + 1) ** dim for k in sizes)
    w = 8 if case.get("prec", "mixed") == "fp64" else 4
    mesh = 4 * (dim + 1) * N + 8 * dim * V
    nbr = 67 if dim == 3 else 12                     # node neighbours of a cell
    grad = {"bytes": (1 + dim) * w * N + mesh, "flops": (1 + 3 * dim) * nbr * N}
    flux = {"bytes": (2 + (dim if case.get("field") else 0) + (1 if case.get("src") else 0)) * w * N + mesh,
            "flops": (2 * (dim + 1) + 14 * (dim + 1) + 10) * N}
    if kind == "gradient":
        return grad
    if kind == "transport":
        times = case["stages"] * case["steps"]
        return {k: times * (flux[k] + (grad["flops"] * case["recon"] if k == "flops" else 0)) for k in flux}
    if kind in ("poisson", "streamer"):
        ws = 8 if case["prec"] == "fp64" else 4
        k = max(sizes)
        # iterations to 1e-8 grow with the cells along a side; a multigrid cycle does about
        # the work of four of them, and about twenty cycles do
        its = 16.0 * k if case["inner"] == 0 else 80.0
        solve = {"bytes": its * N * (4 * 4 + 4 * ws + 6 * ws), "flops": its * N * 20}
        if kind == "poisson":
            return solve
        return {q: case["steps"] * (solve[q] + grad[q] + flux[q]) for q in solve}
    nn = 2 * 3 * 2 * (2 * HIDDEN) * HIDDEN * N       # two evaluations of three layers
    return {"bytes": 24 * N + mesh, "flops": nn if kind == "predict" else 3 * nn}


# ---- exact values: the method's definitions in plain FP64 torch ------------------------------------
class _Plain:
    """Geometry and operators of one mesh; fields have the cells last."""

    def __init__(self, mesh, bcs):
        self.d = d = mesh.dim
        self.x = x = torch.as_tensor(mesh.xyz, device="cuda")
        self.cells = cells = torch.as_tensor(mesh.cells, device="cuda").long()
        self.N, self.V = N, V = cells.shape[0], x.shape[0]
        self.cen = x[cells].mean(dim=1)
        self.vol = _volumes(mesh)
        # faces: a cell's vertices but one, matched by their sorted vertices
        fv = torch.cat([cells[:, [j for j in range(d + 1) if j != k]] for k in range(d + 1)]).sort(dim=1).values
        key = fv[:, 0]
        for a in range(1, d):
            key = key * V + fv[:, a]
        owner = torch.arange(N, device="cuda").repeat(d + 1)
        key, o = key.sort(stable=True)
        owner, fv = owner[o], fv[o]
        first = torch.ones_like(key, dtype=torch.bool)
        first[1:] = key[1:] != key[:-1]
        at = first.nonzero()[:, 0]
        two = torch.zeros_like(at, dtype=torch.bool)
        two[:-1] = at[1:] - at[:-1] == 2
        two[-1] = key.numel() - at[-1] == 2
        a, b = owner[at], torch.where(two, owner[(at + 1).clamp(max=key.numel() - 1)], -1)
        self.L = torch.where(two, torch.minimum(a, b), a)
        self.R = torch.where(two, torch.maximum(a, b), b)
        self.fv, fkey = fv[at], key[at]
        bk = torch.as_tensor(mesh.bface_vert, device="cuda").long().sort(dim=1).values
        k = bk[:, 0]
        for j in range(1, d):
            k = k * V + bk[:, j]
        tag = torch.zeros_like(fkey)
        tag[torch.searchsorted(fkey, k)] = torch.as_tensor(mesh.bface_tag, device="cuda").long()
        self.inner = self.R >= 0
        self.Rs = self.R.clamp(min=0)
        P = x[self.fv]
        self.xf = P.mean(dim=1)
        e1 = torch.where(self.inner[:, None], self.cen[self.Rs], self.xf) - self.cen[self.L]
        if d == 3:
            S = 0.5 * torch.linalg.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
            G = torch.stack([e1, P[:, 0] - P[:, 2], P[:, 1] - P[:, 2]], dim=1)
        else:
            t = P[:, 1] - P[:, 0]
            S = torch.stack([t[:, 1], -t[:, 0]], dim=1)
            G = torch.stack([e1, t], dim=1)
        self.S = torch.where(((e1 * S).sum(dim=1) < 0)[:, None], -S, S)
        self.coef = torch.linalg.solve(G.transpose(1, 2), self.S)
        # boundary conditions: wall faces, Dirichlet faces and vertices (the smallest tag wins)
        self.wall = torch.zeros_like(self.inner)
        self.dirichlet = torch.zeros_like(self.inner)
        self.g = torch.zeros(tag.numel(), dtype=F64, device="cuda")
        self.vdir = torch.full((V,), math.nan, dtype=F64, device="cuda")
        for t in sorted(bcs, reverse=True):
            k, v = bcs[t]
            on = tag == t
            if k == "wall":
                self.wall |= on
            if k == "dirichlet":
                self.dirichlet |= on
                self.g[on] = v
                self.vdir[self.fv[on].reshape(-1)] = v
        # cells around each vertex
        A = cells.reshape(-1)
        o = A.argsort(stable=True)
        self.vA, self.vc = A[o], torch.div(o, d + 1, rounding_mode="floor")
        self.vn = torch.bincount(A, minlength=V)
        self.vp = torch.cat([torch.zeros(1, dtype=torch.long, device="cuda"), self.vn.cumsum(0)])
        # least-squares vertex weights
        r = torch.cat([torch.ones(A.numel(), 1, dtype=F64, device="cuda"), (self.cen[self.vc] - x[self.vA]) / mesh.h], dim=1)
        X = torch.zeros(V, d + 1, d + 1, dtype=F64, device="cuda").index_add_(0, self.vA, r[:, :, None] * r[:, None, :])
        s = X[:, 0, 1:]
        C = X[:, 1:, 1:] - s[:, :, None] * s[:, None, :] / self.vn[:, None, None]
        tr = C.diagonal(dim1=1, dim2=2).sum(dim=1) / d
        flat = (self.vn < d + 1) | ~(torch.linalg.det(C) / tr ** d >= 1e-10)
        X[flat] = torch.eye(d + 1, dtype=F64, device="cuda")
        y = torch.linalg.inv(X)[:, 0]
        self.alpha = torch.where(flat[self.vA], 1.0 / self.vn[self.vA], (r * y[self.vA]).sum(dim=1))

    def gradient(self, u):
        """Algorithm "grad": least squares over the cells sharing a vertex (each once) and the
        centroids of the Dirichlet faces that share one."""
        d, N, top = self.d, self.N, int(self.vn.max())
        out = torch.empty(d, N, dtype=F64, device="cuda")
        slot = torch.arange(top, device="cuda")
        df = self.dirichlet.nonzero()[:, 0]
        far = N + df.numel()
        pts, val = torch.cat([self.cen, self.xf[df]]), torch.cat([u, self.g[df]])
        # Dirichlet faces around each vertex, as further candidates (point N + position in df)
        fvert, fpos = self.fv[df].reshape(-1), torch.arange(df.numel(), device="cuda").repeat_interleave(d)
        o = fvert.argsort()
        fvert, fpos = fvert[o], fpos[o]
        fn = torch.bincount(fvert, minlength=self.V)
        fp = torch.cat([torch.zeros(1, dtype=torch.long, device="cuda"), fn.cumsum(0)])
        ftop = int(fn.max()) if df.numel() else 0
        fslot = torch.arange(ftop, device="cuda")
        for lo in range(0, N, 200_000):
            i = torch.arange(lo, min(N, lo + 200_000), device="cuda")
            v = self.cells[i]
            pick = self.vp[v][:, :, None] + slot
            j = torch.where(slot < self.vn[v][:, :, None], self.vc[pick.clamp(max=self.vc.numel() - 1)], far)
            j = j.reshape(i.numel(), -1)
            if ftop:
                pick = fp[v][:, :, None] + fslot
                k = torch.where(fslot < fn[v][:, :, None], N + fpos[pick.clamp(max=fpos.numel() - 1)], far)
                j = torch.cat([j, k.reshape(i.numel(), -1)], dim=1)
            j = j.sort(dim=1).values
            keep = (j < far) & (j != i[:, None])
            keep[:, 1:] &= j[:, 1:] != j[:, :-1]
            j = j.clamp(max=far - 1)
            dx = torch.where(keep[:, :, None], pts[j] - self.cen[i][:, None], 0.0)
            M = dx.transpose(1, 2) @ dx
            J = dx.transpose(1, 2) @ (val[j] - u[i][:, None])[:, :, None]
            out[:, i] = torch.linalg.solve(M, J)[:, :, 0].T
        return out

    def vertices(self, u, homogeneous=False):
        uv = torch.zeros(*u.shape[:-1], self.V, dtype=F64, device="cuda").index_add_(-1, self.vA, self.alpha * u[..., self.vc])
        fixed = ~self.vdir.isnan()
        uv[..., fixed] = 0.0 if homogeneous else self.vdir[fixed]
        return uv

    def normal_gradient(self, u, homogeneous=False):
        """grad u_f . S_f by the diamond scheme; 0 on wall and Neumann faces."""
        g = torch.zeros_like(self.g) if homogeneous else self.g
        uv = self.vertices(u, homogeneous)
        ur = torch.where(self.inner, u[..., self.Rs], g)
        q = self.coef[:, 0] * (ur - u[..., self.L])
        if self.d == 3:
            c = uv[..., self.fv[:, 2]]
            q = q + self.coef[:, 1] * (uv[..., self.fv[:, 0]] - c) + self.coef[:, 2] * (uv[..., self.fv[:, 1]] - c)
        else:
            q = q + self.coef[:, 1] * (uv[..., self.fv[:, 1]] - uv[..., self.fv[:, 0]])
        return torch.where(self.inner | self.dirichlet, q, 0.0)

    def gather(self, flux):
        """Entering minus leaving."""
        out = torch.zeros(*flux.shape[:-1], self.N, dtype=F64, device="cuda").index_add_(-1, self.L, flux, alpha=-1)
        return out.index_add_(-1, self.R[self.inner], flux[..., self.inner])

    def residual(self, u, vel, diff, src, recon):
        vf = vel[:, self.L]
        vf = 0.5 * (vf + torch.where(self.inner, vel[:, self.Rs], vf))
        vn = (vf * self.S.T).sum(dim=0)
        ghost = torch.where(self.dirichlet, self.g, u[self.L])
        ul, ur = u[self.L], torch.where(self.inner, u[self.Rs], ghost)
        if recon:
            grad = self.gradient(u)
            ends = ((self.L, torch.ones_like(self.inner)), (self.Rs, self.inner))
            dl, dr = ((grad[:, c] * (self.xf - self.cen[c]).T).sum(dim=0) for c, _ in ends)
            hi, lo = u.clone(), u.clone()
            for c, other, on in ((self.L, ur, self.inner | self.dirichlet), (self.Rs, u[self.L], self.inner)):
                hi.scatter_reduce_(0, c[on], other[on], "amax")
                lo.scatter_reduce_(0, c[on], other[on], "amin")
            psi = torch.ones_like(u)
            for (c, on), inc in zip(ends, (dl, dr)):
                r = torch.where(inc > 0, (hi - u)[c] / inc, torch.where(inc < 0, (lo - u)[c] / inc, 1.0))
                psi.scatter_reduce_(0, c[on], r[on], "amin")
            ul = ul + psi[self.L] * dl
            ur = torch.where(self.inner, ur + psi[self.Rs] * dr, ur)
        flux = vn * torch.where(vn >= 0, ul, ur) - diff * self.normal_gradient(u)
        return self.gather(torch.where(self.wall, 0.0, flux)) / self.vol + src

    def poisson(self, f):
        """The discrete solution of Lap phi = f by a dense factorisation."""
        A = torch.empty(self.N, self.N, dtype=F64, device="cuda")
        for lo in range(0, self.N, 1000):
            e = torch.zeros(min(1000, self.N - lo), self.N, dtype=F64, device="cuda")
            e[torch.arange(e.shape[0]), lo + torch.arange(e.shape[0])] = 1.0
            A[:, lo:lo + e.shape[0]] = self.gather(self.normal_gradient(e, homogeneous=True)).T
        b = -self.vol * f - self.gather(self.normal_gradient(torch.zeros_like(f)))
        return torch.linalg.solve(A, b)

    def messages(self):
        w = self.coef[self.inner, 0]
        L, R, w = self.L[self.inner], self.R[self.inner], (w / w.max())[:, None]
        return lambda h: torch.zeros_like(h).index_add(0, L, w * (h[R] - h[L])).index_add(0, R, w * (h[L] - h[R]))

    def levels(self):
        """The cubic aggregates of the cells: per level (parent of each node below, size, messages)."""
        r = max(1, round((self.N / 6.0) ** (1 / 3)))
        lo, hi = self.cen.min(dim=0).values, self.cen.max(dim=0).values
        box = ((self.cen - lo) / (hi - lo) * r).floor().long().clamp(max=r - 1)
        out = []
        while True:
            ids, parent = ((box[:, 0] * r + box[:, 1]) * r + box[:, 2]).unique(return_inverse=True)
            n = ids.numel()
            box = torch.stack([ids // (r * r), ids // r % r, ids % r], dim=1)
            pairs = []
            for a in range(3):
                up = box.clone()
                up[:, a] += 1
                k = (up[:, 0] * r + up[:, 1]) * r + up[:, 2]
                at = torch.searchsorted(ids, k).clamp(max=n - 1)
                ok = (up[:, a] < r) & (ids[at] == k)
                pairs.append(torch.stack([ok.nonzero()[:, 0], at[ok]]))
            a, b = torch.cat(pairs, dim=1)
            out.append((parent, n, lambda h, a=a, b=b: (torch.zeros_like(h).index_add(0, a, h[b] - h[a])
                                                        .index_add(0, b, h[a] - h[b])) / BOX_SLOTS))
            if r <= 2:
                return out
            box, r = box >> 1, (r + 1) // 2

    def network(self, theta, scales, x, multilevel):
        """V s2 (N(f) - N(f with f0 = 0))."""
        V, s0, s1, s2 = scales
        p, o = [], 0
        for shape in [(HIDDEN, 2), (HIDDEN,)] + 3 * [(HIDDEN, 2 * HIDDEN), (HIDDEN,)] + [(HIDDEN,), (1,)]:
            p.append(theta[o:o + math.prod(shape)].reshape(shape))
            o += math.prod(shape)
        face = self.messages()
        layer = lambda k, h, msg: h + torch.relu(torch.cat([h, msg(h)], dim=1) @ p[2 + 2 * k].T + p[3 + 2 * k])  # noqa: E731
        f = torch.stack([E_OVER_EPS0 * x["dq"] * self.vol ** (2 / 3) / (V * s0), x["phi"] / (V * s1)], dim=1)
        levels = self.levels() if multilevel else []

        def net(f):
            h = layer(0, torch.relu(f @ p[0].T + p[1]), face)
            if not multilevel:
                h = layer(1, h, face)
            below, outs = h, []
            for parent, n, msg in levels:
                c = torch.zeros(n, HIDDEN, dtype=F64, device="cuda").index_add(0, parent, below)
                c = c / torch.bincount(parent, minlength=n)[:, None]
                for _ in range(HOPS):
                    c = layer(1, c, msg)
                outs.append(c)
                below = c
            add = None
            for k in range(len(levels) - 1, -1, -1):
                add = (outs[k] if add is None else outs[k] + add)[levels[k][0]]
            return layer(2, h if add is None else h + add, face) @ p[8] + p[9]

        return V * s2 * (net(f) - net(f * torch.tensor([0.0, 1.0], dtype=F64, device="cuda")))


def exact(case, seed):
    kind, dim = case["kind"], case.get("dim", 3)
    cells = 6 * case["n"] ** 3 if dim == 3 else 2 * case["n"] ** 2
    # an iterative solve's answer is fixed by its residual, not by the arithmetic; on small
    # meshes the discrete solution is at hand
    if kind == "streamer" or (kind == "poisson" and cells > 12_000):
        return None
    hosts = _host_meshes(case)
    x = _inputs(case, hosts, seed)
    if case.get("prec") == "mixed" and kind in ("transport", "gradient"):    # the inputs as the library gets them
        x = {k: v.float().double() if torch.is_tensor(v) else v for k, v in x.items()}
    bcs = _bcs(case)
    plain = _Plain(hosts[0], bcs[0] if kind == "transport" or len(bcs) == 1 else bcs[1])
    if kind == "gradient":
        return plain.gradient(x["u"])
    if kind == "poisson":
        return plain.poisson(x["f"])
    if kind == "transport":
        vel = x["vel"] if case["field"] else torch.tensor([1.0, 0.5, 0.25][:dim], dtype=F64, device="cuda")[:, None].expand(dim, plain.N)
        src = x["src"] if case["src"] else 0.0
        u = x["u"]
        for _ in range(case["steps"]):
            u0 = u
            for a in [0.5, 0.5, 1.0] if case["stages"] == 3 else [1.0]:
                u = u0 + a * x["dt"] * plain.residual(u, vel, 0.01, src, case["recon"])
        return u
    theta, scales = _network(hosts)
    theta = theta.double().to("cuda").requires_grad_(kind == "train")
    if kind == "predict":
        return plain.network(theta, scales, x, case["multilevel"])
    loss = ((plain.network(theta, scales, x, case["multilevel"]) - x["dphi"]) / (scales[0] * scales[3])).square().mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grad": theta.grad}
