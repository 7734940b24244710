"""The FP64 least-squares gradient on meshes whose cells are flat or graded, and on parts of
unequal scale packed into one index space, against Algorithm "grad" in extended precision, cell
by cell and component by component.

Tolerance of component c of a cell: each sum J_b of about 70 terms errs by at most about
70 eps S_b, S_b = sum |d_b| |u_j - u_i|, in FP64, and the inverse normal matrix, which is
accurate per component whatever the cells' aspect (scaling a coordinate scales its rows and
columns exactly), by some 1000 eps: 1e-12 sum_b |M^-1_cb| S_b covers both."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.meshgen import jittered_cube  # noqa: E402
from oracle import ls  # noqa: E402
from tests.conftest import geometry_of  # noqa: E402

BC = {t: ("neumann", 0.0) for t in (1, 2, 3, 4)} | {5: ("dirichlet", 0.25), 6: ("dirichlet", 1.5)}
TOL = 1e-12


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_00925_gb300 import build
    build.build()
    from paper_2203_00925_gb300 import capi, device
    return capi, device


def _reference(geo, u):
    """grad u [n][3] and the scale of its components' errors, in extended precision."""
    L = np.longdouble
    u = u.astype(L)
    cen = geo.cen.astype(L)
    i, j = ls.node_neighbour_pairs(geo)
    gi, gf = ls.ghost_point_pairs(geo, BC)
    dx = np.concatenate([cen[j] - cen[i], geo.xf[gf].astype(L) - cen[gi]])
    du = np.concatenate([u[j] - u[i], ls.dirichlet_values(geo, BC)[gf].astype(L) - u[gi]])
    i = np.concatenate([i, gi])
    M, J, S = np.zeros((geo.n_cell, 3, 3), L), np.zeros((geo.n_cell, 3), L), np.zeros((geo.n_cell, 3), L)
    np.add.at(J, i, dx * du[:, None])
    np.add.at(M, i, dx[:, :, None] * dx[:, None, :])
    np.add.at(S, i, np.abs(dx) * np.abs(du)[:, None])
    d = 1 / np.sqrt(np.einsum("nkk->nk", M))           # to unit diagonal
    M = M * d[:, :, None] * d[:, None, :]
    inv = np.linalg.inv(M.astype(np.float64)).astype(L)
    for _ in range(2):                                 # Newton steps to extended precision
        inv = inv @ (2 * np.eye(3, dtype=L) - M @ inv)
    inv = inv * d[:, :, None] * d[:, None, :]
    return (inv @ J[:, :, None])[:, :, 0], (np.abs(inv) @ S[:, :, None])[:, :, 0]


def _mapped(k, seed, f, jitter=0.2):
    """A jittered cube with its points moved by f, and a field smooth in the cube's coordinates."""
    m = jittered_cube(k, seed=seed, jitter=jitter)
    s = m.xyz[m.cells].mean(axis=1)
    m.xyz = np.ascontiguousarray(f(m.xyz))
    return m, np.cos(3 * s[:, 0]) * np.sin(2 * s[:, 1] + s[:, 2]) + s[:, 2]


def _check(got, geo, u, name):
    want, scale = _reference(geo, u)
    err = np.abs(got.T - want.astype(np.float64)) / scale.astype(np.float64)
    assert (err <= TOL).all(), (name, err.max(axis=0), (err > TOL).sum(axis=0))


def _layer(x, z):
    return np.concatenate([x[:, :2], z[:, None]], axis=1)


MAPS = {
    "isotropic": lambda x: x,
    "flat 1e2": lambda x: x * [1.0, 1.0, 1e-2],
    "flat 1e4": lambda x: x * [1.0, 1e-4, 1.0],
    "flat 1e6": lambda x: x * [1e6, 1.0, 1.0],
    "needles": lambda x: x * [1.0, 1e-5, 1e-5],
    "layer at 0": lambda x: _layer(x, x[:, 2] ** 3 / 100),
    "layer at 1": lambda x: _layer(x, 1 - (1 - x[:, 2]) ** 3),
    "geometric layer": lambda x: _layer(x, np.expm1(6 * x[:, 2]) / np.expm1(6.0)),
    "to the corner": lambda x: x ** 8,
    "far away": lambda x: x + [9.0, -5.0, 0.0],
    "about the origin": lambda x: (x - 0.5) * [1.0, 1.0, 1e-3],
}


@pytest.mark.parametrize("name", MAPS)
def test_gradient_of_flat_and_graded_cells(dev, name):
    capi, device = dev
    m, u = _mapped(10, 7, MAPS[name], jitter=0.0 if name == "to the corner" else 0.2)   # (would turn cells over)
    geo = geometry_of(m)
    dm = device.DeviceMesh(m, [BC], prec="fp64")
    out = dm.empty(3, dm.n_cell)
    capi.fvgb_gradient(dm.handle, 0, dm.to_device(u), out)
    _check(dm.to_host(out), geo, u, name)
    dm.free()


@pytest.mark.parametrize("size", [1e-9, 1e-6, 1e-2, 1e3, 1e6, 1e9])
def test_gradient_beside_a_part_of_another_scale(dev, size):
    """Each part to the same tolerance, and with the bits that it has alone."""
    capi, device = dev
    parts = [_mapped(6, 20, lambda x: x), _mapped(7, 21, lambda x: x * size), _mapped(6, 22, lambda x: x + 3.0)]
    meshes = [m for m, _ in parts]
    dm = device.DeviceMesh(meshes, [[BC]] * 3, prec="fp64", ensemble=True)
    out = dm.empty(3, dm.n_cell)
    capi.fvgb_gradient(dm.handle, 0, dm.to_device(np.concatenate([u for _, u in parts])), out)
    got = dm.to_host(out)
    dm.free()
    at = 0
    for m, u in parts:
        mine = got[:, at:at + m.n_cell]
        _check(mine, geometry_of(m), u, size)
        one = device.DeviceMesh(m, [BC], prec="fp64")
        alone = one.empty(3, one.n_cell)
        capi.fvgb_gradient(one.handle, 0, one.to_device(u), alone)
        assert np.array_equal(one.to_host(alone), mine)
        one.free()
        at += m.n_cell
