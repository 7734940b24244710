"""The FP64 least-squares gradient's fixed-point sums (3D meshes of at least one tile of 128
cells) against Algorithm "grad" in extended precision, cell by cell.

Tolerance per cell: the direct FP64 sum of about 70 terms errs by at most about 70 eps times
sum |d| |u_j - u_i| before the normal matrix's inverse M^-1, itself accurate to some 100 eps
on these meshes; 1e-12 of |M^-1| sum |d| |u_j - u_i| covers both, and a unit taken from the
tile's range instead of the cell's would exceed it by orders of magnitude on the steep
fields."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.meshgen import gaussian, jittered_cube  # noqa: E402
from oracle import ls  # noqa: E402
from tests.conftest import geometry_of  # noqa: E402

BC = {t: ("neumann", 0.0) for t in (1, 2, 3, 4)} | {5: ("dirichlet", 0.25), 6: ("dirichlet", 1.5)}


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_00925_gb300 import build
    build.build()
    from paper_2203_00925_gb300 import capi, device
    return capi, device


def _reference(geo, u):
    """grad u and the scale of its error, in extended precision."""
    L = np.longdouble
    u = u.astype(L)
    cen = geo.cen.astype(L)
    i, j = ls.node_neighbour_pairs(geo)
    gi, gf = ls.ghost_point_pairs(geo, BC)
    dx = np.concatenate([cen[j] - cen[i], geo.xf[gf].astype(L) - cen[gi]])
    du = np.concatenate([u[j] - u[i], ls.dirichlet_values(geo, BC)[gf].astype(L) - u[gi]])
    i = np.concatenate([i, gi])
    M, J, scale = np.zeros((geo.n_cell, 3, 3), L), np.zeros((geo.n_cell, 3), L), np.zeros(geo.n_cell, L)
    np.add.at(J, i, dx * du[:, None])
    np.add.at(M, i, dx[:, :, None] * dx[:, None, :])
    np.add.at(scale, i, np.abs(dx).sum(axis=1) * np.abs(du))
    inv = np.linalg.inv(M.astype(np.float64)).astype(L)
    for _ in range(2):                       # Newton steps to extended precision
        inv = inv @ (2 * np.eye(3, dtype=L) - M @ inv)
    return (inv @ J[:, :, None])[:, :, 0], np.abs(inv).sum(axis=(1, 2)) * scale


def _fields(cen, rng):
    smooth = np.cos(3 * cen[:, 0]) * np.sin(2 * cen[:, 1] + cen[:, 2])
    return {"smooth": smooth,
            "offset": 1e6 + smooth,                                    # differences far below the values
            "steep": gaussian(cen, (0.4, 0.6, 0.5), 0.05, 1e16, 1e9),   # decades inside a tile
            "noise": rng.normal(size=cen.shape[0]),
            "step": np.where(cen[:, 0] > 0.5, 1e30, -1e-30),
            "large": 1e300 * smooth,
            "small": 1e-290 * smooth}


@pytest.mark.parametrize("k", [3, 5, 11])
def test_gradient_fixed_point_cell_by_cell(dev, k):
    capi, device = dev
    m = jittered_cube(k, seed=60 + k)
    geo = geometry_of(m)
    dm = device.DeviceMesh(m, [BC], prec="fp64")
    out = dm.empty(3, dm.n_cell)
    for name, u in _fields(geo.cen, np.random.default_rng(k)).items():
        capi.fvgb_gradient(dm.handle, 0, dm.to_device(u), out)
        want, scale = _reference(geo, u)
        err = np.abs(dm.to_host(out).T - want.astype(np.float64)).max(axis=1)
        bad = err > 1e-12 * scale.astype(np.float64) + 1e-300
        assert not bad.any(), (name, int(bad.sum()), float((err / np.maximum(scale.astype(np.float64), 1e-300)).max()))
    dm.free()


def test_gradient_fixed_point_not_finite(dev):
    """A NaN or infinity reaches exactly the cells around it, as in the direct sum."""
    capi, device = dev
    m = jittered_cube(6, seed=70)
    geo = geometry_of(m)
    dm = device.DeviceMesh(m, [BC], prec="fp64")
    u = np.cos(2 * geo.cen[:, 0])
    i, j = ls.node_neighbour_pairs(geo)
    clean, out = dm.empty(3, dm.n_cell), dm.empty(3, dm.n_cell)
    capi.fvgb_gradient(dm.handle, 0, dm.to_device(u), clean)
    for bad in (np.nan, np.inf):
        v = u.copy()
        v[400] = bad
        capi.fvgb_gradient(dm.handle, 0, dm.to_device(v), out)
        hit = np.zeros(geo.n_cell, dtype=bool)
        hit[i[j == 400]] = True
        hit[400] = True
        got = dm.to_host(out)
        assert (np.isfinite(got).all(axis=0) == ~hit).all()
        np.testing.assert_allclose(got[:, ~hit], dm.to_host(clean)[:, ~hit], rtol=1e-11, atol=1e-11)
    dm.free()


def test_gradient_fixed_point_parts_in_one_tile(dev):
    """Small meshes of different scale packed into one index space share tiles: each as alone."""
    capi, device = dev
    meshes = [jittered_cube(3, seed=80), jittered_cube(4, seed=81), jittered_cube(3, seed=82)]
    meshes[1].xyz *= 1e-3
    dm = device.DeviceMesh(meshes, [[BC]] * 3, prec="fp64", ensemble=True)
    geos = [geometry_of(m) for m in meshes]
    us = [np.cos(3 * g.cen[:, 0] / s) + g.cen[:, 2] / s for g, s in zip(geos, (1.0, 1e-3, 1.0))]
    out = dm.empty(3, dm.n_cell)
    capi.fvgb_gradient(dm.handle, 0, dm.to_device(np.concatenate(us)), out)
    got = dm.to_host(out)
    at = 0
    for g, u in zip(geos, us):
        want, scale = _reference(g, u)
        err = np.abs(got[:, at:at + g.n_cell].T - want.astype(np.float64)).max(axis=1)
        assert (err <= 1e-12 * scale.astype(np.float64)).all()
        at += g.n_cell
    dm.free()
