"""fvgb_poisson_solve: in one launch (a CG inner solve of at most 600,000 cells, every ensemble)
against the loop of separate launches, which a mesh whose CG is being timed takes.

Sizes: fewer cells than blocks, rows that do not fill a block, the last size within the line
and the first beyond it. Both stop by the same test on the FP64 residual; the residual formed
anew by fvgb_poisson_apply agrees with the reported one to the rounding of its terms: the rows'
terms are at most ||A|| ||x|| <= 1e5 ||b|| on these meshes, times 2^-53 times their number (30)
gives 4e-10 relative to ||b||, so the recomputed residual is held to rtol = 1e-8 plus that."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.meshgen import gaussian, jittered_cube  # noqa: E402

BC = {1: ("dirichlet", 0.0), 2: ("dirichlet", 3.0), 3: ("neumann", 0.0), 4: ("neumann", 0.0),
      5: ("neumann", 0.0), 6: ("neumann", 0.0)}
RTOL, ROUND = 1e-8, 4e-10


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_00925_gb300 import build
    build.build()
    from paper_2203_00925_gb300 import capi, device
    return capi, device


def _solve(capi, dm, f, opts, launches):
    capi.fvgb_stats_enable(dm.handle, launches)
    phi = torch.zeros(dm.n_cell, dtype=torch.float64, device="cuda")
    _, info = capi.fvgb_poisson_solve(dm.handle, 0, f, phi, opts)
    parts = capi.fvgb_solve_parts(dm.handle, dm.n_part)
    capi.fvgb_stats_enable(dm.handle, False)
    return phi, info, parts


def _residual(capi, dm, f, phi):
    b, y = torch.empty_like(phi), torch.empty_like(phi)
    capi.fvgb_poisson_rhs(dm.handle, 0, f, b)
    capi.fvgb_poisson_apply(dm.handle, 0, phi, y)
    capi.fvgb_sync(dm.handle)
    b, r = dm.to_host(b), dm.to_host(b - y)
    cut = np.r_[dm.part_begin[:-1], dm.n_cell].astype(int)
    nrm = lambda v: np.array([np.linalg.norm(v[i:j]) for i, j in zip(cut[:-1], cut[1:])])  # noqa: E731
    return nrm(r), nrm(b)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [2, 5, 14, 46, 47])
def test_one_launch_and_separate_launches(dev, n, prec):
    capi, device = dev
    m = jittered_cube(n, seed=3)
    dm = device.DeviceMesh(m, [BC], prec=prec)
    cen = m.xyz[m.cells].mean(axis=1)
    f = dm.to_device(-1e3 * gaussian(cen, (0.5, 0.5, 0.5), 0.2), torch.float64)
    opts = capi.solve_opts(rtol=RTOL, prec=capi.FVGB_FP64 if prec == "fp64" else capi.FVGB_FP32)
    outers = []
    for launches in (False, True):
        phi, info, (rel, outer, inner) = _solve(capi, dm, f, opts, launches)
        r, b = _residual(capi, dm, f, phi)
        assert rel[0] <= RTOL and abs(r[0] / b[0] - rel[0]) <= ROUND
        assert outer[0] == info.outer_its >= 1 and inner[0] >= outer[0]
        outers.append(int(outer[0]))
    assert abs(outers[0] - outers[1]) <= 1
    dm.free()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_ensemble_with_a_part_that_has_nothing_to_solve(dev, prec):
    capi, device = dev
    meshes = [jittered_cube(k, seed=40 + k) for k in (2, 9, 5, 12)]
    bcs = [[{t: (k, 0.0) for t, (k, _) in BC.items()}] if i == 2 else [BC] for i in range(4)]
    dm = device.DeviceMesh(meshes, bcs, prec=prec, ensemble=True)
    fs = [np.zeros(m.n_cell) if i == 2 else 50.0 * (i + 1) * np.cos(3 * m.xyz[m.cells].mean(axis=1)[:, 0])
          for i, m in enumerate(meshes)]
    f = dm.to_device(np.concatenate(fs), torch.float64)
    opts = capi.solve_opts(rtol=RTOL, prec=capi.FVGB_FP64 if prec == "fp64" else capi.FVGB_FP32)
    for launches in (False, True):
        phi, _, (rel, outer, inner) = _solve(capi, dm, f, opts, launches)
        r, b = _residual(capi, dm, f, phi)
        live = np.array([0, 1, 3])
        assert np.all(rel <= RTOL) and np.all(np.abs(r[live] / b[live] - rel[live]) <= ROUND)
        assert outer[2] == 0 and inner[2] == 0 and np.all(outer[live] >= 1)
        lo, hi = dm.part_begin[2], dm.part_begin[3]
        assert not dm.to_host(phi)[int(lo):int(hi)].any()
    dm.free()


@pytest.mark.parametrize("n,prec", [(4, "fp64"), (5, "mixed"), (24, "mixed"), (57, "fp64"), (100, "mixed")])
def test_multigrid_levels_of_every_row_width(dev, n, prec):
    """inner = 2: the dense solve alone, small levels, and levels that fill the chip, whose rows
    are summed by 1, 2, 4 and 16 threads."""
    capi, device = dev
    m = jittered_cube(n, seed=3)
    dm = device.DeviceMesh(m, [BC], prec=prec)
    cen = m.xyz[m.cells].mean(axis=1)
    f = dm.to_device(-1e3 * gaussian(cen, (0.5, 0.5, 0.5), 0.2), torch.float64)
    opts = capi.solve_opts(rtol=RTOL, prec=capi.FVGB_FP64 if prec == "fp64" else capi.FVGB_FP32, inner=2)
    phi, info, (rel, outer, inner) = _solve(capi, dm, f, opts, False)
    r, b = _residual(capi, dm, f, phi)
    assert rel[0] <= RTOL and abs(r[0] / b[0] - rel[0]) <= ROUND
    assert 1 <= outer[0] <= 40 and inner[0] == 2 * outer[0]
    dm.free()
