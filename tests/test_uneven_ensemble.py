"""Ensembles of parts of very unequal size: small parts share blocks of the solver and are solved
one after another, large ones get blocks of their own. Every part to its own tolerance, in one
launch and in separate launches.

The residual formed anew by fvgb_poisson_apply agrees with the reported one to the rounding of
its terms: at most ||A|| ||x|| <= 1e5 ||b|| on these meshes, times 2^-53 times their number (30)
gives 4e-10 relative to ||b||."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.meshgen import jittered_cube, jittered_square  # noqa: E402

RTOL, ROUND = 1e-8, 4e-10
BC2 = {1: ("dirichlet", 0.0), 2: ("dirichlet", 3.0), 3: ("neumann", 0.0), 4: ("neumann", 0.0)}
BC3 = BC2 | {5: ("neumann", 0.0), 6: ("neumann", 0.0)}
SIZES = {"one large": (3, [14] + [1, 2, 3, 4] * 12), "two large": (3, [2] * 30 + [11, 13] + [3] * 30),
         "equal": (3, [3] * 128), "2D": (2, [60] + [1, 2, 5, 7] * 25)}


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_00925_gb300 import build
    build.build()
    from paper_2203_00925_gb300 import capi, device
    return capi, device


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", SIZES)
def test_parts_that_share_blocks(dev, name, prec):
    capi, device = dev
    dim, sizes = SIZES[name]
    cubes = {k: jittered_cube(k, seed=40 + k) if dim == 3 else jittered_square(k) for k in set(sizes)}
    meshes = [cubes[k] for k in sizes]
    zero = 5                                     # a part with nothing to solve
    flat = {t: (k, 0.0) for t, (k, _) in (BC3 if dim == 3 else BC2).items()}
    bcs = [[flat if i == zero else BC3 if dim == 3 else BC2] for i in range(len(meshes))]
    dm = device.DeviceMesh(meshes, bcs, prec=prec, ensemble=True)
    f = dm.to_device(np.concatenate([np.zeros(m.n_cell) if i == zero else 50.0 * (i % 7 + 1) * np.cos(
        3 * m.xyz[m.cells].mean(axis=1)[:, 0]) for i, m in enumerate(meshes)]), torch.float64)
    opts = capi.solve_opts(rtol=RTOL, prec=capi.FVGB_FP64 if prec == "fp64" else capi.FVGB_FP32)
    cut = np.r_[dm.part_begin[:-1], dm.n_cell].astype(int)
    phi, b, y = (torch.zeros(dm.n_cell, dtype=torch.float64, device="cuda") for _ in range(3))
    for launches in (False, True):
        capi.fvgb_stats_enable(dm.handle, launches)
        phi.zero_()
        _, info = capi.fvgb_poisson_solve(dm.handle, 0, f, phi, opts)
        rel, outer, inner = capi.fvgb_solve_parts(dm.handle, dm.n_part)
        capi.fvgb_poisson_rhs(dm.handle, 0, f, b)
        capi.fvgb_poisson_apply(dm.handle, 0, phi, y)
        capi.fvgb_sync(dm.handle)
        hb, hr = dm.to_host(b), dm.to_host(b - y)
        for p, (i, j) in enumerate(zip(cut[:-1], cut[1:])):
            if p == zero:
                assert outer[p] == inner[p] == 0 and not dm.to_host(phi)[i:j].any()
                continue
            want = np.linalg.norm(hr[i:j]) / np.linalg.norm(hb[i:j])
            assert rel[p] <= RTOL and abs(want - rel[p]) <= ROUND, (p, want, rel[p])
            assert outer[p] >= 1 and inner[p] >= outer[p]
        assert info.outer_its == outer.max() and info.inner_its_total == inner.max()
    # a block that never arrives, the first (a large part's or its own) and the last (shared)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for launches in (False, True):
        capi.fvgb_stats_enable(dm.handle, launches)
        for block in (0, sms - 1 if name in ("one large", "2D") else 0):
            capi.fvgb_test_barrier(dm.handle, block, 5.0)
            with pytest.raises(capi.FvgbError) as e:
                capi.fvgb_poisson_solve(dm.handle, 0, f, phi.zero_(), opts)
            assert e.value.status == capi.FVGB_ETIMEOUT
            capi.fvgb_test_barrier(dm.handle, -1, 0.0)
    dm.free()


@pytest.mark.parametrize("n,prec,one", [(707, "fp64", True), (708, "fp64", False), (708, "mixed", True)])
def test_line_of_the_one_launch_solve(dev, n, prec, one):
    """FP64 ensembles of more than 1,000,000 cells a part on average run separate launches; the
    launches are counted: some ten a solve, or several an outer step."""
    capi, device = dev
    m = jittered_square(n)
    dm = device.DeviceMesh([m, m], [[BC2], [BC2]], prec=prec, ensemble=True)
    f = dm.to_device(np.tile(np.cos(3 * m.xyz[m.cells].mean(axis=1)[:, 0]), 2), torch.float64)
    phi, b, y = (torch.zeros(dm.n_cell, dtype=torch.float64, device="cuda") for _ in range(3))
    capi.fvgb_stats_get(dm.handle, reset=True)
    _, info = capi.fvgb_poisson_solve(dm.handle, 0, f, phi, capi.solve_opts(
        rtol=1e-4, prec=capi.FVGB_FP64 if prec == "fp64" else capi.FVGB_FP32))
    launches = capi.fvgb_stats_get(dm.handle, reset=True)["kernel_launches"]
    assert info.outer_its >= 2 and (launches <= 10) == one and (launches >= 4 * info.outer_its) != one
    capi.fvgb_poisson_rhs(dm.handle, 0, f, b)
    capi.fvgb_poisson_apply(dm.handle, 0, phi, y)
    for half in (slice(0, dm.n_cell // 2), slice(dm.n_cell // 2, None)):
        assert torch.linalg.norm((b - y)[half]) <= 1.0001e-4 * torch.linalg.norm(b[half])
    dm.free()
