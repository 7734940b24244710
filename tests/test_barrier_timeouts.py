"""Every bounded grid barrier made to run out by the test hook (one block never arrives, the limit
cut to a few milliseconds), without a GPU fault: the CG in its own launches, host-driven and
in a captured step; the one-launch steps of a small mesh; and what a later call sees."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.meshgen import jittered_cube, jittered_square  # noqa: E402
from synth.workloads import StreamerCase  # noqa: E402

PHI3 = {1: ("neumann", 0.0), 2: ("neumann", 0.0), 3: ("neumann", 0.0), 4: ("neumann", 0.0),
        5: ("dirichlet", 0.0), 6: ("dirichlet", 100.0)}
NEU3 = {t: ("neumann", 0.0) for t in range(1, 7)}
CASE = StreamerCase(V=100.0, peak=1e12, background=1e9, sigma=0.2)


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_00925_gb300 import build
    build.build()
    from paper_2203_00925_gb300 import capi, device
    return capi, device


def _status(capi, fn, *args, **kw):
    try:
        fn(*args, **kw)
    except capi.FvgbError as e:
        return e.status
    return capi.FVGB_OK


def _mesh(capi, device, prec):
    m = jittered_cube(8, seed=11)
    dm = device.DeviceMesh(m, [NEU3, PHI3], prec=prec)
    inner_prec = capi.FVGB_FP64 if prec == "fp64" else capi.FVGB_FP32
    f = dm.to_device(np.sin(3 * m.xyz[m.cells].mean(axis=1)[:, 0]) * 1e3, torch.float64)
    phi = torch.zeros(dm.n_cell, dtype=torch.float64, device="cuda")
    ne = dm.to_device(CASE.initial(m)[0])

    def solve(inner):
        phi.zero_()
        return _status(capi, capi.fvgb_poisson_solve, dm.handle, 1, f, phi,
                       capi.solve_opts(rtol=1e-8, prec=inner_prec, inner=inner))

    def step(inner):
        phi.zero_()
        sp = capi.streamer_params(mu=CASE.mu, A=CASE.A, B=CASE.B, De=CASE.De, dt=1e-12,
                                  solve=capi.solve_opts(rtol=1e-8, prec=inner_prec, inner=inner))
        capi.fvgb_set_graph_mode(dm.handle, True)
        st = _status(capi, capi.fvgb_streamer_step, dm.handle, sp, ne.clone(), 1.01 * ne, phi, None, 2)
        capi.fvgb_set_graph_mode(dm.handle, False)
        return st

    return dm, solve, step


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_timeout_of_separate_launches(dev, prec):
    capi, device = dev
    dm, solve, step = _mesh(capi, device, prec)
    capi.fvgb_stats_enable(dm.handle, True)         # the CG in its own launches
    capi.fvgb_test_barrier(dm.handle, 1, 5.0)
    assert solve(0) == capi.FVGB_ETIMEOUT
    assert step(0) == capi.FVGB_ETIMEOUT
    _status(capi, capi.fvgb_sync, dm.handle)        # what the transport latched on that potential
    capi.fvgb_test_barrier(dm.handle, -1, 0.0)
    assert solve(0) == capi.FVGB_OK
    assert step(0) == capi.FVGB_OK
    dm.free()


@pytest.mark.parametrize("launches", [False, True])
def test_multigrid_after_a_timeout(dev, launches):
    """A multigrid solve runs no grid barrier: a timeout reported before is not its own."""
    capi, device = dev
    dm, solve, step = _mesh(capi, device, "mixed")
    capi.fvgb_stats_enable(dm.handle, launches)
    for call in (solve, step):
        capi.fvgb_test_barrier(dm.handle, 1, 5.0)
        assert solve(0) == capi.FVGB_ETIMEOUT
        capi.fvgb_test_barrier(dm.handle, -1, 0.0)
        assert call(2) == capi.FVGB_OK
    dm.free()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_timeout_of_the_one_launch_steps(dev, prec):
    """The steps of a small mesh latch the timeout; fvgb_sync or the next solve reports it once."""
    capi, device = dev
    m = jittered_square(20)
    dm = device.DeviceMesh(m, [{1: ("wall", 0.0), 2: ("neumann", 0.0), 3: ("dirichlet", 0.3), 4: ("wall", 0.0)}], prec=prec)
    tc = capi.tcoef(vel_const=(1.0, -0.5), diff=0.1)
    u0 = dm.to_device(1.0 + m.xyz[m.cells].mean(axis=1)[:, 0])
    f = torch.ones(dm.n_cell, dtype=torch.float64, device="cuda")
    phi = torch.zeros_like(f)
    want = u0.clone()
    capi.fvgb_fv_step(dm.handle, tc, want, 1e-5, 3)
    capi.fvgb_sync(dm.handle)

    def late():
        capi.fvgb_test_barrier(dm.handle, 2, 5.0)
        capi.fvgb_fv_step(dm.handle, tc, u0.clone(), 1e-5, 3)
        capi.fvgb_test_barrier(dm.handle, -1, 0.0)

    late()
    assert _status(capi, capi.fvgb_sync, dm.handle) == capi.FVGB_ETIMEOUT
    assert _status(capi, capi.fvgb_sync, dm.handle) == capi.FVGB_OK
    late()
    opts = capi.solve_opts(rtol=1e-8)
    assert _status(capi, capi.fvgb_poisson_solve, dm.handle, 0, f, phi, opts) == capi.FVGB_ETIMEOUT
    assert _status(capi, capi.fvgb_poisson_solve, dm.handle, 0, f, phi.zero_(), opts) == capi.FVGB_OK
    got = u0.clone()
    capi.fvgb_fv_step(dm.handle, tc, got, 1e-5, 3)
    assert _status(capi, capi.fvgb_sync, dm.handle) == capi.FVGB_OK
    assert torch.equal(got, want)
    dm.free()


def test_captured_step_reports_a_latched_timeout(dev):
    """A latched word met at the end of a captured step is reported as what it is."""
    capi, device = dev
    dm, _, step = _mesh(capi, device, "mixed")
    u = dm.to_device(np.ones(dm.n_cell))
    tc = capi.tcoef(vel_const=(1.0, -0.5, 0.2), diff=0.1)
    assert step(0) == capi.FVGB_OK
    for bad, want in ((None, capi.FVGB_ETIMEOUT), (float("nan"), capi.FVGB_ENONFINITE)):
        if bad is None:
            capi.fvgb_test_barrier(dm.handle, 2, 5.0)
            capi.fvgb_fv_step(dm.handle, tc, u, 1e-6, 2)
            capi.fvgb_test_barrier(dm.handle, -1, 0.0)
        else:
            u[7] = bad
            capi.fvgb_fv_step(dm.handle, tc, u, 1e-6, 2)
        assert step(0) == want
        assert step(0) == capi.FVGB_OK
    dm.free()
