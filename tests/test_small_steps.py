"""fvgb_fv_step on small meshes runs all its stages in one launch (csrc/small.cu): the bits of
the three-kernel path, which a call of a single stage takes.

Sizes: fewer cells than blocks, one and several warps a block, the last size within the
kernel's 128 cells a block (19,456 cells on 152 SMs) and the first beyond it. A three-stage step
is compared with its stages formed from fvgb_fv_residual; the update rounds
u + a dt res differently there, at most a few ulp a stage."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.meshgen import jittered_cube, jittered_square  # noqa: E402

BC2 = {1: ("wall", 0.0), 2: ("neumann", 0.0), 3: ("dirichlet", 0.3), 4: ("wall", 0.0)}
BC3 = BC2 | {5: ("dirichlet", 0.7), 6: ("neumann", 0.0)}
SIZES = [(2, 1), (2, 7), (2, 50), (2, 98), (2, 99), (3, 2), (3, 6), (3, 14), (3, 15)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_00925_gb300 import build
    build.build()
    from paper_2203_00925_gb300 import capi, device
    return capi, device


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("dim,n", SIZES)
def test_steps_in_one_launch_are_the_same_bits(dev, dim, n, prec):
    capi, device = dev
    m = jittered_square(n) if dim == 2 else jittered_cube(n, seed=9)
    dm = device.DeviceMesh(m, [BC2 if dim == 2 else BC3], prec=prec)
    rng = np.random.default_rng(n)
    u0 = dm.to_device(rng.random(m.n_cell) + 0.5)
    vel, src = dm.to_device(rng.normal(size=(dim, m.n_cell))), dm.to_device(rng.normal(size=m.n_cell))
    dt = 0.01 * m.h ** 2
    for kw in ({"vel": vel, "src": src, "diff": 0.2}, {"vel_const": (1.0, -0.5, 0.25)[:dim], "diff": 0.2},
               {"vel": vel, "src": src, "diff": 0.0}):
        tc = capi.tcoef(**kw)
        one, many = u0.clone(), u0.clone()
        for _ in range(5):
            capi.fvgb_fv_step(dm.handle, tc, one, dt, 1)
        capi.fvgb_fv_step(dm.handle, tc, many, dt, 5)
        capi.fvgb_sync(dm.handle)
        assert torch.equal(one, many), kw.keys()
        got = u0.clone()
        capi.fvgb_fv_step(dm.handle, tc, got, dt, 1, [0.5, 0.5, 1.0])
        uk, res = u0.clone(), dm.empty(dm.n_cell)
        for a in (0.5, 0.5, 1.0):
            capi.fvgb_fv_residual(dm.handle, tc, uk, res)
            uk = u0 + a * dt * res
        eps = torch.finfo(dm.real).eps
        assert (got - uk).abs().max() <= 16 * eps * uk.abs().max()
    dm.free()


def test_steps_in_one_launch_latch_not_finite(dev):
    capi, device = dev
    m = jittered_square(20)
    dm = device.DeviceMesh(m, [BC2], prec="fp64")
    u = dm.to_device(np.ones(m.n_cell))
    u[11] = float("inf")
    capi.fvgb_fv_step(dm.handle, capi.tcoef(vel_const=(1.0, 0.5), diff=0.1), u, 1e-5, 4)
    with pytest.raises(capi.FvgbError) as e:
        capi.fvgb_sync(dm.handle)
    assert e.value.status == capi.FVGB_ENONFINITE
    dm.free()
