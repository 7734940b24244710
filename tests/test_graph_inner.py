"""A captured streamer step belongs to the inner solve it was captured with: the same arrays and
parameters with another inner solve are captured anew, and give what the host-driven step
gives."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from synth.meshgen import jittered_cube  # noqa: E402
from synth.workloads import StreamerCase  # noqa: E402


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_00925_gb300 import build
    build.build()
    from paper_2203_00925_gb300 import capi, device
    return capi, device


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_graph_follows_the_inner_solve(dev, prec):
    capi, device = dev
    m = jittered_cube(9, seed=201)
    case = StreamerCase(sigma=0.15, peak=1e13)
    dm = device.DeviceMesh(m, [case.bc_ne(), case.bc_phi()], prec=prec)
    ne0 = dm.to_device(case.initial(m)[0])
    ne, ni = ne0.clone(), ne0.clone()
    phi = torch.zeros(dm.n_cell, dtype=torch.float64, device="cuda")

    def step(inner, graph):
        ne.copy_(ne0)
        ni.copy_(1.02 * ne0)
        phi.zero_()
        sp = capi.streamer_params(mu=case.mu, A=case.A, B=case.B, De=case.De, dt=2e-9, solve=capi.solve_opts(
            rtol=1e-9, prec=capi.FVGB_FP64 if prec == "fp64" else capi.FVGB_FP32, inner=inner))
        capi.fvgb_set_graph_mode(dm.handle, graph)
        info = capi.fvgb_streamer_step(dm.handle, sp, ne, ni, phi, None, 1)[0]
        torch.cuda.synchronize()
        return info["outer_its"], info["inner_its_total"], phi.clone()

    want = {inner: step(inner, False) for inner in (0, 1, 2)}
    for inner in (1, 2):
        assert want[inner][1] == inner * want[inner][0]
    assert want[0][1] > 2 * want[0][0]
    for inner in (0, 2, 1, 0, 2):
        outer, its, p = step(inner, True)
        assert (outer, its) == want[inner][:2], inner
        assert torch.equal(p, want[inner][2])
    dm.free()
