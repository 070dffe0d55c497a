"""Grids with a few nodes in x and y and more planes than short chunks could cover with 65535 CTAs, on the
kernels that take two steps per pass, forward and transposed, and the transposed step on spacings
more than 16 apart: against single steps and the plain kernel."""
import pytest
import torch

from paper_2211_15634_gb300 import api

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def fields(shape, dtype, n=4):
    g = torch.Generator(device="cuda").manual_seed(5)
    return [0.5 + torch.rand(shape, generator=g, device="cuda", dtype=dtype) for _ in range(n)]


@pytest.mark.parametrize("dtype,nt", [(torch.float64, 4), (torch.float32, 4)])
def test_forward_pairs(launch_override, dtype, nt):
    T0, C = fields((2200000, 3, 4), dtype, 2)
    inv, dt, scaled = (2.0, 2.0, 2.0), 0.01, dtype == torch.float64
    if scaled:
        C = api.scale_ci(C, 1.0, dt, inv)
    want = api.run(T0.clone(), T0.clone(), C, 1.0, dt, inv, nt, ci_scaled=scaled)
    if not scaled:
        launch_override(kchunk2=4)  # a size that the default leaves to single steps
    got = api.run(T0.clone(), T0.clone(), C, 1.0, dt, inv, nt, ci_scaled=scaled, temporal2=True)
    assert torch.equal(got, want)
    assert api.device_error() == 0


def test_transposed_pairs():
    y, S1, S0, C = fields((2200000, 3, 4), torch.float32)
    inv, dt = (2.0, 2.5, 3.0), 0.01
    a, b, ca = torch.empty_like(y), torch.empty_like(y), torch.zeros_like(y)
    api.adjoint(a, ca, y, S1, C, 1.0, dt, inv)
    api.adjoint(b, ca, a, S0, C, 1.0, dt, inv)
    got, cb = torch.empty_like(y), torch.zeros_like(y)
    api.adjoint2(got, cb, y, S1, S0, C, 1.0, dt, inv)
    assert torch.equal(got, b) and torch.equal(cb, ca)
    assert api.device_error() == 0


def test_transposed_step_on_far_spacings(launch_override):
    y, T, C = fields((1200000, 3, 4), torch.float64, 3)
    got = []
    for plain in (0, 1):
        launch_override(adj_plain=plain)
        tbar, cbar = torch.empty_like(y), torch.zeros_like(y)
        api.adjoint(tbar, cbar, y, T, C, 1.0, 0.01, (3.0, 0.1, 2.0))
        got.append((tbar, cbar))
    for a, b in zip(*got):  # a few roundings of values below 2
        assert float((a - b).abs().max()) <= 1e-14
    assert api.device_error() == 0
