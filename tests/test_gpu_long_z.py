"""Grids with a few nodes in x and y and more planes than short chunks could cover with 65535 CTAs:
the staged kernels, in loops, single steps and transposed steps, against the plain ones."""
import pytest
import torch

from paper_2211_15634_gb300 import api

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def fields(nx, ny, nz, dtype):
    g = torch.Generator(device="cuda").manual_seed(nx)
    T0, C, y = (torch.rand((nz, ny, nx), generator=g, device="cuda", dtype=dtype) for _ in range(3))
    return 1.2 + 0.5 * T0, 0.5 + 0.5 * C, y - 0.5


@pytest.mark.parametrize("dtype,nx,nz", [(torch.float64, 3, 800001), (torch.float64, 4, 700000),
                                         (torch.float64, 5, 2000001), (torch.float32, 3, 900001),
                                         (torch.float32, 5, 3000001), (torch.float32, 4, 600000)])
def test_forward_and_transposed_steps(launch_override, dtype, nx, nz):
    ny = 3
    T0, C, y = fields(nx, ny, nz, dtype)
    inv = (2.0, 2.5, 3.0)
    dt = 0.01
    got = []
    for plain in (0, 1):
        launch_override(step_plain=plain, adj_plain=plain)
        T = T0.clone()
        loop = api.run(T, T.clone(), C, 1.0, dt, inv, 3)
        one = api.step(T0.clone(), T0, C, 1.0, dt, inv)
        tbar, cbar = torch.empty_like(T0), torch.zeros_like(T0)
        api.adjoint(tbar, cbar, y, T0, C, 1.0, dt, inv)
        got.append((loop, one, tbar, cbar))
    # a few roundings of values below 2 (the plain FP64 transposed step and the staged one round differently)
    tol = 1e-14 if dtype == torch.float64 else 4e-6
    for a, b in zip(*got):
        if torch.is_tensor(a) and torch.is_tensor(b):
            assert float((a - b).abs().max()) <= tol
    assert api.device_error() == 0
