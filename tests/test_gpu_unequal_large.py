"""Unequal spacings on a grid large enough for four nodes per thread: the same bits as the plain
column kernel, in a loop and in a loop that keeps its states (which also writes the boundary)."""
import pytest
import torch

from paper_2211_15634_gb300 import api

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("signed", [False, True])
def test_four_nodes_per_thread_equal_the_column_kernel(launch_override, signed):
    nx, ny, nz = 252, 401, 300  # 30.3 million nodes, ragged against tiles of 128 x 4
    g = torch.Generator(device="cuda").manual_seed(3)
    T0 = torch.rand((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64)
    T0 = T0 - 0.5 if signed else 1.2 + 0.5 * T0
    Ci = 0.5 + 0.5 * torch.rand((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64)
    inv = (nx - 1.0, ny + 0.5, nz - 7.0)
    dt = 1.0 / max(inv) ** 2 / 6.1
    T = T0.clone()
    got = api.run(T, torch.empty_like(T0), Ci, 1.0, dt, inv, 3).clone()
    block = api.StateBlock(T0, 3, boundary=False)
    kept = api.run_states(T0, block, 1, Ci, 1.0, dt, inv, 3).clone()
    launch_override(step_plain=1)
    T = T0.clone()
    want = api.run(T, torch.empty_like(T0), Ci, 1.0, dt, inv, 3)
    assert torch.equal(got, want)
    assert torch.equal(kept, want)
    assert api.device_error() == 0
