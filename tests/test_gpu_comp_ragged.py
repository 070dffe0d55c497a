"""Two-float FP32 steps on rows that are no multiple of 16 bytes (k_comp_rag): bit for bit the column
kernel's states and corrections, at tile edges (128 columns, 16 rows), every residue of nx, of
nx*ny and of the correction fields' start mod 4, with infinities and NaN on the boundary."""
import pytest
import torch

from paper_2211_15634_gb300 import api

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("special", [False, True])
@pytest.mark.parametrize("shape", [(4, 5, 67), (9, 7, 129), (5, 17, 130), (6, 15, 131), (12, 31, 233), (17, 18, 257),
                                   (33, 29, 258), (20, 45, 386), (31, 33, 95), (11, 64, 127), (8, 35, 235)])
def test_equals_column_kernel(launch_override, shape, special):
    nz, ny, nx = shape
    g = torch.Generator(device="cuda").manual_seed(nx)
    T0 = 1.5 + torch.randn(shape, generator=g, device="cuda")
    Ci = 0.5 + 0.5 * torch.rand(shape, generator=g, device="cuda")
    if special:
        T0[0, 0, 0] = T0[0, -1, :] = float("inf")
        T0[-1, -1, -1] = T0[:, 0, 0] = float("nan")
    inv = (nx - 1.0, ny + 0.5, nz - 0.3)
    dt = 1.0 / max(inv) ** 2 / 8.0
    outs = []
    # the column kernel; then short and long chunks (a set chunk also keeps small grids on the march)
    for override in (dict(step_plain=1), dict(step_plain=0, kchunk=1), dict(kchunk=3), dict(kchunk=16)):
        launch_override(**override)
        T, T2 = T0.clone(), torch.full_like(T0, 7.0)
        comp = api.compensation_fields(T)
        api.run(T, T2, Ci, 0.9, dt, inv, 5, comp=comp)
        outs.append(torch.cat([a.reshape(-1) for a in (T, T2, comp)]))
    for o in outs[1:]:
        assert torch.equal(torch.nan_to_num(o, nan=12345.0), torch.nan_to_num(outs[0], nan=12345.0))
    assert api.device_error() == 0
