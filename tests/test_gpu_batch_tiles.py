"""Batched grids whose last columns take each of the tile shapes (wide, narrow, narrow and
quarter, quarter): every problem equals its single run bit for bit."""
import numpy as np
import pytest
import torch

from gpu_helpers import to_dev, to_host
from paper_2211_15634_gb300 import api, inputs

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

# FP64 columns left after whole 64s: 1, 15, 16, 17, 32, 33, 48, 49, 63; twice that in FP32
NX = [3, 17, 18, 19, 34, 35, 50, 51, 65, 66, 82, 98, 114, 130, 162, 163, 226]
NY = [4, 33, 34, 9, 65]


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("smooth", [True, False])
@pytest.mark.parametrize("ny", NY)
def test_every_tile_shape_equals_single_runs(dtype, smooth, ny):
    probs, singles, nt = [], [], 3
    for i, nx in enumerate(NX):
        nz = 3 + i % 5
        T0 = inputs.random_field((nz, ny, nx), 7 + i, -1.0, 1.0)
        if smooth:
            T0 = 1.7 + 0.1 * T0 / (1.0 + np.abs(T0))
        inv = (nx - 1.0,) * 3
        dt = 1.0 / inv[0] ** 2 / 8.1
        fields = []
        for a in (T0, T0, inputs.ci_random(nx, ny, nz)):
            f = api.pitched_empty((nz, ny, nx), dtype)
            f.copy_(to_dev(a, dtype))
            fields.append(f)
        probs.append(dict(T=fields[0], T2=fields[1], Ci=fields[2], lam=0.9, dt=dt, inv_spacing=inv))
        C = fields[2].contiguous()
        if dtype == torch.float64:
            C = api.scale_ci(C, 0.9, dt, inv)
        T = fields[0].contiguous().clone()
        singles.append(to_host(api.run(T, T.clone(), C, 0.9, dt, inv, nt, ci_scaled=dtype == torch.float64)))
    b = api.Batch(probs)
    assert b.kernel == "zmarch"
    b.run(nt)
    for p, want in zip(probs, singles):
        assert np.array_equal(to_host(p["T2"].contiguous()), want)
    assert api.device_error() == 0
