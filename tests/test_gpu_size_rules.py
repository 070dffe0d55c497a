"""Grids thin in y or z, and odd rows: which kernels the size rules pick there, and that it does not show in
the result."""
import numpy as np
import pytest
import torch

from gpu_helpers import to_host
from paper_2211_15634_gb300 import api, inputs

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def fields(shape, dtype):
    nx, ny, nz = shape
    T = 1.0 + inputs.uniform_field_torch(3, nx, ny, nz, "cuda")
    C = 0.5 + 0.25 * inputs.uniform_field_torch(4, nx, ny, nz, "cuda")
    return T.to(dtype), C.to(dtype)


@pytest.mark.parametrize("shape,pairs", [((1024, 6, 512), False), ((1024, 14, 220), True), ((872, 16, 376), False),
                                         ((1023, 8, 512), False), ((1023, 16, 220), True), ((511, 511, 5), True)])
def test_fp32_pairs_by_the_rows_they_use(launch_override, shape, pairs):
    T, C = fields(shape, torch.float32)
    inv, dt, nt = (1.0, 1.0, 1.0), 0.1, 5
    name = api.step_kernel_name(T.clone(), T, C, 1.0, dt, inv, temporal2=True)
    assert name.startswith("k_zpair") == pairs

    def run():
        A, B = T.clone(), torch.full_like(T, 7.0)
        return to_host(api.run(A, B, C, 1.0, dt, inv, nt)), to_host(A), to_host(B)

    got = run()
    launch_override(kchunk=16)
    for a, b in zip(got, run()):
        assert np.array_equal(a, b)
    assert api.device_error() == 0
