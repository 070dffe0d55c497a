"""FP32 step pairs on rows that are no multiple of 16 bytes (k_zpair_rag): bit for bit the single
steps' two buffers, at tile edges (128 columns, 14 rows), every residue of nx and of nx*ny
mod 4, short and long chunks, with infinities and NaN on the boundary."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import to_dev, to_host
from paper_2211_15634_gb300 import api, inputs

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

U32 = 2.0 ** -24
SHAPES = [(3, 3, 3), (9, 7, 5), (5, 17, 130), (6, 15, 129), (12, 31, 131), (17, 18, 257), (33, 29, 258), (20, 45, 386),
          (31, 33, 65), (50, 14, 6), (11, 64, 127), (8, 30, 135)]


def run(launch_override, T0, C, inv, dt, nt, **override):
    launch_override(kchunk=0, kchunk2=0)
    launch_override(**override)
    T = T0.clone()
    T2 = torch.full_like(T, 7.0)
    out = api.run(T, T2, C, 0.9, dt, inv, nt)
    return out, (T2 if out.data_ptr() == T.data_ptr() else T)


def setup(shape, special):
    nz, ny, nx = shape
    T0 = inputs.random_field(shape, 3, -1.0, 1.0).astype(np.float32)
    if special:
        T0[0, 0, 0] = np.inf
        T0[-1, -1, -1] = np.nan
        T0[0, -1, :] = -np.inf
        T0[:, 0, 0] = np.nan
        T0[-1, ny // 2, nx // 2] = np.inf
    C = inputs.ci_random(nx, ny, nz).astype(np.float32)
    inv = (nx - 1.0, ny - 0.5, nz + 0.0)
    return T0, C, inv, 1.0 / max(inv) ** 2 / 8.0


@pytest.mark.parametrize("special", [False, True])
@pytest.mark.parametrize("chunk", [1, 4, 16])
@pytest.mark.parametrize("shape", SHAPES)
def test_forced_pairs_equal_single_steps(launch_override, shape, chunk, special):
    T0, C, inv, dt = setup(shape, special)
    a, b = to_dev(T0, torch.float32), to_dev(C, torch.float32)
    want = run(launch_override, a, b, inv, dt, 9, kchunk=16)
    got = run(launch_override, a, b, inv, dt, 9, kchunk2=chunk)
    for x, y in zip(got, want):
        assert np.array_equal(to_host(x), to_host(y), equal_nan=True)
    assert api.device_error() == 0


@pytest.mark.parametrize("shape", [(129, 129, 129), (70, 120, 383)])
@pytest.mark.parametrize("nt", [3, 8, 13])
def test_default_loop_against_oracle(shape, nt):
    T0, C, inv, dt = setup(shape, False)
    T, Ci = to_dev(T0, torch.float32), to_dev(C, torch.float32)
    out = to_host(api.run(T, torch.empty_like(T), Ci, 0.9, dt, inv, nt))
    ref = oracle.run(T0.astype(np.float64), C.astype(np.float64), 0.9, dt, *inv, nt)
    # a step rounds the update a few times and the state once, and the scheme does not grow errors
    assert np.max(np.abs(out - ref)) <= nt * 13 * U32
