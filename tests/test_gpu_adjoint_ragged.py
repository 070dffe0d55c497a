"""Transposed steps on ragged rows (odd nx in FP64, nx % 4 != 0 in FP32) against the FP64
oracle, at the bounds of the other transposed-step tests: tile edges in x, y and z, even and
odd numbers of rows (a last single row lies outside the FP64 kernel's row-pair map), every
residue of nx mod 4, and the plain column kernel on the same fields."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import rel_linf, to_dev, to_host
from paper_2211_15634_gb300 import api, inputs

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

SHAPES = [(3, 3, 3), (5, 4, 3), (5, 5, 5), (7, 9, 8), (63, 8, 5), (65, 9, 7), (65, 10, 20), (127, 17, 3),
          (129, 7, 9), (131, 16, 18), (193, 11, 6)]
F32_SHAPES = SHAPES + [(6, 5, 4), (66, 9, 6), (130, 13, 5), (254, 9, 7)]


def run(shape, form, smooth=True):
    nx, ny, nz = shape
    T = inputs.t0_gaussian(nx, ny, nz) if smooth else inputs.random_field((nz, ny, nx), 3, -1.0, 1.0)
    Ci, ybar = inputs.ci_random(nx, ny, nz), inputs.random_field((nz, ny, nx), 31, -1.0, 1.0)
    inv = (nx - 1.0, ny - 0.5, nz - 0.7) if form.endswith("unequal") else (max(shape) - 1.0,) * 3
    dt = 1.0 / max(inv) ** 2 / Ci.max() / 6.1
    dtype = torch.float32 if form.startswith("f32") else torch.float64
    if dtype == torch.float32:
        T, Ci, ybar = ((a - (1.7 if a is T and smooth else 0.0)).astype(np.float32).astype(np.float64)
                       for a in (T, Ci, ybar))
    C = to_dev(Ci, dtype)
    if form == "scaled":
        C = api.scale_ci(C, 1.0, dt, inv)
    c0 = inputs.random_field((nz, ny, nx), 9, -1e-3, 1e-3)
    tbar, cibar = to_dev(np.full_like(T, np.nan), dtype), to_dev(c0, dtype)
    api.adjoint(tbar, cibar, to_dev(ybar, dtype), to_dev(T, dtype), C, 1.0, dt, inv, ci_scaled=form == "scaled")
    ref_c = np.zeros_like(T)
    ref_t = oracle.adjoint_step(ybar, T, Ci, ref_c, 1.0, dt, *inv)
    if form == "scaled":
        ref_c = ref_c / (dt * inv[0] * inv[0])  # dL/dCs
    got_c = to_host(cibar)
    return to_host(tbar), got_c, ref_t, ref_c + (c0 if dtype == torch.float64 else c0.astype(np.float32))


@pytest.mark.parametrize("form", ["scaled", "equal", "unequal"])
@pytest.mark.parametrize("smooth", [True, False])
@pytest.mark.parametrize("shape", SHAPES)
def test_fp64_matches_oracle(launch_override, shape, form, smooth):
    for kchunk in (0, 1, 5):
        launch_override(adj_kchunk=kchunk)
        tbar, cbar, ref_t, ref_c = run(shape, form, smooth)
        assert rel_linf(tbar, ref_t) <= 1e-14
        assert rel_linf(cbar, ref_c) <= 1e-14
    assert api.device_error() == 0


@pytest.mark.parametrize("form", ["f32", "f32unequal"])
@pytest.mark.parametrize("smooth", [True, False])
@pytest.mark.parametrize("shape", F32_SHAPES)
def test_fp32_matches_oracle(launch_override, shape, form, smooth):
    for kchunk in (0, 1, 5):
        launch_override(adj_kchunk=kchunk)
        tbar, cbar, ref_t, ref_c = run(shape, form, smooth)
        assert rel_linf(tbar, ref_t) <= 2e-6
        assert rel_linf(cbar, ref_c) <= 2e-6
    assert api.device_error() == 0
