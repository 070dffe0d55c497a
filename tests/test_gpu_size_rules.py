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


@pytest.mark.parametrize("form", ["f32", "comp", "scaled", "equal", "unequal"])
@pytest.mark.parametrize("shape", [(75, 31, 40), (129, 5, 60), (191, 25, 33)])
def test_odd_rows_the_same_bits_by_every_route(launch_override, shape, form):
    """Single steps, the loop, and both with the march or the column kernel asked for."""
    dtype = torch.float32 if form in ("f32", "comp") else torch.float64
    T, C = fields(shape, dtype)
    T[:T.shape[0] // 2, ::3] -= 1.5  # both signs below, one binade above
    inv = (3.0, 2.0, 2.5) if form == "unequal" else (2.0, 2.0, 2.0)
    dt, nt, scaled = 0.01, 3, form == "scaled"
    if scaled:
        C = api.scale_ci(C, 1.0, dt, inv)

    def loop():
        A, B = T.clone(), torch.empty_like(T)
        comp = api.compensation_fields(T) if form == "comp" else None
        out = api.run(A, B, C, 1.0, dt, inv, nt, comp=comp, ci_scaled=scaled)
        return torch.stack([out, comp[nt % 2]]) if form == "comp" else out

    def steps():
        A, B = T.clone(), T.clone()
        E = [torch.zeros_like(T) for _ in range(2)] if form == "comp" else None
        for i in range(nt):
            if form == "comp":
                api.step_compensated(B, A, E[1 - i % 2], E[i % 2], C, 1.0, dt, inv)
            else:
                api.step(B, A, C, 1.0, dt, inv, ci_scaled=scaled)
            A, B = B, A
        return torch.stack([A, E[nt % 2]]) if form == "comp" else A

    want = loop()
    for override in (dict(), dict(kchunk=3), dict(kchunk=0, step_plain=1)):
        launch_override(**override)
        assert torch.equal(loop(), want)
        assert torch.equal(steps(), want)
    assert api.device_error() == 0


@pytest.mark.parametrize("form,shape,name", [
    ("f32", (161, 265, 96), "k_step_basic<float>"), ("f32", (257, 257, 257), "k_zmarch_rag<F32>"),
    ("f32", (391, 8, 3059), "k_step_basic<float>"), ("scaled", (75, 148, 320), "k_step_basic_emu"),
    ("scaled", (257, 257, 257), "k_zmarch_rag<F64_SCALED>"), ("equal", (213, 407, 192), "k_step_basic_emu"),
    ("equal", (257, 257, 257), "k_zmarch_rag<F64_EMU_ISO>"), ("unequal", (93, 512, 257), "k_step_basic_emu"),
    ("unequal", (257, 257, 257), "k_zmarch_rag<F64_EMU_ANISO>")])
def test_odd_rows_kernel_of_a_single_step(form, shape, name):
    T, C = fields(shape, torch.float32 if form == "f32" else torch.float64)
    inv = (1.0, 1.5, 1.2) if form == "unequal" else (1.0, 1.0, 1.0)
    assert api.step_kernel_name(torch.empty_like(T), T, C, 1.0, 0.1, inv, ci_scaled=form == "scaled") == name


@pytest.mark.parametrize("shape,name", [((3000, 3, 300), "k_zmarch<F64_SCALED4>"), ((192, 192, 192), "k_zmarch<F64_SCALED>"),
                                        ((256, 100, 100), "k_zmarch<F64_SCALED4>")])
def test_tile_shape_of_the_pre_scaled_step(shape, name):
    T, C = fields(shape, torch.float64)
    assert api.step_kernel_name(torch.empty_like(T), T, C, 1.0, 0.1, (1.0,) * 3, ci_scaled=True) == name
