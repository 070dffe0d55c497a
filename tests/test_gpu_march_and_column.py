"""The forms of the forward step that a grid's size and row length choose between: the TMA
z-march, its row-by-row form on ragged rows (odd nx; FP32 nx % 4 != 0) and, on small grids
inside a time loop, the column kernel.  All step a node by the same arithmetic, so a loop
gives the same bits through each (a z-chunk override asks for the march), its states keep
every boundary node, and FP64 and FP32 stay within the bounds of the other forward tests."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import rel_linf, to_dev, to_host
from paper_2211_15634_gb300 import api, inputs

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

U32 = 2.0 ** -24
# tile edges in x (64 / 128 nodes, from 0 on even rows and from 1 on ragged ones), y (4 / 8 rows)
# and z; every residue of nx mod 4 and of nx*ny mod 4
SHAPES = [(3, 3, 3), (4, 3, 5), (5, 4, 3), (6, 11, 4), (7, 10, 9), (63, 9, 6), (64, 10, 13), (65, 10, 11),
          (66, 12, 7), (67, 17, 6), (129, 11, 21), (130, 19, 5), (131, 9, 10), (132, 8, 9), (257, 13, 7)]
FORMS = ["scaled", "equal", "unequal", "f32", "comp"]


def setup(form, shape, smooth=True):
    nx, ny, nz = shape
    T0 = inputs.t0_gaussian(nx, ny, nz) if smooth else inputs.random_field((nz, ny, nx), 8, -1.0, 1.0)
    Ci = inputs.ci_random(nx, ny, nz)
    inv = (nx - 1.0, ny - 0.5, nz - 0.7) if form == "unequal" else (max(shape) - 1.0,) * 3
    dt = 1.0 / max(inv) ** 2 / Ci.max() / 6.1
    if form in ("f32", "comp"):
        T0 = (T0 - (1.7 if smooth else 0.0)).astype(np.float32).astype(np.float64)
        Ci = Ci.astype(np.float32).astype(np.float64)
    return T0, Ci, dt, inv


def loop(form, T0, Ci, dt, inv, nt):
    dtype = torch.float32 if form in ("f32", "comp") else torch.float64
    T, C = to_dev(T0, dtype), to_dev(Ci, dtype)
    if form == "scaled":
        C = api.scale_ci(C, 1.0, dt, inv)
    comp = api.compensation_fields(T) if form == "comp" else None
    res = api.run(T, torch.empty_like(T), C, 1.0, dt, inv, nt, comp=comp, ci_scaled=form == "scaled")
    return to_host(res) if comp is None else np.stack([to_host(res), to_host(comp[nt % 2])])


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("shape", SHAPES)
def test_march_equals_column_and_oracle(launch_override, form, shape):
    nt = 3
    for smooth in (True, False):
        T0, Ci, dt, inv = setup(form, shape, smooth)
        got = loop(form, T0, Ci, dt, inv, nt)
        ref = oracle.run(T0, Ci, 1.0, dt, *inv, nt)
        value = got if form != "comp" else got[0] + got[1]
        if form in ("f32", "comp"):
            assert np.max(np.abs(value - ref)) <= nt * 13 * U32 * np.max(np.abs(T0)) + 1e-30
        else:
            assert rel_linf(value, ref) <= 1e-12
        for kchunk in (2, 5, 64):
            launch_override(kchunk=kchunk)
            if form == "equal":  # the one-binade form rounds Ci*K first: another last bit
                assert rel_linf(loop(form, T0, Ci, dt, inv, nt), ref) <= 1e-12
            else:
                assert np.array_equal(loop(form, T0, Ci, dt, inv, nt), got)
        launch_override(kchunk=0)
    assert api.device_error() == 0


@pytest.mark.parametrize("form", ["scaled", "equal", "unequal", "f32"])
@pytest.mark.parametrize("every", [1, 2])
@pytest.mark.parametrize("shape", SHAPES)
def test_kept_states_hold_the_boundary(launch_override, form, every, shape):
    """run_states into unset memory: interior as the loop's, every face node T0's."""
    T0, Ci, dt, inv = setup(form, shape, smooth=False)
    dtype = torch.float32 if form == "f32" else torch.float64
    T, C = to_dev(T0, dtype), to_dev(Ci, dtype)
    if form == "scaled":
        C = api.scale_ci(C, 1.0, dt, inv)
    nt = 4
    for kchunk in (0, 3):
        launch_override(kchunk=kchunk)
        block = api.StateBlock(T, nt // every + 2, boundary=False)
        block.flat.fill_(float("nan"))
        api.run_states(T, block, every, C, 1.0, dt, inv, nt, ci_scaled=form == "scaled")
        for s in range(nt // every):
            assert np.array_equal(to_host(block.grids[s]), loop(form, T0, Ci, dt, inv, (s + 1) * every))
    assert api.device_error() == 0


@pytest.mark.parametrize("shape", [(64, 10, 13), (132, 8, 9), (256, 21, 17)])
def test_forced_pairs_equal_single_steps(launch_override, shape):
    """FP32 pairs leave small grids to the column kernel; forced, they give the same bits."""
    T0, Ci, dt, inv = setup("f32", shape)
    want = loop("f32", T0, Ci, dt, inv, 6)
    for kchunk2 in (0, 1, 4, 40):
        launch_override(kchunk2=kchunk2)
        T = to_dev(T0, torch.float32)
        got = api.run(T, torch.empty_like(T), to_dev(Ci, torch.float32), 1.0, dt, inv, 6, temporal2=True)
        assert np.array_equal(to_host(got), want)
    assert api.device_error() == 0


def test_size_rule_edges():
    """Just below and above the node count at which loops turn to the march, against each other
    through the shared interior of the two grids."""
    for dtype, nx in ((torch.float64, 191), (torch.float64, 192), (torch.float32, 190), (torch.float32, 192)):
        out = []
        for nz in (int(7.5e6) // (nx * 200), int(7.5e6) // (nx * 200) + 1):
            T = 1.0 + inputs.uniform_field_torch(3, nx, 200, nz, "cuda")
            C = 0.5 + 0.25 * inputs.uniform_field_torch(4, nx, 200, nz, "cuda")
            T, C = T.to(dtype), C.to(dtype)
            res = api.run(T, torch.empty_like(T), C, 1.0, 1e-6, (190.0,) * 3, 2)
            out.append(res[:180])
        if dtype == torch.float32:
            assert torch.equal(out[0], out[1])
        else:
            assert float((out[0] - out[1]).abs().max()) <= 2.0 ** -52 * 2
