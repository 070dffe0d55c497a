"""FP64 steps on unequal spacings: the axes' coefficients as integers at one exponent
(spacings within a factor of 16), one rounded product per axis beyond that, and the 2-D
form of both.  Against the FP64 oracle at the bound of the other FP64 steps (1e-12), and
bit for bit between the kernels that share the per-node arithmetic: the z-march takes a
warp's fast, window or general path together, the column kernel node by node."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import rel_linf, to_dev, to_host
from paper_2211_15634_gb300 import api, inputs
from test_gpu_general_path import KINDS, field

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

# _dx : _dy : _dz; the ratio of the largest to the smallest against the factor of 16
RATIOS = {"near": (1.0, 1.5, 0.7), "edge_in": (1.0, 15.99, 3.0), "edge_out": (16.01, 1.0, 2.0),
          "far": (1.0, 0.004, 300.0)}


def inverse_spacings(kind, n):
    inv = tuple(r * (n - 1.0) for r in RATIOS[kind])
    return inv, 1.0 / max(inv) ** 2


def run(T0, Ci, dt, inv, nt):
    T = to_dev(T0)
    return to_host(api.run(T, torch.empty_like(T), to_dev(Ci), 1.0, dt, inv, nt))


@pytest.mark.parametrize("ratios", list(RATIOS))
@pytest.mark.parametrize("values", ["smooth"] + KINDS)
def test_step_matches_oracle_and_column_kernel(launch_override, ratios, values):
    shape = nx, ny, nz = (132, 21, 17)
    T0 = inputs.t0_gaussian(nx, ny, nz) if values == "smooth" else field(values, shape)
    Ci = inputs.ci_random(nx, ny, nz)
    inv, d2 = inverse_spacings(ratios, nx)
    dt = d2 / Ci.max() / 6.1
    got = run(T0, Ci, dt, inv, 3)
    assert rel_linf(got, oracle.run(T0, Ci, 1.0, dt, *inv, 3)) <= 1e-12
    assert np.array_equal(run(-T0, Ci, dt, inv, 3), -got)  # the other sign: the other sign exactly
    launch_override(step_plain=1)
    assert np.array_equal(run(T0, Ci, dt, inv, 3), got)
    assert api.device_error() == 0


@pytest.mark.parametrize("ratios", list(RATIOS))
def test_constant_along_all_but_one_axis(ratios):
    """Sums of the other axes are zero: the smallest coefficient alone carries the update."""
    nx, ny, nz = 68, 19, 23
    inv, d2 = inverse_spacings(ratios, nx)
    for axis, n in enumerate((nz, ny, nx)):
        line = 1.7 + inputs.random_field((n,), 3 + axis, 0.0, 0.2)
        T0 = np.ascontiguousarray(np.broadcast_to(line.reshape([-1 if a == axis else 1 for a in range(3)]),
                                                  (nz, ny, nx)))
        Ci = inputs.ci_random(nx, ny, nz)
        dt = 1.0 / inv[2 - axis] ** 2 / Ci.max() / 6.1  # this axis's own bound: a large update
        got, ref = run(T0, Ci, dt, inv, 1), oracle.run(T0, Ci, 1.0, dt, *inv, 1)
        assert np.max(np.abs(ref - T0)) > 1e-3
        assert rel_linf(got, ref) <= 1e-15  # one step: the update's and the sum's roundings


@pytest.mark.parametrize("ratios", list(RATIOS))
@pytest.mark.parametrize("shape", [(3, 3), (5, 4), (66, 9), (130, 70), (257, 33), (1000, 37)])
def test_2d_matches_oracle(ratios, shape):
    nx, ny = shape
    inv, d2 = inverse_spacings(ratios, nx)
    for T0 in (1.7 + inputs.random_field((ny, nx), 4, 0.0, 1.0), inputs.random_field((ny, nx), 5, -1.0, 1.0)):
        Ci = inputs.ci_random(nx, ny, 1)[0]
        dt = 1.0 / max(inv[:2]) ** 2 / Ci.max() / 4.1
        T = to_dev(T0)
        got = to_host(api.run2d(T, torch.empty_like(T), to_dev(Ci), 1.0, dt, inv[:2], 5))
        assert rel_linf(got, oracle.run2d(T0, Ci, 1.0, dt, *inv[:2], 5)) <= 1e-12


@pytest.mark.parametrize("ratios", ["equal"] + list(RATIOS))
@pytest.mark.parametrize("values", ["smooth", "many_binades"])
@pytest.mark.parametrize("shape", [(3, 3, 3), (68, 19, 13), (132, 21, 17)])
def test_transposed_step_matches_oracle(ratios, values, shape):
    """Ci as given: one coefficient (equal), integers at one exponent, one product per axis."""
    nx, ny, nz = shape
    T = inputs.t0_gaussian(nx, ny, nz) if values == "smooth" else field(values, shape)
    Ci, ybar = inputs.ci_random(nx, ny, nz), inputs.random_field((nz, ny, nx), 31, -1.0, 1.0)
    inv, d2 = ((nx - 1.0,) * 3, 1.0 / (nx - 1.0) ** 2) if ratios == "equal" else inverse_spacings(ratios, nx)
    dt = d2 / Ci.max() / 6.1
    ref_c = np.zeros_like(T)
    ref_t = oracle.adjoint_step(ybar, T, Ci, ref_c, 1.0, dt, *inv)
    tbar, cibar = to_dev(np.full_like(T, np.nan)), to_dev(np.zeros_like(T))
    api.adjoint(tbar, cibar, to_dev(ybar), to_dev(T), to_dev(Ci), 1.0, dt, inv)
    assert rel_linf(to_host(tbar), ref_t) <= 1e-14
    assert rel_linf(to_host(cibar), ref_c) <= 1e-14
    assert api.device_error() == 0
