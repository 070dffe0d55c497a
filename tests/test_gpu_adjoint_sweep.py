"""The reverse sweep as one library call: bit for bit the single transposed steps with the
buffers swapped, on every kernel form, and refusals before anything is launched."""
import numpy as np
import pytest
import torch

from gpu_helpers import to_dev
from paper_2211_15634_gb300 import _lib, api, autograd as ag, inputs

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def setup(shape, dtype, unequal):
    nx, ny, nz = shape
    inv = (nx - 1.0, ny - 0.5, nz - 0.7) if unequal else (max(shape) - 1.0,) * 3
    dt = 1.0 / max(inv) ** 2 / 0.75 / 6.1
    T = to_dev(inputs.t0_gaussian(nx, ny, nz) - (1.7 if dtype == torch.float32 else 0.0), dtype)
    return T, to_dev(inputs.ci_random(nx, ny, nz), dtype), dt, inv


@pytest.mark.parametrize("shape", [(3, 3, 3), (64, 10, 9), (65, 9, 7), (132, 17, 11)])
@pytest.mark.parametrize("dtype,unequal", [(torch.float64, False), (torch.float64, True), (torch.float32, False)])
@pytest.mark.parametrize("n", [0, 1, 4, 5])
def test_sweep_equals_single_steps(shape, dtype, unequal, n):
    T, C, dt, inv = setup(shape, dtype, unequal)
    scaled = dtype == torch.float64 and not unequal
    if scaled:
        C = api.scale_ci(C, 1.0, dt, inv)
    states = [T * (1.0 + 0.1 * i) for i in range(n)]
    y0 = to_dev(inputs.random_field(tuple(T.shape), 4, -1.0, 1.0), dtype)
    ya, ta, ca = y0.clone(), torch.empty_like(y0), torch.zeros_like(y0)
    for s in states:
        api.adjoint(ta, ca, ya, s, C, 1.0, dt, inv, ci_scaled=scaled)
        ya, ta = ta, ya
    for given in (states, [s.data_ptr() for s in states]):
        yb, tb, cb = y0.clone(), torch.full_like(y0, float("nan")), torch.zeros_like(y0)
        res, other = api.adjoint_sweep(tb, cb, yb, given, C, 1.0, dt, inv, ci_scaled=scaled)
        assert (res is tb) == (n % 2 == 1) and other is (yb if n % 2 else tb)
        assert torch.equal(res, ya) and torch.equal(cb, ca)


def test_refused_before_any_launch():
    T, C, dt, inv = setup((64, 10, 9), torch.float64, True)
    y, t, c = torch.ones_like(T), torch.full_like(T, 7.0), torch.full_like(T, 3.0)
    for bad in ([T, t], [T, y], [T, c], [T, T.data_ptr() + 8], [T, 0]):
        with pytest.raises(_lib.PsError):
            api.adjoint_sweep(t, c, y, bad, C, 1.0, dt, inv)
    with pytest.raises(ValueError):
        api.adjoint_sweep(t, c, y, [T[:-1]], C, 1.0, dt, inv)
    torch.cuda.synchronize()
    assert torch.all(t == 7.0) and torch.all(c == 3.0) and torch.all(y == 1.0)


@pytest.mark.parametrize("every", [1, 3, 7, 20])
@pytest.mark.parametrize("nt", [0, 1, 13])
def test_gradient_is_the_step_by_step_sweeps(monkeypatch, every, nt):
    T, C, dt, inv = setup((33, 12, 10), torch.float64, True)
    Tobs = T * 1.01
    got = ag.loss_and_grad(T, C, Tobs, 1.0, dt, inv, nt, every=every)

    def by_step(Tbar, Cibar, ybar, states, Ci, lam, dt, inv, *, ci_scaled=False):
        for s in states:
            if isinstance(s, int):  # the field at that address
                f = torch.empty_like(ybar)
                by_ptr(f, s, ybar)
                s = f
            api.adjoint(Tbar, Cibar, ybar, s, Ci, lam, dt, inv, ci_scaled=ci_scaled)
            ybar, Tbar = Tbar, ybar
        return ybar, Tbar

    def by_ptr(f, address, like):
        nz, ny, nx = like.shape
        # a view of device memory at an address: through the CUDA array interface
        holder = type("A", (), {})()
        holder.__cuda_array_interface__ = dict(shape=(nz, ny, nx), typestr="<f8", data=(address, False), version=3)
        f.copy_(torch.as_tensor(holder, device="cuda"))

    monkeypatch.setattr(api, "adjoint_sweep", by_step)
    want = ag.loss_and_grad(T, C, Tobs, 1.0, dt, inv, nt, every=every)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert np.isfinite(float(got[0]))
