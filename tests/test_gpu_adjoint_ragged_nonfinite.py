"""FP64 transposed step on odd rows with infinities and NaN in the cotangent or the coefficient: non-finite at
the nodes whose stencil meets one, and nowhere else, as the plain column kernel has it; in Tbar the same
value there (in Cibar an infinity times a Laplacian near zero takes either kernel's sign of it), and
within the usual bound where finite."""
import numpy as np
import pytest
import torch

from gpu_helpers import to_dev, to_host
from paper_2211_15634_gb300 import api, inputs

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

FORMS = {"scaled": (1.0, 1.0, 1.0), "equal": (1.0, 1.0, 1.0), "near": (1.0, 1.5, 0.8), "spread": (1.0, 9.0, 3.0)}


def case(shape, where):
    nx, ny, nz = shape
    y = inputs.random_field((nz, ny, nx), 4, -1.0, 1.0)
    C = inputs.ci_random(nx, ny, nz)
    if where == "cotangent":
        y[nz // 2, ny // 2, nx // 2] = np.inf
        y[1, 1, 1] = np.nan
        y[nz - 2, 1, nx - 2] = -np.inf
    elif where == "faces":  # copied to Tbar, read by no other node
        y[0, ny // 2, nx // 2] = np.inf
        y[nz - 1, ny - 1, nx - 1] = np.nan
        y[nz // 2, 0, 0] = -np.inf
    else:
        C[nz // 2, ny // 2, nx // 3 + 1] = np.inf
        C[1, ny - 2, 1] = np.nan
    return y, C


@pytest.mark.parametrize("where", ["cotangent", "faces", "coefficient"])
@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("shape", [(3, 3, 3), (65, 9, 7), (67, 17, 33), (129, 20, 12)])
def test_spread_is_the_stencils(launch_override, shape, form, where):
    nx, ny, nz = shape
    y, C = case(shape, where)
    T = inputs.t0_gaussian(nx, ny, nz)
    inv = tuple(r * (nx - 1.0) for r in FORMS[form])
    dt = 0.1 / max(inv) ** 2
    Cd = to_dev(C)
    if form == "scaled":
        Cd = api.scale_ci(Cd, 1.0, dt, inv)
    got = []
    for plain in (0, 1):
        launch_override(adj_plain=plain)
        tb, cb = to_dev(np.zeros_like(y)), to_dev(np.zeros_like(y))
        api.adjoint(tb, cb, to_dev(y), to_dev(T), Cd, 1.0, dt, inv, ci_scaled=form == "scaled")
        got.append((to_host(tb), to_host(cb)))
    assert not np.isfinite(got[1][0]).all()
    tb, plain_tb = got[0][0], got[1][0]
    assert np.array_equal(tb[~np.isfinite(plain_tb)], plain_tb[~np.isfinite(plain_tb)], equal_nan=True)
    for a, b in zip(*got):
        fin = np.isfinite(b)
        assert np.array_equal(np.isfinite(a), fin)
        if fin.any():
            assert np.max(np.abs(a[fin] - b[fin])) <= 1e-14 * max(np.max(np.abs(b[fin])), np.max(np.abs(y[np.isfinite(y)])))
    assert api.device_error() == 0
