"""2-D steps on rows of any length (strided lanes) and in short chunks: the same bits as the
aligned form gives on the nodes that two grids share, against the oracle by the other 2-D
tests' bounds, at strip edges (64 and 128 columns) and every residue of nx mod 4."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import rel_linf, to_dev, to_host
from paper_2211_15634_gb300 import api, inputs

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

U32 = 2.0 ** -24


@pytest.mark.parametrize("form", ["scaled", "equal", "unequal", "f32"])
@pytest.mark.parametrize("smooth", [True, False])
@pytest.mark.parametrize("nx,ny", [(3, 4), (33, 7), (34, 5), (35, 9), (63, 6), (65, 8), (66, 17), (127, 5), (129, 40),
                                   (130, 9), (131, 6), (193, 12), (257, 33), (385, 10)])
def test_matches_oracle_in_any_chunk(launch_override, form, smooth, nx, ny):
    T0 = inputs.random_field((ny, nx), 5, -1.0, 1.0)
    if smooth:
        T0 = 1.7 + 0.1 * T0 / (1.0 + np.abs(T0))
    Ci = inputs.ci_random(nx, ny, 1)[0]
    inv = (nx - 1.0, ny + 0.5) if form == "unequal" else (nx - 1.0,) * 2
    dt = 1.0 / max(inv) ** 2 / Ci.max() / 4.1
    dtype = torch.float32 if form == "f32" else torch.float64
    if dtype == torch.float32:
        T0, Ci = (a.astype(np.float32).astype(np.float64) for a in (T0, Ci))
    nt = 4
    ref = oracle.run2d(T0, Ci, 1.0, dt, *inv, nt)
    C = to_dev(Ci, dtype)
    if form == "scaled":
        C = api.scale_ci(C, 1.0, dt, inv)
    outs = []
    for chunk in (0, 1, 2, 5, 64):
        launch_override(chunk2d=chunk)
        T = to_dev(T0, dtype)
        outs.append(to_host(api.run2d(T, torch.empty_like(T), C, 1.0, dt, inv, nt, ci_scaled=form == "scaled")))
        assert np.array_equal(outs[-1], outs[0])
    if dtype == torch.float32:
        assert np.max(np.abs(outs[0] - ref)) <= nt * 13 * U32 * np.max(np.abs(T0))
    else:
        assert rel_linf(outs[0], ref) <= 1e-12
