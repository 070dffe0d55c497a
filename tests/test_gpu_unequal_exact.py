"""The weighted Laplacian L of unequal spacings against rational arithmetic, where a call shows it unrounded:
Cibar of a transposed step with ybar = 1 is L(T).

L is one rounding of a sum whose products are cut at 2^-59 of the largest (two units each, three axes), so
|error| <= 2^-53 |L| + 6 * 2^-59 max_d |K_d S_d| at every ratio of the spacings, along whichever axes
the field varies; below the normal range half a unit of 2^-1074 takes the place of the first term."""
from fractions import Fraction as F

import numpy as np
import pytest
import torch

from gpu_helpers import to_dev, to_host
from paper_2211_15634_gb300 import api

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

CUT = F(6, 2 ** 59)


def exact(T, K):
    """{node: (L, largest product)} of the interior nodes; K and T's axes in the order (x, y, z)."""
    T = np.vectorize(lambda v: F(float(v)), otypes=[object])(T)
    out = {}
    for p in np.ndindex(*[n - 2 for n in T.shape]):
        q = tuple(i + 1 for i in p)
        terms = []
        for a, k in enumerate(reversed(K)):
            up, dn = list(q), list(q)
            up[a] += 1
            dn[a] -= 1
            terms.append(k * (T[tuple(up)] + T[tuple(dn)] - 2 * T[q]))
        out[q] = (sum(terms), max(abs(t) for t in terms))
    return out


def check(got, want, where=None):
    for q, (L, big) in want.items():
        if where is None or where[q]:
            err = abs(F(float(got[q])) - L)
            assert err <= max(abs(L) / 2 ** 53, F(1, 2 ** 1075)) + CUT * big, (q, float(got[q]), float(L))


@pytest.mark.parametrize("nx", [9, 10])
@pytest.mark.parametrize("scale,dt", [(2.0 ** -1000, 2.0 ** -67), (2.0 ** -1010, 2.0 ** -60), (2.0 ** -950, 2.0 ** -118),
                                      (2.0 ** -1020, 2.0 ** -130)])
def test_below_the_normal_range(nx, scale, dt):
    """L among the subnormal numbers, and far below the smallest of them."""
    shape, inv = (6, 7, nx), (1.0, 1.5, 2.0)
    T = np.random.default_rng(8).integers(1, 2 ** 20, shape).astype(np.float64) * (scale / 2 ** 20)
    one, cbar = to_dev(np.ones(shape)), to_dev(np.zeros(shape))
    api.adjoint(torch.empty_like(one), cbar, one, to_dev(T), one, 1.0, dt, inv)
    got = to_host(cbar)
    check(got, exact(T, [F(dt) * F(v) ** 2 for v in inv]))
    assert np.count_nonzero(got) > 0 or dt == 2.0 ** -130
