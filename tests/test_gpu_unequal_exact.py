"""The weighted Laplacian L of unequal spacings against rational arithmetic, where a call shows it unrounded:
Cibar of a transposed step with ybar = 1 is L(T), Tbar with Ci = 1 is L(ybar) where ybar = 0, and a step
with Ci = 1 gives L(T) where T = 0.

L is one rounding of a sum whose products are cut at 2^-59 of the largest (two units each, three axes), so
|error| <= 2^-53 |L| + 6 * 2^-59 max_d |K_d S_d|, along whichever axes the field varies and at every ratio of
the spacings; where the K's exponents lie within 5 they are shifted right by up to two bits, which costs that
many of the second term.  (A rounding for each axis: 2^-53 of each term.)  Below the normal range half a unit
of 2^-1074 takes the place of the first term."""
import math
from fractions import Fraction as F
from itertools import permutations

import numpy as np
import pytest
import torch

from gpu_helpers import to_dev, to_host
from paper_2211_15634_gb300 import api

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

# 1 / spacing per axis, up to the factor of 16 within which the axes share one integer sum
RATIOS = [(1.0, 1.3, 1.0), (2.0, 1.5, 1.0), (4.1, 1.0, 3.7), (5.1, 1.0, 2.9), (9.1, 1.0, 2.9), (15.99, 1.0, 1.0), (15.99, 1.0, 15.3)]
DT = 0.1
FIELDS = ["binade", "window", "signed", "x", "y", "z", "pair"]


def coefficients(dt, inv):
    return [F(dt * (v * v)) for v in inv]  # as the library forms them, in FP64


def cut(K):
    e = [math.frexp(float(k))[1] for k in K]
    gap = max(e) - min(e)
    return F(6, 2 ** (59 - min(gap, 2) if gap <= 5 else 59))


def field(kind, shape, seed):
    """Values in one binade, in five, or of both signs; varying along one axis alone; a pair of
    axes whose second differences nearly cancel."""
    rng = np.random.default_rng(seed)
    r = rng.integers(1, 2 ** 52, shape).astype(np.float64) / 2 ** 52
    if kind == "binade":
        return 1.0 + r
    if kind == "window":
        return 1.0 + 20.0 * r
    if kind == "signed":
        return 2.0 * r - 1.0
    axes = [np.arange(n) for n in shape]
    wave = [rng.integers(0, 2 ** 52, n).astype(np.float64) / 2 ** 52 for n in shape]
    z, y, x = np.meshgrid(*[w[a] for w, a in zip(wave, axes)], indexing="ij")
    return {"x": 1.0 + x, "y": 1.0 + y, "z": 1.0 + z, "pair": 1.5 + 0.25 * (x - y)}[kind] + 0.0 * r


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


def check(got, want, cut, where=None):
    for q, (L, big) in want.items():
        if where is None or where[q]:
            err = abs(F(float(got[q])) - L)
            assert err <= max(abs(L) / 2 ** 53, F(1, 2 ** 1075)) + cut * big, (q, float(got[q]), float(L))


def zeros_between(T):
    """T with every second node zero, and where."""
    odd = sum(np.indices(T.shape)) % 2 == 1
    return np.where(odd, 0.0, T), odd


@pytest.mark.parametrize("kind", FIELDS)
@pytest.mark.parametrize("ratio", RATIOS)
@pytest.mark.parametrize("nx", [9, 10])
def test_transposed_step(nx, ratio, kind):
    shape = (6, 7, nx)
    T = field(kind, shape, 5)
    y, odd = zeros_between(field(kind, shape, 6))
    w = y.copy()  # the step writes interior nodes only
    for face in (np.s_[0], np.s_[-1], np.s_[:, 0], np.s_[:, -1], np.s_[:, :, 0], np.s_[:, :, -1]):
        w[face] = 0.0
    one, tbar = to_dev(np.ones(shape)), to_dev(np.zeros(shape))
    for inv in sorted(set(permutations(ratio))):
        K = coefficients(DT, inv)
        cbar = to_dev(np.zeros(shape))
        api.adjoint(tbar, cbar, one, to_dev(T), one, 1.0, DT, inv)
        check(to_host(cbar), exact(T, K), cut(K))
        api.adjoint(tbar, cbar, to_dev(y), to_dev(T), one, 1.0, DT, inv)
        check(to_host(tbar), exact(w, K), cut(K), odd)


@pytest.mark.parametrize("kind", FIELDS)
@pytest.mark.parametrize("ratio", RATIOS)
@pytest.mark.parametrize("nx", [9, 10])
def test_steps(launch_override, nx, ratio, kind):
    shape = (6, 7, nx)
    T, odd = zeros_between(field(kind, shape, 7))
    one = to_dev(np.ones(shape))
    for inv in sorted(set(permutations(ratio))):
        K = coefficients(DT, inv)
        want = exact(T, K)
        for kchunk in (0, 3):  # the column kernel in a loop, the march
            launch_override(kchunk=kchunk)
            check(to_host(api.run(to_dev(T), to_dev(T), one, 1.0, DT, inv, 1)), want, cut(K), odd)
        got = api.run2d(to_dev(T[2]), to_dev(T[2]), one[2].clone(), 1.0, DT, inv[:2], 1)
        check(to_host(got), exact(T[2], K[:2]), cut(K[:2]), odd[2])


@pytest.mark.parametrize("kind", FIELDS)
@pytest.mark.parametrize("inv", [(5.1, 1.0, 2.9), (9.1, 1.0, 2.9), (1.0, 15.3, 15.99), (3.0, 8.0, 1.0)])
def test_same_bits_on_every_kernel(launch_override, inv, kind):
    """Wide spreads: the march on even and odd rows, the column kernel, the batch."""
    for nx in (67, 68):
        T, C = to_dev(field(kind, (9, 19, nx), 9)), to_dev(0.5 + 0.25 * np.random.default_rng(3).random((9, 19, nx)))
        dt, got = 0.1 / max(inv) ** 2, []
        for override in (dict(kchunk=0), dict(kchunk=4), dict(kchunk=0, step_plain=1)):
            launch_override(step_plain=0)
            launch_override(**override)
            got.append(to_host(api.run(T.clone(), T.clone(), C, 1.0, dt, inv, 3)))
        launch_override(step_plain=0)
        A, B = T.clone(), T.clone()
        batch = api.Batch([dict(T=A, T2=B, Ci=C, lam=1.0, dt=dt, inv_spacing=inv)])
        batch.run(3)
        got.append(to_host(B))
        for g in got[1:]:
            assert np.array_equal(g, got[0])


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
    K = coefficients(dt, inv)
    check(got, exact(T, K), cut(K))
    assert np.count_nonzero(got) > 0 or dt == 2.0 ** -130
