"""FP32 step pairs on rows of a multiple of 16 bytes (k_zpair), forced by a z-chunk of their own,
against single steps, forced by the march's: both buffers, and every kept state, bit for bit.  Partial
tiles in x (128 columns) and y (14 rows), unequal spacings, infinities and NaN on edges, corners
and faces of the box (single steps never read an edge), a smooth field so large that a
difference to the zeros outside the grid overflows where no difference inside it does, and zeros
of both signs with a step back in time."""
import numpy as np
import pytest
import torch

from gpu_helpers import to_dev, to_host
from paper_2211_15634_gb300 import api, autograd, inputs

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

SHAPES = [(3, 3, 4), (9, 15, 36), (12, 17, 132), (20, 30, 196), (7, 14, 260), (11, 31, 128)]
FIELDS = ["random", "edges", "faces", "large", "zeros"]


def setup(shape, field):
    nz, ny, nx = shape
    C = inputs.ci_random(nx, ny, nz).astype(np.float32)
    inv = (nx - 1.0, ny - 0.5, nz + 0.0)
    if field == "large":  # spacings of 10 nm, values of 1e23: 1e23 * 1e16 overflows
        inv = (1.0e8, 0.9e8, 0.8e8)
        T0 = 1.0e23 * (1.0 + 0.01 * (inputs.t0_gaussian(nx, ny, nz) - 1.7))
    else:
        T0 = inputs.random_field(shape, 3, -1.0, 1.0)
    T0 = T0.astype(np.float32)
    if field == "edges":
        T0[:, 0, 0] = np.nan
        T0[0, -1, :] = -np.inf
        T0[-1, :, -1] = np.inf
        T0[-1, -1, -1] = np.nan
    elif field == "faces":
        T0[nz // 2, ny // 2, 0] = np.inf
        T0[nz // 2, 0, nx // 2] = np.nan
        T0[-1, ny // 2, nx // 2] = -np.inf
    elif field == "zeros":
        T0 = np.where(np.abs(T0) < 0.9, np.copysign(0.0, T0), T0).astype(np.float32)
    dt = 1.0 / max(inv) ** 2 / 8.0
    return to_dev(T0, torch.float32), to_dev(C, torch.float32), inv, -dt if field == "zeros" else dt


def same(x, y):
    return np.array_equal(x, y, equal_nan=True) and np.array_equal(np.signbit(x)[x == x], np.signbit(y)[y == y])


def check_spread(field, T):
    """What the field is there for: an edge reaches no interior node, the large field stays finite."""
    if field in ("edges", "large"):
        assert np.isfinite(to_host(T)[1:-1, 1:-1, 1:-1]).all()


@pytest.mark.parametrize("field", FIELDS)
@pytest.mark.parametrize("chunk", [1, 4, 40])
@pytest.mark.parametrize("shape", SHAPES)
def test_forced_pairs_equal_single_steps(launch_override, shape, chunk, field):
    T0, C, inv, dt = setup(shape, field)

    def run(nt, temporal2):
        T, T2 = T0.clone(), torch.full_like(T0, 7.0)
        out = api.run(T, T2, C, 0.9, dt, inv, nt, temporal2=temporal2)
        return out, T2 if out is T else T

    for nt in (4, 9):
        launch_override(kchunk=16, kchunk2=0)
        want = run(nt, False)
        launch_override(kchunk=0, kchunk2=chunk)
        assert api.step_kernel_name(T0.clone(), T0, C, 0.9, dt, inv, temporal2=True) == "k_zpair<F32>"
        check_spread(field, want[0])
        for x, y in zip(run(nt, False), want):  # the default loop: its last step a single one
            assert same(to_host(x), to_host(y))
        assert same(to_host(run(nt, True)[0]), to_host(want[0]))
    assert api.device_error() == 0


@pytest.mark.parametrize("field", FIELDS)
@pytest.mark.parametrize("nt,every", [(5, 1), (9, 3)])
@pytest.mark.parametrize("shape", SHAPES)
def test_kept_states_equal_single_steps(launch_override, shape, nt, every, field):
    T0, C, inv, dt = setup(shape, field)

    def run(temporal2):
        block = api.StateBlock(T0, nt // every + (2 if every > 1 else 0), boundary=False)
        block.flat.fill_(7.0)
        out = api.run_states(T0, block, every, C, 0.9, dt, inv, nt, temporal2=temporal2)
        return [to_host(g) for g in block.grids[:nt // every]] + [to_host(out)]

    launch_override(kchunk=16, kchunk2=0)
    want = run(False)
    launch_override(kchunk=0)
    for chunk in (1, 4, 40):
        launch_override(kchunk2=chunk)
        for x, y in zip(run(True), want):
            assert same(x, y)
    assert api.device_error() == 0


# (nt, every) with one pair and one single, pairs only, singles between kept states, no kept state
PLANS = [(1, 1), (2, 1), (3, 1), (8, 1), (7, 2), (9, 3), (10, 5), (4, 7)]


@pytest.mark.parametrize("nt,every", PLANS)
@pytest.mark.parametrize("shape", [(13, 21, 68), (19, 37, 132), (7, 9, 36)])
def test_kept_states_plans_from_the_graph_cache(launch_override, shape, nt, every):
    """Replayed and with unset grids: every kept state, its boundary, and T(nt)."""
    T0, C, inv, dt = setup(shape, "random")
    launch_override(kchunk=16, kchunk2=0)
    cur, want = T0.clone(), []
    nxt = cur.clone()
    for t in range(1, nt + 1):
        api.step(nxt, cur, C, 0.9, dt, inv)
        cur, nxt = nxt, cur
        if t % every == 0:
            want.append(cur.clone())
    launch_override(kchunk=0, kchunk2=4)
    block = api.StateBlock(T0, nt // every + (2 if every > 1 else 0), boundary=False)
    for _ in range(3):  # captured, then replayed
        block.flat.fill_(float("nan"))
        out = api.run_states(T0, block, every, C, 0.9, dt, inv, nt, graph=True, temporal2=True)
        for g, w in zip(block.grids, want):
            assert torch.equal(g, w)
        assert torch.equal(out, cur)
    api.clear_graph_cache()
    assert api.device_error() == 0


@pytest.mark.parametrize("every", [1, 3, 20])
def test_gradient_with_forced_pairs(launch_override, every):
    """Forward pass and recomputes in pairs: the gradient of single steps, bit for bit."""
    D0, C, inv, dt = setup((13, 21, 68), "random")
    Tobs, got = D0 * 0.98, []
    for pairs in (False, True):
        launch_override(kchunk2=4 if pairs else 0)
        got.append(autograd.loss_and_grad(D0, C, Tobs, 0.9, dt, inv, 10, every=every, state_pairs=pairs))
    for a, b in zip(*got):
        assert torch.equal(a, b)
    assert torch.count_nonzero(got[0][2]) > 0


@pytest.mark.parametrize("n,nt", [(1296, 5), (196, 9)])
def test_default_loop_takes_pairs(launch_override, n, nt):
    """Without flag or override, past 2^31 elements and on a size that no tile divides."""
    T0 = inputs.uniform_field_torch(3, n, n, n, "cuda").float()
    C = (0.5 + 0.25 * inputs.uniform_field_torch(4, n, n, n, "cuda")).float()
    assert api.step_kernel_name(T0.clone(), T0, C, 1.0, 1e-7, (n - 1.0,) * 3, temporal2=True) == "k_zpair<F32>"

    def run():
        T, T2 = T0.clone(), torch.empty_like(T0)
        return api.run(T, T2, C, 1.0, 0.1 / n ** 2, (n - 1.0,) * 3, nt), T, T2

    launch_override(kchunk=16)
    want = run()
    launch_override(kchunk=0)
    for a, b in zip(run(), want):
        assert torch.equal(a, b)
    assert api.device_error() == 0
