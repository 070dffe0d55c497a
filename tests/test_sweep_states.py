"""The states that a reverse sweep takes by address: refused like the tensors they stand for when they are no
fields like the cotangent, and, as checkpoints, the list of tensors that they stand for."""
import pytest
import torch

from paper_2211_15634_gb300 import api, autograd as ag


class Block:
    """A state block of host memory."""

    def __init__(self, like, count):
        n = like.numel()
        self.flat = torch.arange(count * n, dtype=like.dtype)
        self.grids = api._GridViews(self.flat, n, count, tuple(like.shape))


def every_state(nt=5, shape=(3, 4, 5)):
    T0 = torch.zeros(shape)
    return ag._EveryState(T0, Block(T0, nt), nt)


@pytest.mark.parametrize("like", [torch.zeros(3, 4, 6), torch.zeros(3, 4, 5, dtype=torch.float64),
                                  torch.zeros(3, 4, 5, device="meta")])
def test_other_fields_are_refused(like):
    kept = every_state()
    for call in (lambda: ag._block_addresses(kept.block, 2, like), lambda: kept.states(5, like)):
        with pytest.raises(ValueError):
            call()


def test_addresses_last_state_first():
    kept = every_state()
    like = torch.ones(3, 4, 5)
    for nt in (0, 1, 4, 5, 9):
        got = kept.states(nt, like)
        assert len(got) == min(nt, 5)
        if got:
            assert got.pop() is kept.T0
            assert got == [kept[i].data_ptr() for i in range(min(nt, 5) - 1, 0, -1)]
    with pytest.raises(IndexError):
        ag._block_addresses(kept.block, 6, like)


def test_checkpoints_read_as_a_list():
    kept = every_state()
    plain = [kept.T0] + [kept.block.grids[i] for i in range(4)]
    same = lambda a, b: len(a) == len(b) and all(torch.equal(x, y) for x, y in zip(a, b))
    assert same(list(kept), plain) and same(kept[1:4], plain[1:4]) and same(kept[::-2], plain[::-2])
    assert same([plain[0]] + kept, [plain[0]] + plain) and same(kept + [plain[0]], plain + [plain[0]])
    assert torch.equal(kept[-1], plain[-1]) and same(list(reversed(kept)), plain[::-1])
    for i in (5, -6):
        with pytest.raises(IndexError):
            kept[i]


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")
@pytest.mark.parametrize("every", [1, 2, 3])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_backward_refuses_other_fields(every, dtype):
    """A cotangent and a coefficient of another grid or type than the forward's, before any launch."""
    shape, inv, dt, nt = (8, 7, 12), (3.0, 3.5, 4.0), 0.001, 6
    T0, Ci = (0.5 + torch.rand(shape, device="cuda", dtype=dtype) for _ in range(2))
    out, ckpts, kept = ag.forward_checkpointed(T0, Ci, 1.0, dt, inv, nt, every)
    other = torch.float32 if dtype == torch.float64 else torch.float64
    for y, C in ((torch.ones((8, 7, 16), device="cuda", dtype=dtype),) * 2, (out.to(other), Ci.to(other)),
                 (torch.ones((7, 8, 12), device="cuda", dtype=dtype),) * 2):
        with pytest.raises((ValueError, TypeError)):
            ag.backward_checkpointed(y, C, 1.0, dt, inv, nt, every, ckpts, kept=None if kept is None else dict(kept))
    dT0, dCi = ag.backward_checkpointed(out.clone(), Ci, 1.0, dt, inv, nt, every, ckpts, kept=kept)
    assert dT0.shape == out.shape and torch.isfinite(dCi).all()
    # the steps asked for, not all that were kept
    if every == 1:
        got = ag.backward_checkpointed(out.clone(), Ci, 1.0, dt, inv, 2, 1, ckpts)
        want = ag.backward_checkpointed(out.clone(), Ci, 1.0, dt, inv, 2, 1, list(ckpts)[:2])
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    torch.cuda.synchronize()
