"""Batches recorded and exchanged after every sweep, over many sweeps: owners that
run ahead of or behind one another between two records must still decide every
pair from the same state.  Planes, slot state and traces agree bit for bit with
the launch shape that shares every lattice (256 threads), and the two halves of
the slot state stay inverse permutations."""
import numpy as np
import pytest
import torch

import paper_1906_06297_gb300 as ising

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    ising.build()


@pytest.mark.parametrize("sides,per,S,n,traced", [
    ([32], 320, 8, 3000, True),      # about one chunk of work per owner and half-sweep
    ([32], 88000, 8, 60, False),     # more lattices per SM than a block has threads
    ([32, 256], 304, 16, 400, True),  # owners with unequal numbers of lattices
    ([96], 608, 4, 400, False),
])
def test_exchanges_after_every_sweep_stay_consistent(sides, per, S, n, traced):
    L = [x for x in sides for _ in range(per)]
    beta = np.linspace(0.40, 0.46, S)
    got = []
    for threads in (256, 512):
        b = ising.Batch(L, S, beta)
        b.config(threads, 4)
        b.init(ising.ISING_INIT_RANDOM, 11)
        tr = torch.zeros((n, b.n, 2), dtype=torch.int64, device="cuda") if traced else None
        b.run(n, 11, 0, 1, True, tr)
        b.run(3, 11, n, 1, True, None)  # the next call goes on from the state this one left
        b.check()
        slot, at = (np.asarray(x).reshape(-1) for x in b.state_numpy())
        assert np.array_equal(np.sort(at), np.arange(b.n))
        assert np.array_equal(slot[at], np.arange(b.n) % S)
        assert (slot != np.arange(b.n) % S).any()  # exchanges happened
        words = 8 * int(b.word_off[-1])
        got.append([b.ws[o:o + words].clone() for o in (b._black_off, b._white_off)] + ([tr] if traced else []) +
                   [torch.from_numpy(slot.copy()), torch.from_numpy(at.copy())])
    for x, y in zip(*got):
        assert torch.equal(x, y)


@pytest.mark.parametrize("sides,per,S", [([32, 64, 128], 4, 4), ([64], 160, 8)])
def test_short_allocation_free_runs_equal_batch_runs(sides, per, S):
    """Runs of a few sweeps, which the allocation-free call lets the grid share, and of
    more, whose lattices it deals to SMs: the same planes, slot state and traces as
    those of a batch that goes on from the same state."""
    L = [x for x in sides for _ in range(per)]
    beta = np.linspace(0.40, 0.46, S)
    ref = ising.Batch(L, S, beta)
    ref.init(ising.ISING_INIT_RANDOM, 4)
    words = 8 * int(ref.word_off[-1])
    parts = ((ref._black_off, words), (ref._white_off, words), (ref._slot_off, 4 * ref.n), (ref._at_off, 4 * ref.n))
    torch.cuda.synchronize()
    mine = [ref.ws[o:o + k].clone() for o, k in parts]
    t = 0
    for n in (1, 2, 3, 4, 5, 1):
        a, b = (torch.zeros((n, ref.n, 2), dtype=torch.int64, device="cuda") for _ in range(2))
        ref.run(n, 4, t, 1, True, a)
        ref.check()
        ising.ising_batch_run_noalloc(L, S, beta, *mine, n, 4, t, 1, True, b)
        t += n
        assert torch.equal(a, b)
        for (o, k), m in zip(parts, mine):
            assert torch.equal(ref.ws[o:o + k], m)
