"""Batches whose lattices are dealt to single SMs, pairs and quads of them, and
batches that the whole grid shares: planes, slot state and traces agree bit for
bit with the launch shape that always shares (256 threads), over runs that leave
an odd and an even number of records behind."""
import numpy as np
import pytest
import torch

import paper_1906_06297_gb300 as ising

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    ising.build()


@pytest.mark.parametrize("sides,per,S", [
    ([32], 320, 8),              # single SMs, some with more lattices than others
    ([64, 128, 256], 48, 16),    # the Binder study's sides
    ([96, 160], 64, 16),         # pairs of SMs
    ([192, 384], 40, 4),
    ([256], 16, 16),             # quads
    ([640], 4, 4),               # shared by the grid
    ([32], 3, 1),                # fewer lattices than SMs, nothing to exchange
])
def test_owned_lattices_equal_shared_ones(sides, per, S):
    L = [x for x in sides for _ in range(per)]
    beta = np.linspace(0.42, 0.46, S) if S > 1 else [0.44]
    got = []
    for threads in (256, 512):
        b = ising.Batch(L, S, beta)
        b.config(threads, 4)
        b.init(ising.ISING_INIT_RANDOM, 5)
        traces = []
        for n, off in ((7, 0), (5, 7)):  # records after sweeps 2, 4, 6 and 8, 10, 12
            ev = b.n_events(n, off, 2)
            tr = torch.full((ev, b.n, 2), 3, dtype=torch.int64, device="cuda")
            b.run(n, 5, off, 2, S > 1, tr)
            traces.append(tr)
        b.run(2, 5, 12, 1, S > 1, None)  # two more, not traced
        b.check()
        got.append((b.ws[b._black_off:b._black_off + 8 * int(b.word_off[-1])].clone(),
                    b.ws[b._white_off:b._white_off + 8 * int(b.word_off[-1])].clone(), *traces,
                    *(torch.from_numpy(x) for x in b.state_numpy())))
    for x, y in zip(*got):
        assert torch.equal(x, y)


def test_trace_needs_only_eight_byte_alignment():
    b = ising.Batch([64] * 8, 4, np.linspace(0.42, 0.46, 4))
    b.init(ising.ISING_INIT_RANDOM, 2)
    buf = torch.zeros(2 * 8 * 3 + 1, dtype=torch.int64, device="cuda")
    b.run(6, 2, 0, 2, True, buf[1:])
    b.check()
    c = ising.Batch([64] * 8, 4, np.linspace(0.42, 0.46, 4))
    c.init(ising.ISING_INIT_RANDOM, 2)
    tr = torch.zeros((3, 8, 2), dtype=torch.int64, device="cuda")
    c.run(6, 2, 0, 2, True, tr)
    c.check()
    assert torch.equal(buf[1:], tr.view(-1))
