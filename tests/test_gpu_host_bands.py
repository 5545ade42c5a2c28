"""Host-resident single sweeps at the edges of their routes: whole planes below
three bands, row bands above, half-sweeps on the bit planes themselves.  Host
planes, trace and the device lattice equal ising_sweep on the device bit for bit
(that path is compared with the oracle elsewhere)."""
import pytest
import torch

import paper_1906_06297_gb300 as ising

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    ising.build()


def rows(lat, t):
    return t.view(lat.L, lat.row_stride_bytes)[:, :lat.row_bytes]


@pytest.mark.parametrize("fmt", ["bits", "msc4"])
@pytest.mark.parametrize("L,beta,pad", [
    (64, 0.4406868, 0), (192, 0.0, 16), (960, 0.6, 0),               # whole planes, one word per row on
    (3968, 0.4406868, 0), (4032, 0.4406868, 48), (7936, 0.0, 0),     # both sides of three bands (MSC4: 4000)
    (8000, 0.4406868, 0), (8064, 0.3, 16), (16448, 0.4406868, 0),    # bit planes from 8000: three, ramped bands
])
def test_host_sweep_equals_the_device_sweep(fmt, L, beta, pad):
    ref = ising.Lattice(L, "msc4")
    ising.ising_init_lattice(ref, ising.ISING_INIT_RANDOM, 3)
    dev = ising.Lattice(L, "msc4", row_stride_bytes=L // 4 + pad)
    nb = ising.ising_bits_bytes(L)
    stage = torch.empty(2 * nb, dtype=torch.uint8, device="cuda")

    def planes():
        if fmt == "msc4":
            return [rows(ref, ref.black).cpu(), rows(ref, ref.white).cpu()]
        bits = torch.empty(2 * nb, dtype=torch.uint8, device="cuda")
        ising.ising_msc4_to_bits(ref, bits[:nb], bits[nb:])
        return [bits[:nb].cpu(), bits[nb:].cpu()]

    host = [h.contiguous().pin_memory() for h in planes()]
    tr = [torch.zeros((1, 2), dtype=torch.int64, device="cuda") for _ in range(2)]
    tr_host = torch.zeros((1, 2), dtype=torch.int64).pin_memory()
    for k in range(3):
        if fmt == "bits":
            ising.ising_sweep_host_bits(dev, host[0], host[1], stage, beta, 1, 7, k, tr[0], tr_host.data_ptr())
        else:
            ising.ising_sweep_host(dev, host[0], host[1], beta, 1, 7, k, tr[0], tr_host.data_ptr())
        ising.ising_sweep(ref, beta, 1, 7, k, tr[1])
        torch.cuda.synchronize()
        assert all(torch.equal(h, e) for h, e in zip(host, planes()))
        assert torch.equal(rows(dev, dev.black), rows(ref, ref.black))
        assert torch.equal(rows(dev, dev.white), rows(ref, ref.white))
        assert torch.equal(tr_host, tr[1].cpu())


def test_philox_counters_above_32_bits():
    """185408^2 is the first side whose last rows need the counter's second word."""
    L = 185408
    ref, dev = ising.Lattice(L, "msc4"), ising.Lattice(L, "msc4")
    ising.ising_init_lattice(ref, ising.ISING_INIT_RANDOM, 3)
    nb = ising.ising_bits_bytes(L)
    stage = torch.empty(2 * nb, dtype=torch.uint8, device="cuda")
    ising.ising_msc4_to_bits(ref, stage[:nb], stage[nb:])
    host = [torch.empty(nb, dtype=torch.uint8, pin_memory=True) for _ in range(2)]
    host[0].copy_(stage[:nb])
    host[1].copy_(stage[nb:])
    tr = torch.zeros((2, 2), dtype=torch.int64, device="cuda")
    ising.ising_sweep_host_bits(dev, host[0], host[1], stage, 0.4406868, 1, 7, 0, tr[:1])
    ising.ising_sweep(ref, 0.4406868, 1, 7, 0, tr[1:])
    torch.cuda.synchronize()
    assert torch.equal(dev.black, ref.black) and torch.equal(dev.white, ref.white)
    assert torch.equal(tr[0], tr[1])
    ising.ising_msc4_to_bits(ref, stage[:nb], stage[nb:])
    assert torch.equal(host[0], stage[:nb].cpu()) and torch.equal(host[1], stage[nb:].cpu())
