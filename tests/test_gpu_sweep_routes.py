"""The kernels that share the work of a sweep call, at the sizes where one
takes over from another: bit-exact against the oracle or against the same
lattice swept along another route."""
import numpy as np
import pytest
import torch

import oracle
import paper_1906_06297_gb300 as ising

pytestmark = pytest.mark.gpu
BETA = 0.4406868


@pytest.fixture(scope="module", autouse=True)
def built():
    ising.build()
    oracle.build()


# 1536 / 1600: one and four half words per thread of the flat kernel (1024 half
# words per SM of 152); the last row of a block's range is ragged in both
@pytest.mark.parametrize("L,stride", [(1536, None), (1600, 1600 // 4 + 16)])
def test_flat_kernel_matches_oracle_at_its_edges(L, stride):
    lat = ising.Lattice(L, "msc4", row_stride_bytes=stride)
    ising.ising_init_lattice(lat, ising.ISING_INIT_RANDOM, 7)
    trace = torch.zeros((2, 2), dtype=torch.int64, device="cuda")
    ising.ising_sweep(lat, BETA, 2, 7, 5, trace)
    s = oracle.init(L, oracle.MODE_RANDOM, 7)
    want = oracle.run(s, BETA, 2, 7, 5)
    assert np.array_equal(oracle.from_planes_msc4(L, *lat.planes_numpy()), s)
    assert np.array_equal(trace.cpu().numpy(), want)


# whole calls in one cluster: one CTA up to 16, one and two half words per
# thread, bands of unequal rows, rows with a partial last half word and draws
# that start inside a Philox block, recorded beyond one block of trace rows, and
# the largest side of that route and the sides above it
@pytest.mark.parametrize("layout,L,n,stride", [
    ("int8", 2, 3, None), ("int8", 4, 2, 3), ("int8", 14, 3, None), ("int8", 34, 3, 20), ("int8", 62, 600, None),
    ("int8", 130, 5, None), ("int8", 144, 4, None), ("msc4", 64, 520, None), ("msc4", 192, 6, 64), ("msc4", 320, 4, None),
    ("int8", 398, 3, None), ("int8", 402, 2, None), ("int8", 496, 2, 300), ("msc4", 512, 3, None), ("int8", 512, 2, None),
    ("msc4", 576, 2, None), ("int8", 766, 2, None), ("int8", 782, 2, None)])
@pytest.mark.parametrize("beta", [0.0, BETA])
def test_small_lattice_calls_match_oracle(layout, L, n, stride, beta):
    lat = ising.Lattice(L, layout, row_stride_bytes=stride)
    lat.black.fill_(85)
    lat.white.fill_(85)
    ising.ising_init_lattice(lat, ising.ISING_INIT_RANDOM, 6)
    s = oracle.init(L, oracle.MODE_RANDOM, 6)
    for off in (3, 2**32 - 1):  # the second call's sweep index crosses 32 bits
        trace = torch.full((n, 2), 77, dtype=torch.int64, device="cuda")
        ising.ising_sweep(lat, beta, n, 6, off, trace)
        want = oracle.run(s, beta, n, 6, off)
        unpack = oracle.from_planes_int8 if layout == "int8" else oracle.from_planes_msc4
        assert np.array_equal(unpack(L, *lat.planes_numpy()), s)
        assert np.array_equal(trace.cpu().numpy(), want)
    assert (lat.black[:, lat.row_bytes:] == 85).all() and (lat.white[:, lat.row_bytes:] == 85).all()


# rows of whole 16-byte and 4-byte words, rows that are neither, and strides
# that take an aligned row length off its alignment; blocks of 4 sites that
# straddle row ends, and the largest L/2 that no kernel but the general one takes
@pytest.mark.parametrize("L,stride", [(6, None), (8, None), (8, 5), (26, None), (30, 17), (32, None), (32, 24),
                                      (34, None), (40, None), (96, None), (96, 50), (1286, None), (2560, None)])
@pytest.mark.parametrize("beta", [0.0, BETA, 50.0])
def test_int8_kernels_match_oracle(L, stride, beta):
    lat = ising.Lattice(L, "int8", row_stride_bytes=stride)
    ising.ising_init_lattice(lat, ising.ISING_INIT_RANDOM, 4)
    n = 3 if L < 1000 else 1
    trace = torch.zeros((n, 2), dtype=torch.int64, device="cuda")
    ising.ising_sweep(lat, beta, n, 4, 2, trace)
    s = oracle.init(L, oracle.MODE_RANDOM, 4)
    want = oracle.run(s, beta, n, 4, 2)
    assert np.array_equal(oracle.from_planes_int8(L, *lat.planes_numpy()), s)
    assert np.array_equal(trace.cpu().numpy(), want)


# 13824^2 / 13888^2 lie on the two sides of the marching kernel's smallest size;
# slabs of a third of their rows take the flat kernel in both cases
@pytest.mark.parametrize("L", [13824, 13888])
def test_flat_and_marching_kernels_agree(L):
    lat = ising.Lattice(L, "msc4")
    ising.ising_init_lattice(lat, ising.ISING_INIT_RANDOM, 3)
    slabs = []
    for r0, rows in ising.slab_partition(L, 3):
        sl = ising.Slab(L, r0, rows)
        ising.ising_slab_init(sl, ising.ISING_INIT_RANDOM, 3)
        slabs.append(sl)
    a, b = (torch.zeros((2, 2), dtype=torch.int64, device="cuda") for _ in range(2))
    ising.ising_sweep(lat, BETA, 2, 3, 0, a)
    ising.ising_slab_sweep(slabs, BETA, 2, 3, 0, b)
    assert torch.equal(a, b)
    for colour in ("black", "white"):
        assert torch.equal(getattr(lat, colour), torch.cat([getattr(sl, colour)[1:-1] for sl in slabs]))


@pytest.mark.parametrize("layout,L,n", [("msc4", 256, 1), ("msc4", 1088, 3), ("int8", 130, 4)])
def test_captured_sweeps_replay_as_called(layout, L, n):
    """A sweep call recorded into a CUDA graph and replayed twice equals the
    same call made twice."""
    a, b = ising.Lattice(L, layout), ising.Lattice(L, layout)
    for lat in (a, b):
        ising.ising_init_lattice(lat, ising.ISING_INIT_RANDOM, 9)
    ta, tb = (torch.zeros((n, 2), dtype=torch.int64, device="cuda") for _ in range(2))
    ising.ising_sweep(a, BETA, n, 9, 0, ta)
    ising.ising_sweep(a, BETA, n, 9, 0, ta)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ising.ising_sweep(b, BETA, n, 9, 0, tb)
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(a.black, b.black) and torch.equal(a.white, b.white) and torch.equal(ta, tb)


# one-byte rows on and off 16-byte boundaries: the wide and the byte-wise conversions
@pytest.mark.parametrize("L,stride", [(64, None), (192, None), (192, 97), (448, 240)])
def test_conversions_at_any_row_alignment(L, stride):
    a, b = ising.Lattice(L, "int8", row_stride_bytes=stride), ising.Lattice(L, "int8", row_stride_bytes=stride)
    m = ising.Lattice(L, "msc4")
    for lat in (a, b):
        lat.black.fill_(85)
        lat.white.fill_(85)
    ising.ising_init_lattice(a, ising.ISING_INIT_RANDOM, 8)
    s = oracle.init(L, oracle.MODE_RANDOM, 8)
    ising.ising_pack(a, m)
    assert np.array_equal(oracle.from_planes_msc4(L, *m.planes_numpy()), s)
    ising.ising_unpack(m, b)
    assert torch.equal(a.black, b.black) and torch.equal(a.white, b.white)
    obs = torch.zeros((2, 2), dtype=torch.int64, device="cuda")
    ising.ising_observables(a, obs[0])
    ising.ising_observables(m, obs[1])
    want = [int(s.sum()), int((s.astype(int) * (np.roll(s, -1, 0) + np.roll(s, -1, 1))).sum())]
    assert obs.tolist() == [want, want]


# the cluster kernel's halo rows over many sweeps: 2 to 16 CTAs, a draw thread
# per half word and two, ragged rows of one and two half words per thread, and
# more sweeps than one launch takes
@pytest.mark.parametrize("layout,L,n", [
    ("int8", 48, 2000), ("msc4", 128, 1500), ("int8", 100, 1500), ("int8", 256, 1500), ("msc4", 384, 400),
    ("int8", 450, 150), ("int8", 498, 130), ("int8", 510, 130), ("int8", 512, 300), ("int8", 32, 16500)])
def test_cluster_sweeps_stay_in_step(layout, L, n):
    lat = ising.Lattice(L, layout)
    ising.ising_init_lattice(lat, ising.ISING_INIT_RANDOM, 8)
    s = oracle.init(L, oracle.MODE_RANDOM, 8)
    trace = torch.full((n, 2), 77, dtype=torch.int64, device="cuda")
    ising.ising_sweep(lat, BETA, n, 8, 1, trace)
    want = oracle.run(s, BETA, n, 8, 1)
    unpack = oracle.from_planes_int8 if layout == "int8" else oracle.from_planes_msc4
    assert np.array_equal(unpack(L, *lat.planes_numpy()), s)
    assert np.array_equal(trace.cpu().numpy(), want)
