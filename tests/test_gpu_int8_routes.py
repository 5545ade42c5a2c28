"""One-byte kernels at sides and strides that the routes of whole sweep calls keep
from them: single sweeps beside the cluster kernel's largest sides, and half-sweeps,
which never take that kernel, on rows of every alignment.  Bit-exact against the
oracle."""
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


@pytest.mark.parametrize("L,stride", [(254, None), (258, None), (318, 161), (398, None), (400, None), (416, 224), (448, None),
                                      (510, 256), (512, None)])
def test_single_sweeps_match_oracle(L, stride):
    lat = ising.Lattice(L, "int8", row_stride_bytes=stride)
    ising.ising_init_lattice(lat, ising.ISING_INIT_RANDOM, 4)
    s = oracle.init(L, oracle.MODE_RANDOM, 4)
    for t in range(3):
        trace = torch.full((1, 2), 77, dtype=torch.int64, device="cuda")
        ising.ising_sweep(lat, BETA, 1, 4, t, trace)
        want = oracle.run(s, BETA, 1, 4, t)
        assert np.array_equal(oracle.from_planes_int8(L, *lat.planes_numpy()), s)
        assert np.array_equal(trace.cpu().numpy(), want)


# rows of whole aligned 16-byte groups, dense and padded (int8_words_kernel); the same
# L/2 with a stride or a plane that is not (int8_rows_kernel); a single site per row, rows
# shorter than a unit, and rows whose Philox blocks straddle their ends; units of one
# word up to 512 of them per SM, else of four, dense and padded
@pytest.mark.parametrize("L,stride,offset", [
    (32, None, 0), (32, 32, 0), (96, 64, 0), (2560, 1312, 0),
    (32, 24, 0), (96, 50, 0), (96, None, 4), (96, None, 16), (96, None, 1), (2560, 1284, 0),
    (2, None, 0), (6, 5, 3), (30, 17, 0), (34, None, 2),
    (1024, 514, 0), (1286, None, 0), (1286, 647, 5), (2050, None, 0),
])
@pytest.mark.parametrize("beta", [0.0, BETA, 50.0])
def test_half_sweeps_match_oracle(L, stride, offset, beta):
    """Planes that start `offset` bytes into an allocation; the bytes around their
    rows stay what they were."""
    stride = stride or L // 2
    bufs = [torch.full((L * stride + offset + 64,), 85, dtype=torch.int8, device="cuda") for _ in range(2)]
    s = np.where(np.random.default_rng(L).random((L, L)) < 0.55, 1, -1).astype(np.int8)
    planes = [b[offset:offset + L * stride].view(L, stride) for b in bufs]
    for p, h in zip(planes, oracle.to_planes_int8(s)):
        p[:, :L // 2] = torch.from_numpy(h).cuda()
    lat = ising.ising_lattice_t(planes[0].data_ptr(), planes[1].data_ptr(), L, ising.ISING_INT8, 0, stride)
    obs = torch.zeros(2, dtype=torch.int64, device="cuda")
    for colour in (0, 1):
        ising.ising_half_sweep(lat, beta, colour, 9, 2**32 + 3, obs if colour else None)
        oracle.half_sweep(s, beta, colour, 9, 2**32 + 3)
    got = [p[:, :L // 2].cpu().numpy() for p in planes]
    assert np.array_equal(oracle.from_planes_int8(L, *got), s)
    assert np.array_equal(obs.cpu().numpy(), oracle.observables(s))
    for b, p in zip(bufs, planes):
        p[:, :L // 2] = 85
        assert (b == 85).all()
