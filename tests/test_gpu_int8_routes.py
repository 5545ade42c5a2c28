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
