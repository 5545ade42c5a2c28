"""The bounded waits of the small-lattice sweeps: one that runs out is reported by
ising_sweep_check, once, and neither refuses nor disturbs any other sweep."""
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


def swept(layout, L):
    lat = ising.Lattice(L, layout)
    ising.ising_init_lattice(lat, ising.ISING_INIT_RANDOM, 5)
    return lat


def assert_right(lat, n, unpack):
    s = oracle.init(lat.L, oracle.MODE_RANDOM, 5)
    oracle.run(s, BETA, n, 5)
    assert np.array_equal(unpack(lat.L, *lat.planes_numpy()), s)


# two CTAs, each of them both neighbours of the other; four; ragged rows; 16 CTAs, one
# and two half words per thread
@pytest.mark.parametrize("layout,L", [("int8", 48), ("msc4", 64), ("int8", 100), ("int8", 256), ("msc4", 512), ("int8", 510)])
def test_a_wait_that_runs_out_is_reported_once(layout, L):
    unpack = oracle.from_planes_int8 if layout == "int8" else oracle.from_planes_msc4
    torch.cuda.synchronize()
    ising.ising_sweep_check()
    bad, other = swept(layout, L), swept(layout, L)
    ising.ising_sweep_wait_selftest(bad)
    ising.ising_sweep(other, BETA, 7, 5)  # not refused, and not told
    with pytest.raises(ising.IsingError) as e:
        ising.ising_sweep_check()
    assert e.value.status == ising.ISING_ETIMEOUT
    ising.ising_sweep_check()  # the flag was cleared
    assert_right(other, 7, unpack)
    again = swept(layout, L)  # the device stays usable, on another stream too
    with torch.cuda.stream(torch.cuda.Stream()):
        torch.cuda.current_stream().wait_stream(torch.cuda.default_stream())
        ising.ising_sweep(again, BETA, 7, 5)
        ising.ising_sweep_check()
    assert_right(again, 7, unpack)


def test_the_self_test_refuses_lattices_that_one_cta_sweeps():
    for layout, L in (("int8", 8), ("msc4", 576)):
        with pytest.raises(ising.IsingError) as e:
            ising.ising_sweep_wait_selftest(swept(layout, L))
        assert e.value.status == ising.ISING_EINVAL
