"""Which sweep calls take the cluster kernel, against a fake of the runtime's answer
to how many clusters fit (no GPU): a device that cannot place a call's cluster
must leave it to the launches that serve every side."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_1906_06297_gb300 import _build

_SRC = r"""
#include <cuda_runtime.h>

static int g_limit, g_device, g_queries;

// A device with room for clusters of up to g_limit CTAs; below zero the query fails.
static cudaError_t fake_clusters(int *n, const cudaLaunchConfig_t *cfg)
{
    ++g_queries;
    if (g_limit < 0) return cudaErrorInvalidValue;
    *n = (int)cfg->attrs[0].val.clusterDim.x <= g_limit ? 1 : 0;
    return cudaSuccess;
}

#define cudaOccupancyMaxActiveClusters(n, kernel, cfg) fake_clusters(n, cfg)
#define cudaFuncSetAttribute(...) cudaSuccess
#define cudaGetDevice(d) (*(d) = g_device, cudaSuccess)
#define cudaGetLastError() cudaSuccess
#include "resident.cu"

extern "C" __attribute__((visibility("default"))) int fits(int device, int limit, long long L, long long n, int bytes, int *queries)
{
    g_device = device;
    g_limit = limit;
    g_queries = 0;
    const bool f = ising::resident_fits(L, n, bytes != 0);
    *queries = g_queries;
    return f;
}
"""


@pytest.fixture(scope="module")
def fits(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("resident")
    (d / "fits.cu").write_text(_SRC)
    subprocess.run([nvcc, *_build.NVCC_FLAGS, f"-I{_build.CSRC}", "-shared", str(d / "fits.cu"), "-o", str(d / "fits.so")],
                   check=True)
    fn = ctypes.CDLL(str(d / "fits.so")).fits
    fn.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int,
                   ctypes.c_void_p]

    def ask(device, limit, L, n=100, layout="int8"):
        q = ctypes.c_int(0)
        return bool(fn(device, limit, L, n, layout == "int8", ctypes.byref(q))), q.value

    return ask


def test_a_whole_device_takes_every_small_side(fits):
    for L in (2, 32, 64, 100, 254, 256, 384, 398, 498, 510, 512):
        assert fits(0, 16, L)[0]
    for L in (514, 576, 65536):
        assert fits(0, 16, L) == (False, 0)
    # asked once per kernel
    for L in (64, 100, 384, 510):
        assert fits(0, 16, L) == (True, 0)


@pytest.mark.parametrize("limit,fit,not_fit", [
    (-1, (2, 10, 32), (48, 64, 256, 512)),        # the query itself fails: single CTAs alone
    (1, (2, 10, 32), (48, 64, 100, 256, 512)),
    (4, (32, 48, 64), (128, 256, 254, 384, 512)),
    (8, (64, 100), (256, 384, 512, 510)),
])
def test_a_device_without_room_for_the_cluster_takes_the_launches(fits, limit, fit, not_fit):
    device = 10 + limit
    for L in fit:
        assert fits(device, limit, L)[0]
    for L in not_fit:
        assert not fits(device, limit, L)[0]


def test_single_sweeps_of_large_one_byte_lattices_take_the_launches(fits):
    """A cluster that loads, sweeps once and stores takes longer there than two
    launches of whatever kernel."""
    for L, n, layout, want in ((256, 1, "int8", True), (254, 1, "int8", True), (258, 1, "int8", False), (350, 1, "int8", False),
                               (398, 1, "int8", False), (400, 1, "int8", True), (416, 1, "int8", False),
                               (512, 1, "int8", False), (512, 1, "msc4", True), (512, 2, "int8", True),
                               (398, 2, "int8", True), (402, 2, "int8", False), (402, 6, "int8", True)):
        assert fits(30, 16, L, n, layout)[0] == want
