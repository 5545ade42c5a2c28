"""The one-byte kernel for planes of 2^32 sites and more (sides from 92682 on), whose
indices are 64-bit throughout.  Compiled here on its own and launched on small planes,
any of which it takes: bit-exact against the oracle."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
import paper_1906_06297_gb300 as ising
from paper_1906_06297_gb300 import _build

pytestmark = pytest.mark.gpu

_SRC = r"""
#include "int8.cu"

namespace ising {
cudaError_t device_info(DeviceInfo *info)
{
    return cudaDeviceGetAttribute(&info->sm_count, cudaDevAttrMultiProcessorCount, 0);
}
}

// One sweep of planes of L rows of `stride` bytes (black's, then white's, in place; host arrays).
extern "C" __attribute__((visibility("default"))) int run_sweep(long long L, long long stride, unsigned long long T3,
                                                                unsigned long long T4, unsigned long long seed,
                                                                unsigned long long t, void *planes, long long *obs_out)
{
    using namespace ising;
    const size_t plane = (size_t)L * stride;
    if (L < 2 || L % 2 || stride < L / 2) return -1;
    int8_t *d = nullptr;
    long long *obs = nullptr;
    cudaError_t e = cudaMalloc(&d, 2 * plane);
    if (e == cudaSuccess) e = cudaMalloc(&obs, 16);
    if (e == cudaSuccess) e = cudaMemcpy(d, planes, 2 * plane, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(obs, 0, 16);
    if (e == cudaSuccess) {
        Int8SweepParams p = {};
        p.L = L;
        p.half = L / 2;
        p.stride = stride;
        p.nblk = (L * (L / 2) + 3) / 4;
        p.c2 = (uint32_t)t;
        p.acc.T3_64 = T3;
        p.acc.T4_64 = T4;
        p.rk = make_round_keys(seed);
        p.obs = obs;
        const unsigned grid = (unsigned)((p.nblk + 4 * kThreads - 1) / (4 * kThreads));  // some threads take several blocks
        p.tgt = d, p.src = d + plane;
        p.c3 = counter_word3(0, kPurposeMetropolis, t);
        int8_sweep_kernel<0, false><<<grid, kThreads>>>(p);
        p.tgt = d + plane, p.src = d;
        p.c3 = counter_word3(1, kPurposeMetropolis, t);
        int8_sweep_kernel<1, true><<<grid, kThreads>>>(p);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(planes, d, 2 * plane, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(obs_out, obs, 16, cudaMemcpyDeviceToHost);
    cudaFree(d);
    cudaFree(obs);
    return (int)e;
}
"""


@pytest.fixture(scope="module")
def sweep(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    oracle.build()
    ising.build()
    d = tmp_path_factory.mktemp("int8")
    (d / "sweep.cu").write_text(_SRC)
    subprocess.run([nvcc, *_build.NVCC_FLAGS, f"-I{_build.CSRC}", "-shared", str(d / "sweep.cu"), "-o", str(d / "sweep.so")],
                   check=True)
    fn = ctypes.CDLL(str(d / "sweep.so")).run_sweep
    i64, u64, P = ctypes.c_longlong, ctypes.c_uint64, ctypes.c_void_p
    fn.argtypes = [i64, i64, u64, u64, u64, u64, P, P]
    return fn


@pytest.mark.parametrize("L,stride", [(2, 1), (6, 3), (10, 8), (34, 17), (64, 32), (130, 80), (258, 129)])
@pytest.mark.parametrize("beta", [0.0, 0.4406868, 50.0])
def test_general_kernel_matches_oracle(sweep, L, stride, beta):
    s = np.where(np.random.default_rng(L).random((L, L)) < 0.55, 1, -1).astype(np.int8)
    planes = np.full((2, L, stride), 85, dtype=np.int8)
    planes[:, :, :L // 2] = np.stack(oracle.to_planes_int8(s))
    T = ising.ising_thresholds(beta)
    obs = np.zeros(2, dtype=np.int64)
    assert sweep(L, stride, int(T[3]), int(T[4]), 9, 2**32 + 3, planes.ctypes.data, obs.ctypes.data) == 0
    for colour in (0, 1):
        oracle.half_sweep(s, beta, colour, 9, 2**32 + 3)
    assert np.array_equal(oracle.from_planes_int8(L, *planes[:, :, :L // 2]), s)
    assert (planes[:, :, L // 2:] == 85).all()
    assert np.array_equal(obs, oracle.observables(s))
