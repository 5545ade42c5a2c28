"""Every compile-time form of the threshold marks gives the same marks, in the flat
kernels' half words and in the cluster kernel's, which may start inside a Philox
block: the count of thresholds that each of the oracle's draws fails."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_1906_06297_gb300 import _build

pytestmark = pytest.mark.gpu

_SRC = r"""
#include "resident.cu"

namespace ising {
// Thread i: draws site[i] .. + 7 of the black half-sweep at t = 0.
__global__ void marks_kernel(const uint32_t *site, int n, DrawCtx dc, RoundKeys rk, uint32_t *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t b = site[i] >> 2, o = site[i] & 3u;
    out[3 * i] = marks8<true>(b, o, dc, rk);
    out[3 * i + 1] = o == 0 ? marks8<false>(b, 0u, dc, rk) : out[3 * i];
    out[3 * i + 2] = o == 0 && (b & 1) == 0 ? half_marks(b, 0u, dc, rk) : out[3 * i];
}
}

extern "C" __attribute__((visibility("default"))) int run_marks(const uint32_t *site, int n, unsigned T3, unsigned T4,
                                                                unsigned long long seed, uint32_t *out)
{
    using namespace ising;
    uint32_t *d = nullptr;
    cudaError_t e = cudaMalloc(&d, (size_t)n * 16);
    if (e == cudaSuccess) e = cudaMemcpy(d, site, (size_t)n * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        const DrawCtx dc{0u, counter_word3(0, kPurposeMetropolis, 0), T3, T4, 0u};
        marks_kernel<<<(n + 127) / 128, 128>>>(d, n, dc, make_round_keys(seed), d + n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, d + n, (size_t)n * 12, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
"""


@pytest.mark.parametrize("form", [0, 1, 2])
def test_marks_count_the_failed_thresholds(form, tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    oracle.build()
    (tmp_path / "marks.cu").write_text(_SRC)
    subprocess.run([nvcc, *_build.NVCC_FLAGS, f"-DISING_MSC4_MARK={form}", f"-I{_build.CSRC}", "-shared",
                    str(tmp_path / "marks.cu"), "-o", str(tmp_path / "marks.so")], check=True)
    fn = ctypes.CDLL(str(tmp_path / "marks.so")).run_marks
    P = ctypes.c_void_p
    fn.argtypes = [P, ctypes.c_int, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_uint64, P]
    seed, T3, T4 = 77, 3000000000, 1200000000
    site = np.arange(300, dtype=np.uint32)
    out = np.zeros((site.size, 3), dtype=np.uint32)
    assert fn(site.ctypes.data, site.size, T3, T4, seed, out.ctypes.data) == 0
    for i in range(site.size):
        want = 0
        for k in range(8):
            u = oracle.draw_stream(seed, 0, int(site[i]) + k, 0, 0)
            want |= (int(u >= T3) + int(u >= T4)) << (4 * k)
        assert list(out[i]) == [want] * 3
