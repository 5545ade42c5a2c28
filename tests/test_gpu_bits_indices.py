"""The bit-plane half-sweeps on rows whose word indices in the plane pass 2^32
(sides above 524288).  Such planes take 180 GB, so the kernel is compiled here on
its own and given plane pointers from which only the rows around the band exist:
an index that lost its high bits would not reach them."""
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
#include "bits.cu"

namespace ising {
cudaError_t device_info(DeviceInfo *info)
{
    return cudaDeviceGetAttribute(&info->sm_count, cudaDevAttrMultiProcessorCount, 0);
}
}

// Rows row0 - 1 .. row0 + rows of both bit planes in (black's, then white's), the
// same of the swept plane and its MSC4 rows row0 .. out, for one half-sweep of `rows`
// rows that touch neither end of the plane (host arrays).
extern "C" __attribute__((visibility("default"))) int run_band(int colour, long long L, long long row0, long long rows, unsigned T3, unsigned T4,
                        unsigned always, unsigned long long seed, unsigned long long t, const void *planes, void *bits_out,
                        void *msc4_out, long long *obs_out)
{
    using namespace ising;
    if (colour < 0 || colour > 1 || L % 64 || row0 < 1 || rows < 1 || row0 + rows >= L) return -1;
    const size_t plane = (size_t)(rows + 2) * (L / 64) * 4, msc4 = (size_t)rows * (L / 32) * 8;
    char *d = nullptr;
    cudaError_t e = cudaMalloc(&d, 2 * plane + msc4 + 16);
    if (e != cudaSuccess) return (int)e;
    long long *obs = (long long *)(d + 2 * plane + msc4);
    e = cudaMemcpy(d, planes, 2 * plane, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(obs, 0, 16);
    BitsSweepParams p = {};
    for (int c = 0; c < 2; ++c) {
        p.bits[c] = (uint32_t *)((uintptr_t)(d + c * plane) - (uintptr_t)(row0 - 1) * (L / 64) * 4);
        p.msc4[c] = (uint64_t *)((uintptr_t)(d + 2 * plane) - (uintptr_t)row0 * (L / 32) * 8);
    }
    p.L = L;
    p.stride_words = L / 32;
    p.c2 = (uint32_t)t;
    p.c3 = counter_word3(0, kPurposeMetropolis, t);
    p.acc.T3 = T3;
    p.acc.T4 = T4;
    p.acc.always = always;
    p.rk = make_round_keys(seed);
    p.obs = obs;
    p.n = 1;
    p.band[0] = BitsBand{colour, row0, rows};
    if (e == cudaSuccess) e = bits_half_sweeps(p, 0);
    if (e == cudaSuccess) e = cudaMemcpy(bits_out, d + colour * plane, plane, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(msc4_out, d + 2 * plane, msc4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(obs_out, obs, 16, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
"""


@pytest.fixture(scope="module")
def band(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    oracle.build()
    ising.build()
    d = tmp_path_factory.mktemp("bits")
    (d / "band.cu").write_text(_SRC)
    subprocess.run([nvcc, *_build.NVCC_FLAGS, f"-I{_build.CSRC}", "-shared", str(d / "band.cu"), "-o", str(d / "band.so")],
                   check=True)
    fn = ctypes.CDLL(str(d / "band.so")).run_band
    i64, u32, u64, P = ctypes.c_longlong, ctypes.c_uint32, ctypes.c_uint64, ctypes.c_void_p
    fn.argtypes = [ctypes.c_int, i64, i64, i64, u32, u32, u32, u64, u64, P, P, P, P]
    return fn


def colour_bits(s, colour, first):
    """Sites of one colour of rows `first` .. of the lattice as 0/1, in column order."""
    return np.stack([(s[k, (first + k + colour) % 2::2] > 0) for k in range(len(s))]).astype(np.uint8)


# word index 2^32 lies between rows 508400 and 508401 of 540672^2; 185408^2 is the
# first side with 64-bit counters, 32768^2 is far below either
@pytest.mark.parametrize("L,row0", [(540672, 508398), (540672, 540660), (185408, 185400), (32768, 20000)])
@pytest.mark.parametrize("colour", [0, 1])
@pytest.mark.parametrize("beta", [0.4406868, 0.0])
def test_band_rows_match_the_oracle(band, L, row0, colour, beta):
    rows, seed, t = 6, 0x1234567890ABCDEF, 2**33 + 5
    s = np.where(np.random.default_rng(row0).random((rows + 2, L)) < 0.6, 1, -1).astype(np.int8)
    planes = [np.packbits(colour_bits(s, c, row0 - 1), axis=1, bitorder="little") for c in (0, 1)]
    src = np.ascontiguousarray(np.stack(planes))
    got, msc4, obs = np.zeros_like(planes[0]), np.zeros((rows, L // 4), np.uint8), np.zeros(2, np.int64)
    T = ising.ising_thresholds(beta)
    T3, T4 = (min(int(T[k]), 2**32 - 1) for k in (3, 4))
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    rc = band(colour, L, row0, rows, T3, T4, int(T[3] >= 2**32), seed, t, ptr(src), ptr(got), ptr(msc4), ptr(obs))
    assert rc == 0
    want = s.copy()
    for k in range(1, rows + 1):
        oracle.update_row(L, s[k - 1].copy(), want[k], s[k + 1].copy(), row0 - 1 + k, colour, beta, seed, t)
    bits = colour_bits(want, colour, row0 - 1)
    assert np.array_equal(got, np.packbits(bits, axis=1, bitorder="little"))
    assert np.array_equal(msc4, bits[1:-1, 0::2] | (bits[1:-1, 1::2] << 4))
    if colour == 1:
        w = want.astype(np.int64)
        side = np.roll(w, 1, 1) + np.roll(w, -1, 1)
        bonds = sum(int((w[k] * (w[k - 1] + w[k + 1] + side[k]))[(row0 + k) % 2::2].sum()) for k in range(1, rows + 1))
        assert list(obs) == [int(w[1:-1].sum()), bonds]
    else:
        assert list(obs) == [0, 0]
