// bits.cu -- the bit-packed I/O format of the host-resident sweep (one bit per
// spin in the order of the MSC4 nibbles, L/16 bytes per plane row): conversions
// from and to MSC4 colour planes, and half-sweeps on the bits.  Not part of the paper's method:
// MSC4 (Sec. 3.3) spends four bits per spin on the bit-parallel neighbour
// sums; storage and host transfers need one.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <type_traits>

#include "common.cuh"
#include "launch.h"

namespace ising {

// ---------------------------------------------------------------------------
// MSC4 plane rows <-> the bit-packed format (one bit per spin, L/16 bytes per
// row, dense rows): a thread converts pairs of words (32 spins each) <-> uint32.
// MSC4 -> bits: V adjacent pairs, 4 where that makes one aligned 16-byte store of
// bits, else 1 (16384^2, four planes in turn: 16.5 and 20.6 us per plane; four pairs
// a block's width apart 22.7); bits -> MSC4: kConvPairs pairs a block's width apart, so
// that each warp store is contiguous (16.7 us; by rows, with blocks that 256 pairs
// per row left three quarters idle, 20.5).  HBM-bound: 84 MB, 5.1 TB/s.
// ---------------------------------------------------------------------------
constexpr int kConvThreads = 256, kConvPairs = 4;

template <typename I, int V>
__global__ void __launch_bounds__(kConvThreads) msc4_to_bits_kernel(const uint64_t *plane, uint32_t *bits,
                                                                    int64_t stride_words, I pairs, I n)
{
    const I p = ((I)blockIdx.x * kConvThreads + threadIdx.x) * V;
    if (p >= n) return;
    const I r = p / pairs;
    const ulonglong2 *src =
        reinterpret_cast<const ulonglong2 *>(plane + (int64_t)r * stride_words) + (int64_t)(p - r * pairs);
    uint32_t out[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const ulonglong2 w = src[v];
        out[v] = msc4_word_to_bits(w.x) | (msc4_word_to_bits(w.y) << 16);
    }
    if constexpr (V == 4) *reinterpret_cast<uint4 *>(bits + p) = make_uint4(out[0], out[1], out[2], out[3]);
    else bits[p] = out[0];
}

template <typename I>
__global__ void __launch_bounds__(kConvThreads) bits_to_msc4_kernel(const uint32_t *bits, uint64_t *plane,
                                                                    int64_t stride_words, I pairs, I n)
{
    const I base = (I)blockIdx.x * (kConvThreads * kConvPairs) + threadIdx.x;
    uint32_t b[kConvPairs];
#pragma unroll
    for (int v = 0; v < kConvPairs; ++v) b[v] = base + kConvThreads * v < n ? bits[base + kConvThreads * v] : 0u;
#pragma unroll
    for (int v = 0; v < kConvPairs; ++v) {
        const I i = base + kConvThreads * v;
        if (i < n) {
            const I r = i / pairs;
            *reinterpret_cast<ulonglong2 *>(plane + (int64_t)r * stride_words + 2 * (int64_t)(i - r * pairs)) =
                make_ulonglong2(bits_to_msc4_word(b[v] & 0xFFFFu), bits_to_msc4_word(b[v] >> 16));
        }
    }
}

// Calls go(index, blocks) with an index type wide enough for n pairs, `per` of
// them per block.
template <typename Go>
cudaError_t conv_launch(int64_t n, int per, Go go)
{
    const int64_t blocks = (n + per - 1) / per;
    if (blocks > INT32_MAX) return cudaErrorInvalidConfiguration;
    if (n < (int64_t(1) << 31)) go(uint32_t{}, (unsigned)blocks);
    else go(uint64_t{}, (unsigned)blocks);
    return cudaGetLastError();
}

cudaError_t msc4_to_bits(const uint64_t *plane, int64_t stride_words, uint32_t *bits, int64_t L, int64_t rows,
                         cudaStream_t s)
{
    const int64_t pairs = L / 64, n = rows * pairs;
    const bool wide = pairs % 4 == 0 && (uintptr_t)bits % 16 == 0;
    return conv_launch(n, kConvThreads * (wide ? 4 : 1), [&](auto index, unsigned blocks) {
        using I = decltype(index);
        if (wide) msc4_to_bits_kernel<I, 4><<<blocks, kConvThreads, 0, s>>>(plane, bits, stride_words, (I)pairs, (I)n);
        else msc4_to_bits_kernel<I, 1><<<blocks, kConvThreads, 0, s>>>(plane, bits, stride_words, (I)pairs, (I)n);
    });
}

cudaError_t bits_to_msc4(const uint32_t *bits, uint64_t *plane, int64_t stride_words, int64_t L, int64_t rows,
                         cudaStream_t s)
{
    const int64_t pairs = L / 64, n = rows * pairs;
    return conv_launch(n, kConvThreads * kConvPairs, [&](auto index, unsigned blocks) {
        using I = decltype(index);
        bits_to_msc4_kernel<I><<<blocks, kConvThreads, 0, s>>>(bits, plane, stride_words, (I)pairs, (I)n);
    });
}

// ---------------------------------------------------------------------------
// Half-sweeps on the bit-packed planes themselves: a thread takes a 32-bit word
// of a row (32 sites, the 8 Philox blocks from 8 x its index in the plane on) and
// decides all of it with bitwise sums, about ten logic instructions per 32 sites
// where the MSC4 kernels need as many per 8, writes the word and its MSC4 form.
// One launch sweeps up to three row bands of either colour.  Bound by Philox's
// multiplies and the marks' compares: 24.6 us per 33.5 million sites, as the flat
// MSC4 kernel (25.8), which needed two conversions of 9.5 us around it here; a
// host sweep of 32768^2 in 22 bands took 1339 us with four launches per band,
// with this kernel's one 1140.  The MSC4 words come from a table of the bytes'
// half words (spread by shifts: 25.7 us, the logic pipe being the fuller one).
//
// With the planes' bits: of the up, down, centre and side neighbours d differ
// from the spin t.  For a = up ^ down ^ centre and m their majority, d is odd
// where a ^ side, and 2 or more where (m ^ t) | (a ^ t) & (side ^ t).  A spin
// flips iff d >= 2, or d = 1 and its draw is below T3, or its draw is below T4
// (T4 <= T3).
// ---------------------------------------------------------------------------
namespace {

constexpr int kBitsThreads = 512;

// Sets `bit` in g3 where u >= T3 and in g4 where u >= T4 (each bit once).
__device__ __forceinline__ void mark_planes(uint32_t &g3, uint32_t &g4, uint32_t u, uint32_t T3, uint32_t T4,
                                            uint32_t bit)
{
    asm("{\n\t"
        ".reg .pred p3, p4;\n\t"
        "setp.ge.u32 p3, %2, %4;\n\t"
        "setp.ge.u32 p4, %2, %5;\n\t"
        "@p3 add.u32 %0, %0, %3;\n\t"
        "@p4 add.u32 %1, %1, %3;\n\t"
        "}"
        : "+r"(g3), "+r"(g4)
        : "r"(u), "r"(bit), "r"(T3), "r"(T4));
}

struct BitsSplit {
    uint32_t items, per;  // words of all bands, words per block
    uint32_t upr;         // words per row
    uint32_t white;       // the white bands' first word
    uint32_t end[kMaxBitsBands];  // cumulative rows of the bands
};

// Q64: the Philox counter q = site / 4 needs 64 bits (L above 185363), and so do the
// plane's word indices from L = 524352 on; below, these stay under 2^30.
template <bool ALWAYS, bool Q64>
__global__ void __launch_bounds__(kBitsThreads, 2)
    bits_sweep_kernel(const __grid_constant__ BitsSweepParams p, const __grid_constant__ BitsSplit f)
{
    using I = typename std::conditional<Q64, uint64_t, uint32_t>::type;
    const uint32_t lo = blockIdx.x * f.per, end = min(f.items, lo + f.per), L = (uint32_t)p.L;
    uint32_t rcat = (lo + threadIdx.x) / f.upr, u = lo + threadIdx.x - rcat * f.upr;
    const uint32_t step_rows = blockDim.x / f.upr, step_u = blockDim.x - step_rows * f.upr;
    __shared__ __align__(16) char tab[1024];  // the MSC4 half word of each byte
    for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x)
        reinterpret_cast<uint32_t *>(tab)[i] = (uint32_t)bits_to_msc4_word(i);
    __syncthreads();
    uint32_t ones = 0, anti = 0;
    for (uint32_t e = lo + threadIdx.x; e < end; e += blockDim.x) {
        const int j = (int)(rcat >= f.end[0]) + (int)(rcat >= f.end[1]);
        const BitsBand &b = p.band[j];
        const uint32_t row = (uint32_t)b.row0 + rcat - (j ? f.end[j - 1] : 0u);
        const uint32_t *src = p.bits[1 - b.colour];
        const I at = (I)row * f.upr + u;
        uint32_t *tp = p.bits[b.colour] + at;
        const bool left = ((row + (uint32_t)b.colour) & 1) == 0;
        const uint32_t up = src[(I)(row == 0 ? L - 1 : row - 1) * f.upr + u];
        const uint32_t dn = src[(I)(row + 1 == L ? 0 : row + 1) * f.upr + u];
        const uint32_t cur = src[at], t = *tp;
        const uint32_t edge = src[left ? (u == 0 ? at + f.upr : at) - 1 : (u + 1 == f.upr ? at + 1 - f.upr : at + 1)];
        uint32_t ns;
        const uint32_t side = left ? __funnelshift_l(edge, cur, 1) : __funnelshift_r(cur, edge, 1);
        const uint32_t a = up ^ dn ^ cur, m = (up & dn) | (up & cur) | (dn & cur);
        if (ALWAYS) {
            ns = ~t;
        } else {
            const uint32_t c0 = 8 * (uint32_t)at, c1 = Q64 ? (uint32_t)((uint64_t)at >> 29) : 0u, c3 = p.c3 | (uint32_t)b.colour;
            uint32_t g3 = 0, g4 = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint4 r = philox(c0 | k, c1, p.c2, c3, p.rk);
                mark_planes(g3, g4, r.x, p.acc.T3, p.acc.T4, 1u << (4 * k));
                mark_planes(g3, g4, r.y, p.acc.T3, p.acc.T4, 2u << (4 * k));
                mark_planes(g3, g4, r.z, p.acc.T3, p.acc.T4, 4u << (4 * k));
                mark_planes(g3, g4, r.w, p.acc.T3, p.acc.T4, 8u << (4 * k));
            }
            const uint32_t two = (m ^ t) | ((a ^ t) & (side ^ t));
            ns = t ^ (two | ((a ^ side) & ~g3) | ~g4);
        }
        *tp = ns;
        auto spread = [&](uint32_t at4) { return *reinterpret_cast<const uint32_t *>(tab + (at4 & 0x3FCu)); };
        reinterpret_cast<uint4 *>(p.msc4[b.colour] + (int64_t)row * p.stride_words)[u] =
            make_uint4(spread(ns << 2), spread(ns >> 6), spread(ns >> 14), spread(ns >> 22));
        if (p.obs != nullptr && b.colour == 1) {
            ones += __popc(ns) + __popc(cur);
            anti += __popc(a ^ side) + 2 * (__popc(m ^ ns) + __popc((a ^ ns) & (side ^ ns)));
        }
        rcat += step_rows;
        u += step_u;
        if (u >= f.upr) {
            u -= f.upr;
            ++rcat;
        }
    }
    if (p.obs != nullptr && end > f.white) {
        // 32 white and 32 black spins and 128 bonds per white word
        const long long n = end - max(lo, f.white);
        block_count_add2(ones, anti, 2, -64 * n, -2, 128 * n, p.obs);
    }
}

template <bool ALWAYS>
cudaError_t launch_bits(const BitsSweepParams &p, const BitsSplit &f, unsigned grid, unsigned threads, cudaStream_t s)
{
    if ((uint64_t)p.L * (uint64_t)p.L / 8 > 0xFFFFFFFFull) bits_sweep_kernel<ALWAYS, true><<<grid, threads, 0, s>>>(p, f);
    else bits_sweep_kernel<ALWAYS, false><<<grid, threads, 0, s>>>(p, f);
    return cudaGetLastError();
}

}  // namespace

cudaError_t bits_half_sweeps(const BitsSweepParams &p, cudaStream_t s)
{
    DeviceInfo info;
    cudaError_t e = device_info(&info);
    if (e != cudaSuccess) return e;
    BitsSplit f;
    f.upr = (uint32_t)(p.L / 64);
    uint64_t rows = 0, black = 0;
    for (int j = 0; j < kMaxBitsBands; ++j) {
        if (j < p.n) {
            rows += (uint64_t)p.band[j].rows;
            if (p.band[j].colour == 0) black = rows;
        }
        f.end[j] = (uint32_t)rows;
    }
    if (rows * f.upr > (uint64_t)INT32_MAX) return cudaErrorInvalidConfiguration;
    f.items = (uint32_t)rows * f.upr;
    f.white = (uint32_t)black * f.upr;
    if (f.items == 0) return cudaSuccess;
    // equal ranges of words in as few equal steps as fit, as the flat MSC4 kernel
    uint32_t blocks = (uint32_t)info.sm_count;
    if (f.items > 3 * kBitsThreads * blocks) blocks *= 2;
    const uint32_t share = (f.items + blocks - 1) / blocks, steps = (share + kBitsThreads - 1) / kBitsThreads;
    const unsigned threads = ((share + steps - 1) / steps + 31) / 32 * 32;
    f.per = std::max<uint32_t>(share, 32);
    const unsigned grid = (f.items + f.per - 1) / f.per;
    return p.acc.always ? launch_bits<true>(p, f, grid, threads, s) : launch_bits<false>(p, f, grid, threads, s);
}

}  // namespace ising
