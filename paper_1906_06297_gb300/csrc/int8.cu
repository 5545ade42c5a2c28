// int8.cu -- kernels on the one-byte-per-spin lattice (Sec. 3.1 of the paper):
// two colour planes of L rows x L/2 int8 spins (+1 / -1), compacted along rows.
//
// The per-site update is the basic kernel of Fig. 2: the three vertically and
// horizontally aligned source sites (i-1, j), (i, j), (i+1, j) plus the side
// site (i, joff), where joff = j+1 for black on odd rows and white on even
// rows, j-1 otherwise (periodic), and an acceptance test equivalent to
// rand < exp(-2 beta nn s).  Here the random number is the site's keyed
// Philox draw and the test is the exact integer form u < T[a].
//
// A thread owns one Philox block (4 consecutive sites of the plane in row-major
// order, which may straddle a row end when L/2 is not a multiple of 4) or a run of
// sites of one row.  int8_words_kernel takes planes whose rows are whole aligned
// 16-byte groups, int8_rows_kernel the other ones, and int8_sweep_kernel what
// their 32-bit indices do not reach.
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "launch.h"
#include "sweep_core.cuh"

namespace ising {

namespace {

constexpr int kThreads = 256;
// Flat kernels: blocks of up to 512 threads at 64 registers, one per SM (so that a
// block of the next kernel fits beside it), or two from four steps per block on.
constexpr int kFlatThreads = 512;

// ---------------------------------------------------------------------------
// Four spins at once, one per byte of a 32-bit word (+1 = 0x01, -1 = 0xFF): bits 1
// to 7 of a byte all say "down", so any of them can hold a plane of a bitwise sum.
// With a = up ^ down ^ centre and m their majority, the number d of neighbours that
// differ from the spin t is odd where a ^ side, and 2 or more where (m ^ t) |
// (a ^ t) & (side ^ t).  A spin flips iff d >= 2, or d = 1 and its draw is below T3, or
// its draw is below T4 (T4 <= T3); the draws' marks have bit 6 of a byte set where
// u >= T3, bit 7 where u >= T4.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t byte_signs(uint32_t x)  // 0xFF where the byte's top bit is set
{
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, 0xBA98;" : "=r"(r) : "r"(x));
    return r;
}

__device__ __forceinline__ void mark_byte(uint32_t &g, uint32_t u, uint32_t T3, uint32_t T4, uint32_t bit6, uint32_t bit7)
{
    asm("{\n\t"
        ".reg .pred p3, p4;\n\t"
        "setp.ge.u32 p3, %1, %3;\n\t"
        "setp.ge.u32 p4, %1, %4;\n\t"
        "@p3 add.u32 %0, %0, %2;\n\t"
        "@p4 add.u32 %0, %0, %5;\n\t"
        "}"
        : "+r"(g)
        : "r"(u), "r"(bit6), "r"(T3), "r"(T4), "r"(bit7));
}

__device__ __forceinline__ uint32_t block_marks(uint32_t q, const DrawCtx &dc, const RoundKeys &rk)
{
    const uint4 u = philox(q, 0u, dc.c2, dc.c3, rk);
    uint32_t g = 0;
    mark_byte(g, u.x, dc.T3, dc.T4, 1u << 6, 1u << 7);
    mark_byte(g, u.y, dc.T3, dc.T4, 1u << 14, 1u << 15);
    mark_byte(g, u.z, dc.T3, dc.T4, 1u << 22, 1u << 23);
    mark_byte(g, u.w, dc.T3, dc.T4, 1u << 30, 1u << 31);
    return g;
}

__device__ __forceinline__ uint32_t majority(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (a & c) | (b & c); }

// Adds the down spins among t and the centres to `down` and t's differing
// neighbours to `anti`, over the bytes of mask `in`: d is the plane a ^ side plus
// twice two others, so one count of bits takes them all from bits of their own.
__device__ __forceinline__ void count_bytes(uint32_t t, uint32_t a, uint32_t m, uint32_t cur, uint32_t side, uint32_t in,
                                            uint32_t &down, uint32_t &anti)
{
    const uint32_t two = (a ^ t) & (side ^ t);
    const uint32_t d = ((a ^ side) & 0x02020202u) | ((m ^ t) & 0x0C0C0C0Cu) | (two & 0x30303030u);
    const uint32_t n = (t & 0x02020202u) | (cur & 0x04040404u);
    anti += __popc(d & in);
    down += __popc(n & in);
}

// New values of the four spins t; with OBS, counts them over the bytes of mask `in`.
template <bool OBS, bool ALWAYS>
__device__ __forceinline__ uint32_t decide_bytes(uint32_t t, uint32_t up, uint32_t cur, uint32_t dn, uint32_t side,
                                                 uint32_t g, uint32_t in, uint32_t &down, uint32_t &anti)
{
    const uint32_t a = up ^ dn ^ cur, m = majority(up, dn, cur);
    uint32_t nt;
    if (ALWAYS) {
        nt = t ^ 0xFEFEFEFEu;
    } else {
        const uint32_t two = (m ^ t) | ((a ^ t) & (side ^ t)), one = ((a ^ side) & ~g) << 1;
        nt = t ^ (byte_signs(two | one | ~g) & 0xFEFEFEFEu);
    }
    if (OBS) count_bytes(nt, a, m, cur, side, in, down, anti);
    return nt;
}

struct FlatSplit {
    uint32_t items, per;  // items of the plane, items per block
    uint32_t upr;         // units per row (words kernel)
    int32_t colour;
};

// Planes whose rows are whole 16-byte groups (L/2, the row stride and the plane
// addresses multiples of 16).  Bound by Philox's multiplies
// as the multi-spin-coded kernel is; the byte-wise arithmetic takes about twice
// its logic instructions per spin.  Launched as msc4_flat_kernel is (one block
// per SM, marks before the wait for the kernel before it).  2560^2, us per
// sweep: thread per Philox block with 64-bit site indices and byte accesses
// 36.9, this kernel with sums of two-bit fields and a compare per byte 8.55, with the
// bitwise planes 8.3 (9.0 with the observables either way).
template <bool OBS, bool ALWAYS>
__global__ void __launch_bounds__(kFlatThreads, 2)
    int8_words_kernel(const __grid_constant__ Int8SweepParams p, const __grid_constant__ FlatSplit f)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t end = min(f.items, (blockIdx.x + 1) * f.per);
    const DrawCtx dc{p.c2, p.c3, p.acc.T3, p.acc.T4, p.acc.zero};
    constexpr int WORDS = 4;
    const uint32_t L = (uint32_t)p.L;
    uint32_t down = 0, anti = 0;
    bool waited = false;
    for (uint32_t e = blockIdx.x * f.per + threadIdx.x; e < end; e += blockDim.x) {
        const uint32_t row = e / f.upr, u = e - row * f.upr;
        uint32_t g[WORDS];
#pragma unroll
        for (int h = 0; h < WORDS; ++h) g[h] = ALWAYS ? 0u : block_marks(WORDS * e + h, dc, p.rk);
        if (!waited) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            waited = true;
        }
        const uint32_t ru = row == 0 ? L - 1 : row - 1, rd = row + 1 == L ? 0 : row + 1;
        const int8_t *col = p.src + 4 * WORDS * u;
        const uint32_t *crow = reinterpret_cast<const uint32_t *>(col + row * p.stride);
        const uint32_t *urow = reinterpret_cast<const uint32_t *>(col + ru * p.stride);
        const uint32_t *drow = reinterpret_cast<const uint32_t *>(col + rd * p.stride);
        uint32_t *tp = reinterpret_cast<uint32_t *>(p.tgt + row * p.stride + 4 * WORDS * u);
        const bool left = ((row + f.colour) & 1) == 0;
        const int32_t last = (int32_t)f.upr - 1;
        const int32_t off = left ? (u == 0 ? WORDS * last + WORDS - 1 : -1)
                                 : ((int32_t)u == last ? -WORDS * last : WORDS);
        const uint4 a = *reinterpret_cast<const uint4 *>(urow), b = *reinterpret_cast<const uint4 *>(crow),
                    c = *reinterpret_cast<const uint4 *>(drow), d = *reinterpret_cast<const uint4 *>(tp);
        const uint32_t up[WORDS] = {a.x, a.y, a.z, a.w}, cur[WORDS] = {b.x, b.y, b.z, b.w},
                       dn[WORDS] = {c.x, c.y, c.z, c.w};
        uint32_t tg[WORDS] = {d.x, d.y, d.z, d.w};
        const uint32_t edge = crow[off];
#pragma unroll
        for (int h = 0; h < WORDS; ++h) {
            const uint32_t prev = h == 0 ? edge : cur[h - 1], next = h == WORDS - 1 ? edge : cur[h + 1];
            const uint32_t side = left ? __funnelshift_l(prev, cur[h], 8) : __funnelshift_r(cur[h], next, 8);
            tg[h] = decide_bytes<OBS, ALWAYS>(tg[h], up[h], cur[h], dn[h], side, g[h], 0xFFFFFFFFu, down, anti);
        }
        *reinterpret_cast<uint4 *>(tp) = make_uint4(tg[0], tg[1], tg[2], tg[3]);
    }
    if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (OBS) {
        // n white and n black spins, 4 n bonds
        const long long n = 16 * (long long)(end - blockIdx.x * f.per);
        block_count_add2(down, anti, -2, 2 * n, -2, 4 * n, p.obs);
    }
}

// The 4 WORDS bytes from p on, of which the first nv are asked for, from the
// aligned words that hold any of those (so nothing outside the row's own words
// is read); the other bytes of x are arbitrary.
template <int WORDS>
__device__ __forceinline__ void ld_bytes(const int8_t *p, uint32_t nv, uint32_t (&x)[WORDS])
{
    const uint32_t a = (uint32_t)(uintptr_t)p & 3u;
    const uint32_t *w = reinterpret_cast<const uint32_t *>(p - a);
    uint32_t v[WORDS + 1];
#pragma unroll
    for (int h = 0; h <= WORDS; ++h) v[h] = 4 * h < nv + a ? w[h] : 0u;
#pragma unroll
    for (int h = 0; h < WORDS; ++h) x[h] = __funnelshift_r(v[h], v[h + 1], 8 * a);
}

// Mask of the bytes of word h of a unit of nv sites that hold one of them.
__device__ __forceinline__ uint32_t bytes_in(uint32_t h, uint32_t nv)
{
    return 4 * h + 4 <= nv ? 0xFFFFFFFFu : (4 * h >= nv ? 0u : (1u << (8 * (nv & 3))) - 1u);
}

// The side neighbours of word h of a unit of nv centres: the bytes before them, or
// after them, where `edge` is the one before the first or after the last.
template <int WORDS>
__device__ __forceinline__ uint32_t row_side(const uint32_t (&cur)[WORDS], uint32_t edge, bool left, int h, uint32_t nv)
{
    const uint32_t prev = h == 0 ? edge << 24 : cur[h > 0 ? h - 1 : 0];
    uint32_t c = cur[h], next = h + 1 < WORDS ? cur[h + 1 < WORDS ? h + 1 : h] : edge;
    if ((nv >> 2) == (uint32_t)h) c = (c & ~(0xFFu << (8 * (nv & 3)))) | (edge << (8 * (nv & 3)));
    if ((nv >> 2) == (uint32_t)h + 1 && (nv & 3) == 0) next = edge;
    return left ? __funnelshift_l(prev, cur[h], 8) : __funnelshift_r(c, next, 8);
}

// Any other plane with fewer than 2^32 sites: a thread takes up to 4 WORDS
// consecutive sites of one row, at any byte offset.  Their draws start in the
// middle of a Philox block when row x L/2 is not a multiple of 4: one block
// more, and the marks are shifted by whole bytes as the spins are.  Only the
// bytes at the two ends that fill no aligned word are stored singly.  2562^2
// (L/2 = 1281), us per sweep: general kernel 37.3, a Philox block per thread
// with its sites' bytes 24.2, this kernel 15.9; 8194^2 305 and 117.
template <bool OBS, bool ALWAYS, int WORDS>
__global__ void __launch_bounds__(kFlatThreads, 2)
    int8_rows_kernel(const __grid_constant__ Int8SweepParams p, const __grid_constant__ FlatSplit f)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t end = min(f.items, (blockIdx.x + 1) * f.per);
    const DrawCtx dc{p.c2, p.c3, p.acc.T3, p.acc.T4, p.acc.zero};
    const uint32_t L = (uint32_t)p.L, half = (uint32_t)p.half;
    uint32_t down = 0, anti = 0;
    bool waited = false;
    for (uint32_t e = blockIdx.x * f.per + threadIdx.x; e < end; e += blockDim.x) {
        const uint32_t row = e / f.upr, j = 4 * WORDS * (e - row * f.upr);
        const uint32_t nv = min(4u * WORDS, half - j), site = row * half + j, o = site & 3u;
        uint32_t g[WORDS + 1];
#pragma unroll
        for (int h = 0; h < WORDS; ++h) g[h] = ALWAYS ? 0u : block_marks((site >> 2) + h, dc, p.rk);
        g[WORDS] = 0;
        if (!ALWAYS && o != 0) g[WORDS] = block_marks((site >> 2) + WORDS, dc, p.rk);
        if (!waited) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            waited = true;
        }
        const uint32_t ru = row == 0 ? L - 1 : row - 1, rd = row + 1 == L ? 0 : row + 1;
        const int8_t *srow = p.src + row * p.stride;
        int8_t *tp = p.tgt + row * p.stride + j;
        const bool left = ((row + f.colour) & 1) == 0;
        uint32_t up[WORDS], cur[WORDS], dn[WORDS], tg[WORDS];
        ld_bytes<WORDS>(p.src + ru * p.stride + j, nv, up);
        ld_bytes<WORDS>(srow + j, nv, cur);
        ld_bytes<WORDS>(p.src + rd * p.stride + j, nv, dn);
        ld_bytes<WORDS>(tp, nv, tg);
        const uint32_t edge = (uint8_t)srow[left ? (j == 0 ? half : j) - 1 : (j + nv == half ? 0 : j + nv)];
#pragma unroll
        for (int h = 0; h < WORDS; ++h) {
            const uint32_t side = row_side<WORDS>(cur, edge, left, h, nv), m = bytes_in(h, nv);
            tg[h] = decide_bytes<OBS, ALWAYS>(tg[h], up[h], cur[h], dn[h], side, __funnelshift_r(g[h], g[h + 1], 8 * o), m,
                                              down, anti);
        }
        const uint32_t a = (uint32_t)(uintptr_t)tp & 3u;
        uint32_t *tw = reinterpret_cast<uint32_t *>(tp - a);
#pragma unroll
        for (int h = 0; h <= WORDS; ++h) {
            // bytes 4 h - a .. 4 h - a + 3 of the unit
            const uint32_t w = __funnelshift_l(h > 0 ? tg[h > 0 ? h - 1 : 0] : 0u, h < WORDS ? tg[h < WORDS ? h : 0] : 0u, 8 * a);
            if (4 * h >= a && 4 * h + 4 <= nv + a) {
                tw[h] = w;
            } else if (4 * h < nv + a) {
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k)
                    if (4 * h + k >= a && 4 * h + k < nv + a) tp[(int)(4 * h + k) - (int)a] = (int8_t)(w >> (8 * k));
            }
        }
    }
    if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (OBS) {
        // the sites of units [lo, end): whole rows of L / 2 and what is left of the last
        auto sites = [&](uint32_t e) { return (long long)(e / f.upr) * half + min(4u * WORDS * (e % f.upr), half); };
        const long long n = sites(end) - sites(blockIdx.x * f.per);
        block_count_add2(down, anti, -2, 2 * n, -2, 4 * n, p.obs);
    }
}

// One block per SM over equal ranges of `items`, which may start beside the
// kernel before it in the stream (it waits for it itself).
template <typename K>
cudaError_t launch_flat(K kernel, const Int8SweepParams &p, int colour, uint32_t items, uint32_t upr, cudaStream_t s)
{
    DeviceInfo info;
    cudaError_t e = device_info(&info);
    if (e != cudaSuccess) return e;
    uint32_t blocks = (uint32_t)info.sm_count;
    if (items > 3 * kFlatThreads * blocks) blocks *= 2;  // see kFlatThreads
    const uint32_t share = (items + blocks - 1) / blocks, steps = (share + kFlatThreads - 1) / kFlatThreads;
    FlatSplit f;
    f.items = items;
    f.per = std::max<uint32_t>(share, 32);
    f.upr = upr;
    f.colour = colour;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((items + f.per - 1) / f.per);
    cfg.blockDim = dim3(((share + steps - 1) / steps + 31) / 32 * 32);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, p, f);
}

// The kernel for a plane, by L/2 and the alignment of its rows; units of one
// word while one per thread fits (770^2: 4.3 us per sweep against 4.8 with four
// words, 1026^2, two steps of one word: 6.0 against 4.4).
template <bool OBS, bool ALWAYS>
cudaError_t launch_small_index(const Int8SweepParams &p, int colour, cudaStream_t s)
{
    const uint64_t align = (uint64_t)p.half | (uint64_t)p.stride | (uintptr_t)p.src | (uintptr_t)p.tgt;
    if (align % 16 == 0)
        return launch_flat(int8_words_kernel<OBS, ALWAYS>, p, colour, (uint32_t)(p.nblk / 4), (uint32_t)(p.half / 16), s);
    DeviceInfo info;
    cudaError_t e = device_info(&info);
    if (e != cudaSuccess) return e;
    const uint32_t u1 = (uint32_t)((p.half + 3) / 4), u4 = (uint32_t)((p.half + 15) / 16);
    if (p.L * u1 <= kFlatThreads * info.sm_count)
        return launch_flat(int8_rows_kernel<OBS, ALWAYS, 1>, p, colour, (uint32_t)p.L * u1, u1, s);
    return launch_flat(int8_rows_kernel<OBS, ALWAYS, 4>, p, colour, (uint32_t)p.L * u4, u4, s);
}

// The general form: 64-bit indices, any L.
template <int COLOR, bool OBS>
__global__ void __launch_bounds__(kThreads) int8_sweep_kernel(const __grid_constant__ Int8SweepParams p)
{
    const int64_t nsites = p.L * p.half;
    long long sum_s = 0, sum_b = 0;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < p.nblk;
         q += (int64_t)gridDim.x * blockDim.x) {
        const uint4 u4 = philox((uint32_t)q, (uint32_t)((uint64_t)q >> 32), p.c2, p.c3, p.rk);
        const uint32_t us[4] = {u4.x, u4.y, u4.z, u4.w};
        const int64_t site0 = 4 * q;
        int64_t i = site0 / p.half;
        int64_t j = site0 - i * p.half;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (site0 + k < nsites) {
                const int64_t iu = i == 0 ? p.L - 1 : i - 1;
                const int64_t id = i + 1 == p.L ? 0 : i + 1;
                const int64_t jl = j == 0 ? p.half - 1 : j - 1;
                const int64_t jr = j + 1 == p.half ? 0 : j + 1;
                const bool odd = (i & 1) != 0;
                const int64_t joff = (COLOR == 0) ? (odd ? jr : jl) : (odd ? jl : jr);
                const int8_t *srow = p.src + i * p.stride;
                const int centre = srow[j];
                const int nn = p.src[iu * p.stride + j] + p.src[id * p.stride + j] + centre + srow[joff];
                int8_t *tp = p.tgt + i * p.stride + j;
                const int s = *tp;
                const int a = (4 + s * nn) >> 1;  // aligned neighbours
                const uint64_t u = us[k];
                const bool flip = a <= 2 || (a == 3 ? u < p.acc.T3_64 : u < p.acc.T4_64);
                const int ns = flip ? -s : s;
                if (flip) *tp = (int8_t)ns;
                if (OBS) {
                    sum_s += ns + centre;
                    sum_b += ns * nn;
                }
            }
            if (++j == p.half) {
                j = 0;
                ++i;
            }
        }
    }
    if (OBS) block_reduce_add2<kThreads>(sum_s, sum_b, p.obs);
}

__global__ void int8_init_kernel(int8_t *plane, int64_t L, int64_t stride, int mode, uint32_t c3,
                                 const __grid_constant__ RoundKeys rk)
{
    const int64_t half = L / 2, nsites = L * half, nblk = (nsites + 3) / 4;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nblk;
         q += (int64_t)gridDim.x * blockDim.x) {
        uint32_t us[4] = {0, 0, 0, 0};
        if (mode == 0) {
            const uint4 u4 = philox((uint32_t)q, (uint32_t)((uint64_t)q >> 32), 0u, c3, rk);
            us[0] = u4.x; us[1] = u4.y; us[2] = u4.z; us[3] = u4.w;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t site = 4 * q + k;
            if (site < nsites) {
                const int64_t i = site / half, j = site - i * half;
                int8_t v = mode == 1 ? 1 : (mode == 2 ? -1 : (us[k] < 0x80000000u ? 1 : -1));
                plane[i * stride + j] = v;
            }
        }
    }
}

// Observables without an update: each white site's s (sum of its 4 black
// neighbours) visits every bond once, s_w + s_b every site once.  A thread takes
// up to 16 sites of a row, as int8_rows_kernel does; WIDE: its rows are whole
// aligned 16-byte groups.  16384^2: thread per site 649 us, here 97, WIDE 51.6
// (5.2 TB/s).
template <typename I, bool WIDE>
__global__ void __launch_bounds__(256) int8_obs_kernel(const int8_t *__restrict__ black,
                                                       const int8_t *__restrict__ white, int64_t L, int64_t stride,
                                                       long long *out)
{
    const uint32_t half = (uint32_t)(L / 2);
    const I upr = (I)((half + 15) / 16), items = (I)L * upr, step = (I)gridDim.x * 256;
    long long n = 0, down_sum = 0, anti_sum = 0;
    for (I e = (I)blockIdx.x * 256 + threadIdx.x; e < items; e += step) {
        const I row = e / upr;
        const uint32_t j = 16 * (uint32_t)(e - row * upr), nv = WIDE ? 16u : min(16u, half - j);
        const I ru = row == 0 ? (I)L - 1 : row - 1, rd = row + 1 == (I)L ? 0 : row + 1;
        const int8_t *srow = black + (int64_t)row * stride;
        const bool left = (row & 1) != 0;
        uint32_t up[4], cur[4], dn[4], t[4];
        auto load = [&](const int8_t *p, uint32_t (&x)[4]) {
            if constexpr (WIDE) {
                const uint4 v = *reinterpret_cast<const uint4 *>(p);
                x[0] = v.x, x[1] = v.y, x[2] = v.z, x[3] = v.w;
            } else {
                ld_bytes<4>(p, nv, x);
            }
        };
        load(black + (int64_t)ru * stride + j, up);
        load(srow + j, cur);
        load(black + (int64_t)rd * stride + j, dn);
        load(white + (int64_t)row * stride + j, t);
        const uint32_t edge = (uint8_t)srow[left ? (j == 0 ? half : j) - 1 : (j + nv == half ? 0 : j + nv)];
        uint32_t down = 0, anti = 0;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const uint32_t m = bytes_in(h, nv);
            const uint32_t side = row_side<4>(cur, edge, left, h, nv);
            count_bytes(t[h], up[h] ^ dn[h] ^ cur[h], majority(up[h], dn[h], cur[h]), cur[h], side, m, down, anti);
        }
        n += nv;
        down_sum += down;
        anti_sum += anti;
    }
    block_reduce_add2<256>(2 * n - 2 * down_sum, 4 * n - 2 * anti_sum, out);
}

unsigned grid_for(int64_t n, int threads, int per_sm)
{
    DeviceInfo info{1};
    device_info(&info);
    const int64_t cap = (int64_t)info.sm_count * per_sm;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(cap, (n + threads - 1) / threads));
}

}  // namespace

cudaError_t int8_half_sweep(const Int8SweepParams &p, int colour, cudaStream_t s)
{
    const unsigned g = grid_for(p.nblk, kThreads, 8);
    const bool obs = p.obs != nullptr;
    if (p.L * p.half < (int64_t(1) << 32)) {  // 32-bit site indices
        if (p.acc.always) return obs ? launch_small_index<true, true>(p, colour, s) : launch_small_index<false, true>(p, colour, s);
        return obs ? launch_small_index<true, false>(p, colour, s) : launch_small_index<false, false>(p, colour, s);
    }
    if (colour == 0) {
        if (obs) int8_sweep_kernel<0, true><<<g, kThreads, 0, s>>>(p);
        else int8_sweep_kernel<0, false><<<g, kThreads, 0, s>>>(p);
    } else {
        if (obs) int8_sweep_kernel<1, true><<<g, kThreads, 0, s>>>(p);
        else int8_sweep_kernel<1, false><<<g, kThreads, 0, s>>>(p);
    }
    return cudaGetLastError();
}

cudaError_t int8_init(int8_t *plane, int colour, int64_t L, int64_t stride, int mode, uint64_t seed,
                      cudaStream_t s)
{
    const RoundKeys rk = make_round_keys(seed);
    const int64_t nblk = (L * (L / 2) + 3) / 4;
    int8_init_kernel<<<grid_for(nblk, 256, 8), 256, 0, s>>>(plane, L, stride, mode,
                                                            counter_word3(colour, kPurposeInit, 0), rk);
    return cudaGetLastError();
}

cudaError_t int8_observables(const int8_t *black, const int8_t *white, int64_t L, int64_t stride, long long *out,
                             cudaStream_t s)
{
    const int64_t items = L * ((L / 2 + 15) / 16);
    const unsigned g = grid_for(items, 256, 8);
    const bool wide = ((uint64_t)(L / 2) | (uint64_t)stride | (uintptr_t)black | (uintptr_t)white) % 16 == 0;
    auto go = [&](auto kernel) { kernel<<<g, 256, 0, s>>>(black, white, L, stride, out); };
    if (items < (int64_t(1) << 31)) wide ? go(int8_obs_kernel<uint32_t, true>) : go(int8_obs_kernel<uint32_t, false>);
    else wide ? go(int8_obs_kernel<uint64_t, true>) : go(int8_obs_kernel<uint64_t, false>);
    return cudaGetLastError();
}

}  // namespace ising
