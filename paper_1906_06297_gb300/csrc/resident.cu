// resident.cu -- whole sweep calls of small lattices in one launch of one
// thread-block cluster.
//
// A half-sweep of a small lattice is too little work for a launch: at 256^2 the
// multiplies of its draws take the whole chip 17 ns, while two launches per
// sweep cost 3.6 us of host time alone.  Here up to 16 CTAs of one cluster hold
// the lattice in shared memory for all sweeps of the call, a band of rows each,
// and meet at the cluster's hardware barrier after every half-sweep.  256^2,
// 1000 recorded sweeps: 8.2 us per sweep with two launches of a thread per Philox
// block, 3.55 with two overlapped flat launches, 1.15 here.  Of ~860 cycles per
// half-sweep then ~500 are the marks (a chain of ten Philox rounds that two
// warps per scheduler do not hide), ~200 the decision and its shared-memory
// reads, ~100 the rest of the barrier.
//
// Both layouts are held the same way: 8 spins of a row to a 32-bit half word,
// one per nibble (0/1), ceil(L/2 / 8) half words per row and colour.  A thread
// owns up to K half words of each colour for the whole call.  Per half-sweep it
// forms their draws' marks, then waits for the other CTAs' last half-sweep,
// then decides; so the barrier's latency passes behind the generator, which is
// nearly all of the arithmetic.  The first and last row of a band are also
// copied into the halo rows of the CTAs above and below (distributed shared
// memory), so every read after the wait is local.  A neighbour's halo row of one
// colour is only written after that neighbour has passed the barrier behind its
// last reads of it, one half-sweep of the other colour earlier.
//
// RAGGED: rows of one-byte lattices with L/2 not a multiple of 8.  The last half
// word of a row holds fewer spins (its other nibbles stay 0) and a half word's
// draws may start in the middle of a Philox block.
//
// One warp of each CTA computes nothing: behind the CTA's own barrier it copies
// the band's first and last rows into the neighbours and alone makes the
// cluster-wide release.  (A release by every thread costs each half-sweep ~280
// cycles of fence on top of the ~100 of the hardware barrier, which the marks,
// ~500 cycles, then no longer hide.  64-bit shared atomics for the sums cost another
// 600 per sweep; each warp has a word of its own instead.)
//
// The observables of each sweep are added up in the CTAs' shared memory and
// written by the first CTA every kTraceRows sweeps.
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "launch.h"
#include "sweep_core.cuh"

namespace ising {

namespace {

constexpr int kMaxThreads = 1024;
constexpr int kMaxCluster = 16;
constexpr int kTraceRows = 128;
// Half words per CTA and colour below which the cluster is not doubled: 64^2 takes
// 0.95 us per sweep with at least 64, 0.99 with 128 and 1.12 with 256.
constexpr int64_t kItems = 64;
// Sweeps per launch (some 10 ms): another stream's work is not kept waiting for
// the whole of a long call.
constexpr int64_t kMaxSweeps = 16384;

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_relaxed()
{
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// The address of this CTA's shared-memory address `a` in CTA `rank`.
__device__ __forceinline__ uint32_t peer_addr(uint32_t a, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

__device__ __forceinline__ void peer_store(uint32_t a, uint32_t v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned long long peer_load(uint32_t a)
{
    unsigned long long v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}

// Half word u of one plane row, and back (one-byte rows: nv spins of it).
__device__ __forceinline__ uint32_t load_half(const ResidentSweep &p, int colour, int row, int u, int nv)
{
    const char *r = static_cast<const char *>(p.plane[colour]) + row * p.stride;
    if (!p.bytes) return reinterpret_cast<const uint32_t *>(r)[u];
    uint32_t x = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (k < nv) x |= (uint32_t)(reinterpret_cast<const int8_t *>(r)[8 * u + k] > 0) << (4 * k);
    return x;
}

__device__ __forceinline__ void store_half(const ResidentSweep &p, int colour, int row, int u, int nv, uint32_t x)
{
    char *r = static_cast<char *>(p.plane[colour]) + row * p.stride;
    if (!p.bytes) {
        reinterpret_cast<uint32_t *>(r)[u] = x;
        return;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (k < nv) reinterpret_cast<int8_t *>(r)[8 * u + k] = ((x >> (4 * k)) & 1u) ? 1 : -1;
}

// The marks of half_marks for 8 draws that start at draw o of block b, one
// counter per block (half_marks' single one is a chain of 16 dependent adds).
template <bool RAGGED>
__device__ __forceinline__ uint32_t marks8(uint32_t b, uint32_t o, const DrawCtx &dc, const RoundKeys &rk)
{
    uint32_t m[3] = {0, 0, 0}, unused = 0;
#pragma unroll
    for (int i = 0; i < (RAGGED ? 3 : 2); ++i) {
        if (i == 2 && o == 0) break;
        const uint4 u = philox(b + i, 0u, dc.c2, dc.c3, rk);
        mark_ge(m[i], unused, u.x, dc.T3, dc.T4, 1u);
        mark_ge(m[i], unused, u.y, dc.T3, dc.T4, 1u << 4);
        mark_ge(m[i], unused, u.z, dc.T3, dc.T4, 1u << 8);
        mark_ge(m[i], unused, u.w, dc.T3, dc.T4, 1u << 12);
    }
    const uint32_t lo = m[0] | (m[1] << 16);
    return RAGGED ? __funnelshift_r(lo, m[2], 4 * o) : lo;
}

template <int K, bool RAGGED>
__global__ void __launch_bounds__(kMaxThreads, 1) resident_kernel(const __grid_constant__ ResidentSweep p)
{
    extern __shared__ __align__(16) uint32_t res_smem[];
    const int L = p.L, hpr = p.hpr, half = L / 2, tid = threadIdx.x, lane = tid & 31;
    const int nc = (int)blockDim.x - 32;  // threads that compute; the last warp exchanges the halo rows
    const bool halo = tid >= nc;
    const int cs = (int)gridDim.x, rank = (int)cluster_rank();
    const int r0 = rank * L / cs, rows = (rank + 1) * L / cs - r0;
    const int plane_words = ((L + cs - 1) / cs + 2) * hpr;
    // each traced sweep's sums [kTraceRows] (up spins in the high half, anti-
    // aligned pairs in the low half), the same per warp (16 bits each), then the
    // black and the white plane: local rows 0 (halo above), 1 .. rows, rows + 1
    // (halo below)
    const int nw = nc >> 5;
    unsigned long long *tr = reinterpret_cast<unsigned long long *>(res_smem);
    uint32_t *tw = res_smem + 2 * kTraceRows;
    uint32_t *pl = tw + kTraceRows * nw;
    const int last_nv = half - 8 * (hpr - 1);  // spins of a row's last half word

    for (int i = tid; i < (rows + 2) * hpr; i += blockDim.x) {
        const int lr = i / hpr, u = i - lr * hpr;
        int row = r0 - 1 + lr;
        row = row < 0 ? row + L : (row >= L ? row - L : row);
        const int nv = u == hpr - 1 ? last_nv : 8;
#pragma unroll
        for (int c = 0; c < 2; ++c) pl[c * plane_words + i] = load_half(p, c, row, u, nv);
    }
    // this thread's half words: local index and first draw
    int at[K], u[K];
    bool odd[K];  // parity of the lattice row
    uint32_t blk[K], off[K];
    const int items = rows * hpr;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int it = tid + k * nc;
        const int row = it / hpr;
        u[k] = it - row * hpr;
        at[k] = it < items && !halo ? it + hpr : -1;
        odd[k] = ((r0 + row) & 1) != 0;
        const uint32_t site = (uint32_t)(r0 + row) * (uint32_t)half + 8u * (uint32_t)u[k];
        blk[k] = site >> 2;
        off[k] = site & 3u;
    }
    // where the halo rows of the CTAs above (its row below) and below (its row above) are
    const uint32_t pl_u32 = (uint32_t)__cvta_generic_to_shared(pl);
    const int above = rank == 0 ? cs - 1 : rank - 1, below = rank + 1 == cs ? 0 : rank + 1;
    const int rows_above = (above + 1) * L / cs - above * L / cs;
    const uint32_t to_above = peer_addr(pl_u32 + 4u * (uint32_t)((rows_above + 1) * hpr), (uint32_t)above);
    const uint32_t to_below = peer_addr(pl_u32, (uint32_t)below);
    const uint32_t last_mask = last_nv == 8 ? 0xFFFFFFFFu : (1u << (4 * last_nv)) - 1u;
    const bool always = p.acc.always != 0;
    cluster_arrive();

    int traced = 0;  // sweeps summed in tr
    for (int s = 0; s < p.n_sweeps; ++s) {
        const uint64_t t = p.t0 + (uint64_t)s;
#pragma unroll 1
        for (int colour = 0; colour < 2; ++colour) {
            const DrawCtx dc{(uint32_t)t, counter_word3(colour, kPurposeMetropolis, t), p.acc.T3, p.acc.T4, p.acc.zero};
            uint32_t *tgt = pl + colour * plane_words;
            const uint32_t *src = pl + (1 - colour) * plane_words;
            if (halo) {
                cluster_wait();
                __syncthreads();  // the colour is updated
                const uint32_t o = 4u * (uint32_t)(colour * plane_words);
                for (int i = lane; i < hpr; i += 32) {
                    peer_store(to_above + o + 4u * i, tgt[hpr + i]);
                    peer_store(to_below + o + 4u * i, tgt[rows * hpr + i]);
                }
                cluster_arrive();
                continue;
            }
            uint32_t g[K];
#pragma unroll
            for (int k = 0; k < K; ++k) g[k] = at[k] >= 0 && !always ? marks8<RAGGED>(blk[k], off[k], dc, p.rk) : 0u;
            uint32_t sums = 0;
            cluster_wait();
#pragma unroll
            for (int k = 0; k < K; ++k) {
                if (at[k] < 0) continue;
                const int i = at[k];
                const uint32_t cur = src[i], tg = tgt[i];
                const bool left = odd[k] == (colour == 1), last = u[k] == hpr - 1;
                uint32_t side;
                if (left) {
                    uint32_t prev = src[u[k] == 0 ? i + hpr - 1 : i - 1];
                    if (RAGGED && u[k] == 0) prev <<= 4 * (8 - last_nv);
                    side = __funnelshift_l(prev, cur, 4);
                } else {
                    const uint32_t next = src[last ? i - u[k] : i + 1];
                    if (RAGGED && last && last_nv < 8)
                        side = (cur | (next << (4 * last_nv))) >> 4;
                    else
                        side = __funnelshift_r(cur, next, 4);
                }
                const uint32_t e = src[i - hpr] + src[i + hpr] + cur;
                const uint32_t a8 = e + side + 0x88888888u, b8 = 0xCCCCCCCCu - e - side;
                uint32_t none = 0;
                uint32_t nt = always ? tg ^ kNibbleLsb : decide_sums<false, false>(tg, a8, b8, g[k], none);
                if (RAGGED && last) nt &= last_mask;
                tgt[i] = nt;
                if (colour == 1 && p.trace != nullptr) {
                    const uint32_t m = nt * 15u;
                    uint32_t d2 = ((a8 & ~m) | (b8 & m)) & 0x77777777u;  // anti-aligned neighbours
                    if (RAGGED && last) d2 &= last_mask;
                    const uint32_t by = (d2 & 0x0F0F0F0Fu) + (d2 >> 4 & 0x0F0F0F0Fu);
                    sums += ((by * 0x01010101u) >> 24) | ((uint32_t)(__popc(nt) + __popc(cur)) << 16);
                }
            }
            __syncthreads();
            cluster_arrive_relaxed();
            if (colour == 1 && p.trace != nullptr) {
                // at most 32 K of each per lane: both sums of a warp fit 16 bits
                sums = __reduce_add_sync(0xffffffffu, sums);
                if (lane == 0) tw[traced * nw + (tid >> 5)] = sums;
            }
        }
        if (p.trace != nullptr && (++traced == kTraceRows || s + 1 == p.n_sweeps)) {
            // every CTA adds up its warps; behind one more barrier the first CTA
            // adds up the CTAs, and behind another the sums may be written again
            cluster_wait();
            __syncthreads();
            for (int i = tid; i < traced; i += blockDim.x) {
                unsigned long long v = 0;
                for (int w = 0; w < nw; ++w) {
                    const uint32_t x = tw[i * nw + w];
                    v += ((unsigned long long)(x >> 16) << 32) | (x & 0xFFFFu);
                }
                tr[i] = v;
            }
            cluster_arrive();
            cluster_wait();
            if (rank == 0) {
                const uint32_t tr_u32 = (uint32_t)__cvta_generic_to_shared(tr);
                const long long area = (long long)L * L;
                for (int i = tid; i < traced; i += blockDim.x) {
                    long long ones = 0, anti = 0;
                    for (int c = 0; c < cs; ++c) {
                        const unsigned long long v = peer_load(peer_addr(tr_u32 + 8u * (uint32_t)i, (uint32_t)c));
                        ones += (long long)(v >> 32);
                        anti += (long long)(v & 0xFFFFFFFFull);
                    }
                    // L^2 / 2 white spins with 4 bonds each, as many black ones
                    long long *row = p.trace + 2 * (int64_t)(s + 1 - traced + i);
                    row[0] = 2 * ones - area;
                    row[1] = 2 * area - 2 * anti;
                }
            }
            traced = 0;
            cluster_arrive();
        }
    }
    cluster_wait();  // no CTA leaves while another may still write its halo rows
    for (int i = tid; i < items; i += blockDim.x) {
        const int row = i / hpr, uu = i - row * hpr;
#pragma unroll
        for (int c = 0; c < 2; ++c)
            store_half(p, c, r0 + row, uu, uu == hpr - 1 ? last_nv : 8, pl[c * plane_words + hpr + i]);
    }
}

template <int K, bool RAGGED>
cudaError_t launch(const ResidentSweep &p, int cs, int threads, size_t smem, cudaStream_t s)
{
    auto kernel = resident_kernel<K, RAGGED>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cs);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

}  // namespace

// Where the line lies, us per recorded sweep here / with two launches per sweep
// (the host's rate): 512^2 2.7 / 3.4, 576^2 3.5 / 3.4 (16 SMs' multipliers bind);
// ragged rows 258^2 2.0 / 3.6, 510^2 4.2 / 3.5.
bool resident_fits(int64_t L) { return L <= (L % 16 ? 400 : 512); }

cudaError_t resident_sweep(ResidentSweep p, int64_t n_sweeps, cudaStream_t s)
{
    const int half = p.L / 2;
    p.hpr = (half + 7) / 8;
    int cs = 1;
    while (cs < kMaxCluster && 2 * cs <= p.L && (int64_t)p.L * p.hpr >= kItems * 2 * cs) cs *= 2;
    const int rows = (p.L + cs - 1) / cs, items = rows * p.hpr;
    const int k = (items + kMaxThreads - 33) / (kMaxThreads - 32);
    const int threads = ((items + k - 1) / k + 31) / 32 * 32 + 32;
    const size_t smem = ((2 + (threads - 32) / 32) * kTraceRows + 2 * (size_t)(rows + 2) * p.hpr) * sizeof(uint32_t);
    while (n_sweeps > 0) {
        p.n_sweeps = (int32_t)std::min<int64_t>(n_sweeps, kMaxSweeps);
        // at most 1024 half words per CTA on this route: one or two per thread
        cudaError_t e = half % 8 ? (k == 1 ? launch<1, true>(p, cs, threads, smem, s) : launch<2, true>(p, cs, threads, smem, s))
                                 : (k == 1 ? launch<1, false>(p, cs, threads, smem, s) : launch<2, false>(p, cs, threads, smem, s));
        if (e != cudaSuccess) return e;
        n_sweeps -= p.n_sweeps;
        p.t0 += (uint64_t)p.n_sweeps;
        if (p.trace) p.trace += 2 * p.n_sweeps;
    }
    return cudaSuccess;
}

}  // namespace ising
