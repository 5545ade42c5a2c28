// resident.cu -- whole sweep calls of small lattices in one launch of one
// thread-block cluster.
//
// A half-sweep of a small lattice is too little work for a launch: at 256^2 the
// multiplies of its draws take the whole chip 17 ns, while two launches per
// sweep cost 3.6 us of host time alone.  Here up to 16 CTAs of one cluster hold
// the lattice in shared memory for all sweeps of the call, a band of rows each.
//
// Both layouts are held the same way: 8 spins of a row to a 32-bit half word,
// one per nibble (0/1), ceil(L/2 / 8) half words per row and colour.  The last
// warps of a CTA decide, up to K half words of each colour per thread, whose own
// spins stay in registers; the others form the marks of the next sweep's draws
// meanwhile, in shared memory, a buffer per parity of the sweep.  The deciding
// warps meet between the colours, all of them behind each sweep.  What a band's
// first and last row become goes to the halo rows of the CTAs above and below as
// asynchronous remote stores that count at a barrier there (one per colour),
// which only the threads of the edge rows wait for.  Such a word is
// overwritten, two half-sweeps later, only after the row of the thread that reads
// it, sent behind that read, has arrived at its writer; so no other order is
// needed between CTAs.
//
// RAGGED: rows of one-byte lattices with L/2 not a multiple of 8.  The last half
// word of a row holds fewer spins (its other nibbles stay 0) and a half word's
// draws may start in the middle of a Philox block.
//
// Bound at 64^2 to 256^2 by the remote stores' way (~400 cycles per half-sweep)
// and a decision's chain of loads and logic (~150), beyond by the 16 SMs'
// multipliers.  us per sweep of 1000 recorded ones, with two launches per sweep /
// with marks, decisions and a cluster barrier with a release (~500 cycles of fence
// and remote stores) one after the other / this way: 32^2 3.6 / 0.89 / 0.44, 64^2 3.6 /
// 0.91 / 0.53, 256^2 3.6 / 1.12 / 0.79, 384^2 3.6 / 1.79 / 1.48, 512^2 3.6 / 2.66 / 2.32.
// On the way there: the same barrier with drawing warps 1.11 at 256^2, remote
// stores with branching decisions from addresses worked out in each of them 1.08 to
// 1.23.  (64-bit shared atomics for the sums cost 600 cycles per sweep; each warp
// has a word of its own instead.)
//
// The observables of each sweep are added up in the CTAs' shared memory and
// written by the first CTA every kTraceRows sweeps.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "launch.h"
#include "sweep_core.cuh"

namespace ising {

namespace {

constexpr int kMaxThreads = 1024;
constexpr int kMaxCluster = 16;
constexpr int kTraceRows = 128;
// Half words per CTA and colour below which the cluster is not doubled: 64^2 takes
// 0.51 us per sweep with at least 64, 0.64 with 128 and 0.71 with 256; 32^2, with at
// least 32, 0.51 in two CTAs and 0.38 in one.
constexpr int64_t kItems = 64;
// Sweeps per launch (7 ms at 32^2, 38 at 512^2): another stream's work is not kept
// waiting for the whole of a long call.
constexpr int64_t kMaxSweeps = 16384;
constexpr long long kWaitCycles = 4000000000LL;  // ~2 s
// What a cluster in which a wait gave up lingers at its end: remote stores issued
// before its last barrier have long landed then.
constexpr long long kLingerCycles = 200000LL;  // ~0.1 ms

// Set by a wait that gave up; resident_check reads and clears it.
__device__ int g_resident_error;
__device__ int g_resident_seen;  // what resident_check found

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
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

// Where `on`, writes v to the cluster address `a` and counts its bytes at the
// barrier `bar` of the same CTA.
__device__ __forceinline__ void peer_store_if(bool on, uint32_t a, uint32_t v, uint32_t bar)
{
    asm volatile("{\n\t"
                 ".reg .pred q;\n\t"
                 "setp.ne.u32 q, %3, 0;\n\t"
                 "@q st.async.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];\n\t"
                 "}" ::"r"(a), "r"(v), "r"(bar), "r"((uint32_t)on)
                 : "memory");
}

__device__ __forceinline__ void bar_init(uint32_t bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Waits until the barrier's phase of the given parity is over, at most `limit`
// cycles; sets `dead` if that was too short.
__device__ __forceinline__ void bar_wait(uint32_t bar, uint32_t parity, long long limit, bool &dead)
{
    if (dead) return;
    const long long start = clock64();
    for (;;) {
        uint32_t done;
        asm volatile("{\n\t"
                     ".reg .pred q;\n\t"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 q, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, q;\n\t"
                     "}"
                     : "=r"(done)
                     : "r"(bar), "r"(parity)
                     : "memory");
        if (done) return;
        if (clock64() - start > limit) {
            atomicExch(&g_resident_error, 1);
            dead = true;
            return;
        }
    }
}

__device__ __forceinline__ unsigned long long peer_load(uint32_t a)
{
    unsigned long long v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}

// Half word u of one plane row, and back (one-byte rows: nv spins of it, eight
// as one access where the rows are 8-byte aligned).
__device__ __forceinline__ uint32_t load_half(const ResidentSweep &p, int colour, int row, int u, int nv)
{
    const char *r = static_cast<const char *>(p.plane[colour]) + row * p.stride;
    if (!p.bytes) return reinterpret_cast<const uint32_t *>(r)[u];
    if (nv == 8 && p.wide) {
        const uint2 v = reinterpret_cast<const uint2 *>(r)[u];
        const uint32_t lo = __vcmpgts4(v.x, 0u) & 0x01010101u, hi = __vcmpgts4(v.y, 0u) & 0x01010101u;
        return __byte_perm(lo, hi, 0x6420) | (__byte_perm(lo, hi, 0x7531) << 4);
    }
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
    if (nv == 8 && p.wide) {
        auto bytes = [](uint32_t h, uint32_t sel) {  // four nibbles to +1 (0x01) or -1 (0xFF)
            return 0xFFFFFFFFu ^ (__byte_perm(h & 0x01010101u, (h >> 4) & 0x01010101u, sel) * 0xFEu);
        };
        reinterpret_cast<uint2 *>(r)[u] = make_uint2(bytes(x, 0x5140), bytes(x, 0x7362));
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
    uint32_t m[3] = {0, 0, 0}, other[3] = {0, 0, 0};  // other stays 0 where mark_ge keeps one counter
#pragma unroll
    for (int i = 0; i < (RAGGED ? 3 : 2); ++i) {
        if (i == 2 && o == 0) break;
        const uint4 u = philox(b + i, 0u, dc.c2, dc.c3, rk);
        mark_ge(m[i], other[i], u.x, dc.T3, dc.T4, 1u);
        mark_ge(m[i], other[i], u.y, dc.T3, dc.T4, 1u << 4);
        mark_ge(m[i], other[i], u.z, dc.T3, dc.T4, 1u << 8);
        mark_ge(m[i], other[i], u.w, dc.T3, dc.T4, 1u << 12);
        m[i] += other[i];
    }
    const uint32_t lo = m[0] | (m[1] << 16);
    return RAGGED ? __funnelshift_r(lo, m[2], 4 * o) : lo;
}

// What a CTA of the cluster works on; offsets into its shared memory in words.
struct Resident {
    int hpr, half, rows, r0, items;
    int nc;           // deciding threads, the last ones; the others draw
    int plane_words;  // per colour: local rows 0 (halo above), 1 .. rows, rows + 1 (halo below)
    int mark_words;   // per colour and sweep parity
    int last_nv;      // spins of a row's last half word
    int tw, plane, marks;
};

extern __shared__ __align__(16) uint32_t res_smem[];

// The marks of one half-sweep of a CTA's band, half words tid + k nc.
template <int K, bool RAGGED>
struct Drawer {
    uint32_t site[K];

    __device__ __forceinline__ Drawer(const Resident &c, int tid)
    {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int it = min(tid + k * c.nc, c.items - 1), row = it / c.hpr;
            site[k] = (uint32_t)(c.r0 + row) * (uint32_t)c.half + 8u * (uint32_t)(it - row * c.hpr);
        }
    }

    __device__ __forceinline__ void draw(const ResidentSweep &p, const Resident &c, int tid, uint64_t t, int colour, int to)
    {
        const DrawCtx dc{(uint32_t)t, counter_word3(colour, kPurposeMetropolis, t), p.acc.T3, p.acc.T4, p.acc.zero};
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (tid + k * c.nc < c.items)
                res_smem[to + k * c.nc] = marks8<RAGGED>(site[k] >> 2, site[k] & 3u, dc, p.rk);
    }
};

// Half words tid + k nc of a CTA's band, their current spins and what deciding
// them takes.  Everything that can be is worked out before the first sweep and
// nothing branches: a decision is a chain of loads and logic that one or two
// warps per scheduler do not hide.
template <int K, bool RAGGED>
struct Decider {
    int at[K];              // index in a plane
    int up[K], dn[K];       // rows above and below
    int left[K], right[K];  // the word beside it in its row, periodically
    uint32_t spins[2][K];
    uint32_t odd;           // bit k: odd row
    uint32_t ends;          // RAGGED, bit k: first of its row, bit k + 16: last
    uint32_t dst[K];        // where the halo copy of an edge row's word goes, as a cluster address; 0: nowhere
    uint32_t dst_bar[K];
    bool edge;

    // Sends no more halo words.
    __device__ __forceinline__ void mute()
    {
#pragma unroll
        for (int k = 0; k < K; ++k) dst[k] = 0u;
    }

    __device__ __forceinline__ Decider(const Resident &c, int tid, bool alone, uint32_t to_above, uint32_t to_below,
                                       uint32_t bar_above, uint32_t bar_below)
    {
        edge = false;
        odd = ends = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool ok = tid + k * c.nc < c.items;
            const int it = ok ? tid + k * c.nc : 0, row = it / c.hpr, u = it - row * c.hpr;
            at[k] = it + c.hpr;
            up[k] = alone && row == 0 ? at[k] + (c.rows - 1) * c.hpr : at[k] - c.hpr;
            dn[k] = alone && row == c.rows - 1 ? at[k] - (c.rows - 1) * c.hpr : at[k] + c.hpr;
            left[k] = at[k] + (u == 0 ? c.hpr - 1 : -1);
            right[k] = at[k] + (u == c.hpr - 1 ? 1 - c.hpr : 1);
            odd |= (uint32_t)((c.r0 + row) & 1) << k;
            ends |= (u == 0 ? 1u << k : 0u) | (u == c.hpr - 1 ? 0x10000u << k : 0u);
            // a band has two rows at least
            dst[k] = alone || !ok ? 0u : row == 0 ? to_above + 4u * u : row == c.rows - 1 ? to_below + 4u * u : 0u;
            dst_bar[k] = row == 0 ? bar_above : bar_below;
            edge = edge || dst[k] != 0u;
            for (int b = 0; b < 2; ++b) spins[b][k] = res_smem[c.plane + b * c.plane_words + at[k]];
        }
    }

    // Half word k of `colour`; its sums are added to `sums` for white.
    template <int COLOUR>
    __device__ __forceinline__ void decide(const Resident &c, int k, bool ok, uint32_t g, bool always, uint32_t &sums)
    {
        const int src = c.plane + (1 - COLOUR) * c.plane_words, tgt = c.plane + COLOUR * c.plane_words;
        const bool on_left = ((odd >> k) & 1u) == (uint32_t)COLOUR;
        const uint32_t above = res_smem[src + up[k]], below = res_smem[src + dn[k]], cur = spins[1 - COLOUR][k];
        const uint32_t w = res_smem[src + (on_left ? left[k] : right[k])];
        uint32_t sl, sr, mask = 0xFFFFFFFFu;
        if (RAGGED) {
            const uint32_t n4 = 4u * (uint32_t)c.last_nv;  // 4 .. 32 bits of a row's last half word
            const bool first = (ends >> k) & 1u, last = (ends >> (k + 16)) & 1u;
            sl = (cur << 4) | (w >> (first ? n4 - 4 : 28u));
            sr = (cur >> 4) | (w << (last ? n4 - 4 : 28u));
            if (last) mask = 0xFFFFFFFFu >> (32u - n4);
        } else {
            sl = __funnelshift_l(w, cur, 4);
            sr = __funnelshift_r(cur, w, 4);
        }
        const uint32_t e = above + below + cur + (on_left ? sl : sr);
        const uint32_t a8 = e + 0x88888888u, b8 = 0xCCCCCCCCu - e, tg = spins[COLOUR][k];
        uint32_t none = 0;
        uint32_t nt = always ? tg ^ kNibbleLsb : decide_sums<false, false>(tg, a8, b8, g, none);
        if (RAGGED) nt &= mask;
        spins[COLOUR][k] = nt;
        if (ok) res_smem[tgt + at[k]] = nt;
        peer_store_if(dst[k] != 0u, dst[k] + 4u * (COLOUR * c.plane_words), nt, dst_bar[k] + 8u * COLOUR);
        if (COLOUR == 1) {
            const uint32_t m = nt * 15u;
            uint32_t d2 = ((a8 & ~m) | (b8 & m)) & 0x77777777u;  // anti-aligned neighbours
            if (RAGGED) d2 &= mask;
            const uint32_t by = (d2 & 0x0F0F0F0Fu) + (d2 >> 4 & 0x0F0F0F0Fu);
            const uint32_t v = ((by * 0x01010101u) >> 24) | ((uint32_t)(__popc(nt) + __popc(cur)) << 16);
            sums += ok ? v : 0u;
        }
    }
};

template <int K, bool RAGGED>
__global__ void __launch_bounds__(kMaxThreads, 1) resident_kernel(const __grid_constant__ ResidentSweep p)
{
    __shared__ __align__(8) uint64_t halo_bar[2];  // per colour: the halo rows of its next update have arrived
    const int L = p.L, tid = threadIdx.x, lane = tid & 31;
    const int cs = (int)gridDim.x, rank = (int)cluster_rank();
    Resident c;
    c.hpr = p.hpr;
    c.half = L / 2;
    c.r0 = rank * L / cs;
    c.rows = (rank + 1) * L / cs - c.r0;
    c.items = c.rows * c.hpr;
    c.nc = p.deciders;
    const int most_rows = (L + cs - 1) / cs;
    c.plane_words = (most_rows + 2) * c.hpr;
    c.mark_words = most_rows * c.hpr;
    c.last_nv = c.half - 8 * (c.hpr - 1);
    // each traced sweep's sums [kTraceRows] (up spins in the high half, anti-
    // aligned pairs in the low half), the same per deciding warp (16 bits each),
    // the planes, the marks of two sweeps
    const int nw = c.nc >> 5;
    unsigned long long *tr = reinterpret_cast<unsigned long long *>(res_smem);
    c.tw = 2 * kTraceRows;
    c.plane = c.tw + kTraceRows * nw;
    c.marks = c.plane + 2 * c.plane_words;
    const int hpr = c.hpr, rows = c.rows, r0 = c.r0;
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(halo_bar), halo_bytes = 8u * (uint32_t)hpr;

    if (tid == 0) {
        for (int b = 0; b < 2; ++b) bar_init(bar + 8 * b);
        for (int b = 0; b < 2; ++b) bar_expect(bar + 8 * b, halo_bytes);
    }
    for (int i = tid; i < (rows + 2) * hpr; i += blockDim.x) {
        const int lr = i / hpr, u = i - lr * hpr;
        int row = r0 - 1 + lr;
        row = row < 0 ? row + L : (row >= L ? row - L : row);
#pragma unroll
        for (int b = 0; b < 2; ++b)
            res_smem[c.plane + b * c.plane_words + i] = load_half(p, b, row, u, u == hpr - 1 ? c.last_nv : 8);
    }
    const bool always = p.acc.always != 0, trace = p.trace != nullptr, draws = tid < (int)blockDim.x - c.nc;
    const int me = draws ? tid : tid - ((int)blockDim.x - c.nc);
    const bool two = (int)blockDim.x == 2 * c.nc;  // a drawing thread serves both colours
    // a wait ran out: no further ones, so that the launch ends, and nothing more is
    // sent or expected, so that no barrier counts what it was not told of
    bool dead = false;
    int traced = 0;     // sweeps summed in tr

    // Behind the sweeps of a trace's rows, by all threads: every CTA adds up its
    // warps; behind one more barrier the first CTA adds up the CTAs, and behind
    // another the sums may be written again.
    auto sweep_end = [&](int s) {
        __syncthreads();
        if (!trace || (++traced < kTraceRows && s + 1 < p.n_sweeps)) return;
        for (int i = tid; i < traced; i += blockDim.x) {
            unsigned long long v = 0;
            for (int w = 0; w < nw; ++w) {
                const uint32_t x = res_smem[c.tw + i * nw + w];
                v += ((unsigned long long)(x >> 16) << 32) | (x & 0xFFFFu);
            }
            tr[i] = v;
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();
        if (rank == 0) {
            const uint32_t tr_u32 = (uint32_t)__cvta_generic_to_shared(tr);
            const long long area = (long long)L * L;
            for (int i = tid; i < traced; i += blockDim.x) {
                long long ones = 0, anti = 0;
                for (int b = 0; b < cs; ++b) {
                    const unsigned long long v = peer_load(peer_addr(tr_u32 + 8u * (uint32_t)i, (uint32_t)b));
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
        __syncwarp();
        cluster_arrive();
        cluster_wait();
    };

    if (draws) {
        const int colour = me >= c.nc, mine = me - colour * c.nc;
        const int to = c.marks + colour * c.mark_words + mine;
        Drawer<K, RAGGED> drawer(c, mine);
        if (!always) drawer.draw(p, c, mine, p.t0, colour, to);
        if (two && !always) drawer.draw(p, c, mine, p.t0, 1, to + c.mark_words);
        __syncthreads();
        cluster_arrive();
        cluster_wait();
        for (int s = 0; s < p.n_sweeps; ++s) {
            if (!always && s + 1 < p.n_sweeps) {
                drawer.draw(p, c, mine, p.t0 + (uint64_t)s + 1, colour, to + 2 * ((s + 1) & 1) * c.mark_words);
                if (two) drawer.draw(p, c, mine, p.t0 + (uint64_t)s + 1, 1, to + (2 * ((s + 1) & 1) + 1) * c.mark_words);
            }
            sweep_end(s);
        }
    } else {
        __syncthreads();
        // the halo rows of the CTAs above (its row below) and below (its row above), and their barriers
        const uint32_t plane = (uint32_t)__cvta_generic_to_shared(res_smem + c.plane);
        const int above = rank == 0 ? cs - 1 : rank - 1, below = rank + 1 == cs ? 0 : rank + 1;
        const int rows_above = (above + 1) * L / cs - above * L / cs;
        Decider<K, RAGGED> d(c, me, cs == 1, peer_addr(plane + 4u * (uint32_t)((rows_above + 1) * hpr), (uint32_t)above),
                             peer_addr(plane, (uint32_t)below), peer_addr(bar, (uint32_t)above),
                             peer_addr(bar, (uint32_t)below));
        if (p.withhold && rank == 0) d.mute();
        __syncwarp();
        cluster_arrive();
        cluster_wait();
        for (int s = 0; s < p.n_sweeps; ++s) {
            uint32_t sums = 0;
            auto half_sweep = [&](auto colour_constant) {
                constexpr int COLOUR = decltype(colour_constant)::value;
                uint32_t g[K];
#pragma unroll
                for (int k = 0; k < K; ++k)
                    g[k] = res_smem[c.marks + (2 * (s & 1) + COLOUR) * c.mark_words + min(me + k * c.nc, c.items - 1)];
                if (d.edge && (s > 0 || COLOUR == 1)) {
                    // the other colour's halo rows: its update s, or s - 1 before black's
                    const uint32_t b = bar + 8 * (1 - COLOUR);
                    bar_wait(b, (uint32_t)(COLOUR == 1 ? s : s - 1) & 1u, p.wait_cycles, dead);
                    if (dead) d.mute();
                    else if (me == 0) bar_expect(b, halo_bytes);
                }
#pragma unroll
                for (int k = 0; k < K; ++k)
                    d.template decide<COLOUR>(c, k, me + k * c.nc < c.items, g[k], always, sums);
            };
            half_sweep(std::integral_constant<int, 0>{});
            // not bar.sync, which wants whole warps: edge and inner rows may share one, whose
            // lanes leave the wait above one by one
            asm volatile("barrier.sync 1, %0;" ::"r"(c.nc) : "memory");
            half_sweep(std::integral_constant<int, 1>{});
            if (trace) {
                // at most 32 K of each per lane: both sums of a warp fit 16 bits
                sums = __reduce_add_sync(0xffffffffu, sums);
                if (lane == 0) res_smem[c.tw + traced * nw + (me >> 5)] = sums;
            }
            sweep_end(s);
        }
        // no CTA leaves while another's halo words are on their way to it
        if (d.edge) bar_wait(bar + 8, (uint32_t)(p.n_sweeps - 1) & 1u, p.wait_cycles, dead);
        __syncwarp();
    }
    cluster_arrive();
    cluster_wait();
    // set by any CTA of this cluster before the barrier (or by an earlier launch)
    const int gave_up = *(volatile int *)&g_resident_error;
    for (int i = tid; i < c.items; i += blockDim.x) {
        const int row = i / hpr, uu = i - row * hpr;
#pragma unroll
        for (int b = 0; b < 2; ++b)
            store_half(p, b, r0 + row, uu, uu == hpr - 1 ? c.last_nv : 8, res_smem[c.plane + b * c.plane_words + hpr + i]);
    }
    if (gave_up)
        for (const long long start = clock64(); clock64() - start < kLingerCycles;) __nanosleep(1000);
}

__global__ void resident_flag_kernel() { g_resident_seen = atomicExch(&g_resident_error, 0); }

// How a side is cut: half words per row, CTAs, half words per deciding thread and
// colour, deciding threads and threads of a CTA, its shared memory.
struct Plan {
    int hpr, cs, k, deciders, threads;
    size_t smem;
};

Plan plan_of(int L)
{
    Plan q;
    const int half = L / 2;
    q.hpr = (half + 7) / 8;
    q.cs = 1;
    while (q.cs < kMaxCluster && 2 * q.cs <= L && (int64_t)L * q.hpr >= kItems * 2 * q.cs) q.cs *= 2;
    const int rows = (L + q.cs - 1) / q.cs, items = rows * q.hpr;
    // at most 1024 half words per CTA on this route: one or two per thread
    q.k = (items + kMaxThreads / 2 - 1) / (kMaxThreads / 2);
    q.deciders = ((items + q.k - 1) / q.k + 31) / 32 * 32;
    // as many threads draw, or twice as many where drawing takes longest and the
    // block has room: at two half words per thread (384^2 1.64 -> 1.43 us per sweep)
    // and with ragged rows, three Philox blocks per half word (100^2 0.89 -> 0.69; but
    // 256^2, one word each, 0.80 -> 0.84)
    q.threads = q.deciders * ((q.k > 1 || half % 8) && 3 * q.deciders <= kMaxThreads ? 3 : 2);
    q.smem = ((2 + q.deciders / 32) * kTraceRows + 2 * (size_t)(rows + 2) * q.hpr + 4 * (size_t)items) * sizeof(uint32_t);
    return q;
}

// Calls go(kernel) with the kernel of a plan.
template <typename Go>
auto with_kernel(const Plan &q, int L, Go go)
{
    if (L / 2 % 8) return q.k == 1 ? go(resident_kernel<1, true>) : go(resident_kernel<2, true>);
    return q.k == 1 ? go(resident_kernel<1, false>) : go(resident_kernel<2, false>);
}

struct Config {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];

    Config(int cs, int threads, size_t smem, cudaStream_t s)
    {
        cfg.gridDim = dim3((unsigned)cs);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cs;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};

// Whether the device has the SMs of one graphics processing cluster that a plan's
// CTAs need; a partition of it, or a limit on a process's SMs, may not.  A device on
// which the largest cluster fits (asked once per kernel) has room for every other.
constexpr size_t kMaxSmem = 40 * 1024;  // no plan takes more (512^2 36 KB)
constexpr int kMaxDevices = 64;
std::atomic<uint8_t> g_room[kMaxDevices][4];  // 0: not asked, 1: for any plan, 2: not for all

bool cluster_fits(const Plan &q, int L)
{
    if (q.cs == 1) return true;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return false;
    std::atomic<uint8_t> &room = g_room[dev][(q.k - 1) * 2 + (L / 2 % 8 ? 1 : 0)];
    if (room == 1) return true;
    return with_kernel(q, L, [&](auto kernel) {
        auto fits = [&](int cs, int threads, size_t smem) {
            int n = 0;
            Config c(cs, threads, smem, nullptr);
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                cudaOccupancyMaxActiveClusters(&n, kernel, &c.cfg) == cudaSuccess)
                return n > 0;
            cudaGetLastError();
            return false;
        };
        if (room == 0) room = fits(kMaxCluster, kMaxThreads, kMaxSmem) ? 1 : 2;
        return room == 1 || fits(q.cs, q.threads, q.smem);
    });
}

}  // namespace

// Where the line lies, us per recorded sweep here / with two launches per sweep
// (the host's rate): 512^2 2.3 / 3.6, 576^2 3.35 / 3.6 (16 SMs' multipliers bind);
// ragged rows 430^2 2.7 / 3.6, 510^2 3.4 / 3.6, 530^2 4.9 / 3.6.  A single call of
// few sweeps of ragged rows is no faster here from about 400^2 on (510^2, us per
// call of 1 / 3 / 10 sweeps: 14.7 / 22.6 / 45.5 here, 12.5 / 21.3 / 50.5 launched).
// One sweep of a one-byte lattice, us with nothing behind it / among others, here and
// launched: 256^2 20.4 / 8.7 and 18.9 / 10.5, 512^2 23.2 / 8.8 and 19.2 / 10.5, ragged
// 254^2 21.6 / 8.9 and 19.1 / 10.6, 398^2 24.5 / 10.3 and 19.3 / 10.6; a general kernel in
// two launches 22.5 / 10.9 at any of these sides, which is where the line lies.  (One
// MSC4 sweep 22.4 / 8.7 here at 512^2.)  Where the cluster has no room the launches serve any side.
bool resident_fits(int64_t L, int64_t n_sweeps, bool bytes)
{
    const bool ragged = L % 16 != 0, single = bytes && n_sweeps == 1;
    const int64_t most = single ? (ragged ? 256 : 400) : ragged && n_sweeps < 6 ? 400 : 512;
    return L <= most && cluster_fits(plan_of((int)L), (int)L);
}

cudaError_t resident_check(bool *gave_up, cudaStream_t s)
{
    static std::mutex mu;  // g_resident_seen serves one caller at a time
    std::lock_guard<std::mutex> lock(mu);
    int seen = 0;
    resident_flag_kernel<<<1, 1, 0, s>>>();
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyFromSymbolAsync(&seen, g_resident_seen, sizeof(int), 0, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    *gave_up = seen != 0;
    return e;
}

cudaError_t resident_sweep(ResidentSweep p, int64_t n_sweeps, cudaStream_t s)
{
    const Plan q = plan_of(p.L);
    p.hpr = q.hpr;
    p.deciders = q.deciders;
    p.wide = ((uintptr_t)p.plane[0] | (uintptr_t)p.plane[1] | (uint64_t)p.stride) % 8 == 0;
    if (p.wait_cycles == 0) p.wait_cycles = kWaitCycles;
    Config c(q.cs, q.threads, q.smem, s);
    while (n_sweeps > 0) {
        p.n_sweeps = (int32_t)std::min<int64_t>(n_sweeps, kMaxSweeps);
        cudaError_t e = with_kernel(q, p.L, [&](auto kernel) { return cudaLaunchKernelEx(&c.cfg, kernel, p); });
        if (e != cudaSuccess) return e;
        n_sweeps -= p.n_sweeps;
        p.t0 += (uint64_t)p.n_sweeps;
        if (p.trace) p.trace += 2 * p.n_sweeps;
    }
    return cudaSuccess;
}

}  // namespace ising
