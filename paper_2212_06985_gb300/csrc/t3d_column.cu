// Lattices whose syndrome and flip words fit one SM: a block keeps the whole lattice of one (or
// a few) 64-sample words in shared memory and runs a schedule of flip / p-flip applications
// -- or a whole Monte Carlo run, noise and measurement included -- without going back to global
// memory and without a launch per step.
//
// Samples are independent, so a word's column of the bit-sliced arrays never needs another
// column: what separates two applications is a barrier of one block instead of a kernel
// boundary.  Up to L = 14 the syndrome, the flip and the error words (72 bytes per site and word)
// fit the 227 KB a block can have.
//
// An application is two phases between barriers: every site decides its own three edges from
// the old syndrome (7 shared reads: the z-neighbour's words are the thread's previous ones)
// and writes the flip words; then every site's three faces take the flips of their edges (7
// shared reads, again the z-neighbour's kept in registers).  Each edge is decided once, where
// the one-pass kernel for larger lattices decides nine edges per site.
//
// Up to L = 10 a thread has one site and keeps its words in registers (k_column_one).  Above, thread
// (xy, word) of z-part zp walks the sites z0 <= z < z1 of one lattice column, so its x and y neighbour
// offsets are fixed for the whole kernel, and a column of random words shares the generator's first
// rounds (PhiloxColumn).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "t3d_device.cuh"
#include "t3d_host.hpp"
#include "t3d_items.cuh"

namespace t3d {
namespace {

constexpr size_t kColumnSmem = 227 * 1024;
constexpr int kColumnThreads = 1024;

struct ColumnProgram {
    uint64_t seed;
    uint64_t sched;        // bit k: letter k of the schedule is 'P'
    uint64_t thr_p, thr_q; // run: Bernoulli thresholds of noise and measurement
    uint32_t cycle0;       // sweeps: the cycle that keys the coins; run: cycles cycle0 + 1 ..
    uint32_t sweep0;
    int slen, n_apply;
    int cycles;            // run: noisy cycles
    int perfect;           // run: noiseless round decoded by up to this many applications, -1 = none
    int until_clear;       // sweeps: stop once the column's syndrome is clear
    int zt;                // z-parts of a lattice column (threads per (xy, word))
    int32_t* sweeps_done;  // until_clear: maximum over the columns (nullable)
};

// The rows of a column in global memory: word (row, w + wl) of a bit-sliced array.
struct Rows {
    uint64_t* p;
    int64_t W;
    __device__ __forceinline__ uint64_t& at(int row) const { return p[(int64_t)row * W]; }
};

// kRun: whole runs (sweeps otherwise, E gathering the flips for e).
template <bool kRun>
__global__ void __launch_bounds__(kColumnThreads, 1)
k_column(const __grid_constant__ ItemDesc d, const __grid_constant__ ColumnProgram pr)
{
    extern __shared__ uint64_t sm[];
    const int L = d.lat.L, L2 = d.lat.L2, L3 = d.lat.L3, Wt = d.tx;
    const int P = L2 * Wt, N = L3 * Wt;   // a z-plane, the lattice
    uint64_t* const S0 = sm;
    uint64_t* const F0 = sm + 3 * N;
    uint64_t* const E0 = sm + 6 * N;

    const int t = threadIdx.x;
    const int zp = t / P, u = t - zp * P, wl = u % Wt, xy = u / Wt;
    const int y = xy / L, x = xy - y * L;
    const bool mine = zp < pr.zt;
    const int z0 = mine ? zp * L / pr.zt : 0, z1 = mine ? (zp + 1) * L / pr.zt : 0;
    const int xm = (x == 0 ? L - 1 : -1) * Wt, xp = (x + 1 == L ? 1 - L : 1) * Wt;
    const int ym = (y == 0 ? L - 1 : -1) * L * Wt, yp = (y + 1 == L ? 1 - L : 1) * L * Wt;

    const int64_t words = d.nw ? d.nw : d.W;
    const int64_t have = d.live ? min(words, *d.live - d.w0) : words;
    for (int64_t w0 = (int64_t)blockIdx.x * Wt; w0 < have; w0 += (int64_t)gridDim.x * Wt) {
        const int64_t w = w0 + wl;
        const bool act = mine && w < have;
        const int zb = act ? z0 : 0, ze = act ? z1 : 0;   // empty for threads without a word
        const uint64_t group = act ? word_group(d, w) : 0;
        const Rows e{d.e + w, d.W}, s{d.s + w, d.W};

        // one application; returns whether this thread's faces keep an unsatisfied check
        auto apply = [&](bool prob, uint32_t cycle, uint32_t sweep) -> uint64_t {
            {
                PhiloxColumn pc;
                PhiloxBlock b0, b1;
                if (prob) {
                    pc = philox_column(pr.seed, kStreamCoin, cycle, sweep, group);
                    b0 = philox_block(pc, 0);
                    b1 = philox_block(pc, 1);
                }
                int i = zb * P + u;
                const int below = (zb == 0 ? L - 1 : zb - 1) * P + u;
                uint64_t s0m = 0, s1m = 0;
                if (zb < ze) {
                    s0m = S0[below];
                    s1m = S0[N + below];
                }
                for (int z = zb; z < ze; ++z, i += P) {
                    const uint64_t s0 = S0[i], s1 = S0[N + i], s2 = S0[2 * N + i];
                    const uint64_t s2y = S0[2 * N + i + ym], s2x = S0[2 * N + i + xm], s1x = S0[N + i + xm],
                                   s0y = S0[i + ym];
                    uint64_t f[3] = {at_least_three(s2, s2y, s1, s1m), at_least_three(s2, s2x, s0, s0m),
                                     at_least_three(s1, s1x, s0, s0y)};
                    if (prob) {
                        const PhiloxSite ps = philox_site(pc, (uint32_t)(z * L2 + xy));
                        const U32x4 a = philox_finish(pc, ps, b0), b = philox_finish(pc, ps, b1);
                        f[0] |= exactly_two(s2, s2y, s1, s1m) & ((uint64_t)a.v[0] | ((uint64_t)a.v[1] << 32));
                        f[1] |= exactly_two(s2, s2x, s0, s0m) & ((uint64_t)a.v[2] | ((uint64_t)a.v[3] << 32));
                        f[2] |= exactly_two(s1, s1x, s0, s0y) & ((uint64_t)b.v[0] | ((uint64_t)b.v[1] << 32));
                    }
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        F0[k * N + i] = f[k];
                        if (f[k]) E0[k * N + i] ^= f[k];
                    }
                    s0m = s0;
                    s1m = s1;
                }
            }
            __syncthreads();
            uint64_t nz = 0;
            {
                int i = (ze - 1) * P + u;
                const int above = (ze == L ? 0 : ze) * P + u;
                uint64_t fxp = 0, fyp = 0;
                if (zb < ze) {
                    fxp = F0[above];
                    fyp = F0[N + above];
                }
                for (int z = ze - 1; z >= zb; --z, i -= P) {
                    const uint64_t fx = F0[i], fy = F0[N + i], fz = F0[2 * N + i];
                    const uint64_t fzy = F0[2 * N + i + yp], fzx = F0[2 * N + i + xp], fxy = F0[i + yp],
                                   fyx = F0[N + i + xp];
                    const uint64_t n0 = S0[i] ^ fy ^ fyp ^ fz ^ fzy, n1 = S0[N + i] ^ fx ^ fxp ^ fz ^ fzx,
                                   n2 = S0[2 * N + i] ^ fx ^ fxy ^ fy ^ fyx;
                    S0[i] = n0;
                    S0[N + i] = n1;
                    S0[2 * N + i] = n2;
                    nz |= n0 | n1 | n2;
                    fxp = fx;
                    fyp = fy;
                }
            }
            return nz;
        };

        // up to `most` flip applications, stopping once the column is clear: the applications that ran
        auto flip_until_clear = [&](int most) -> int {
            uint64_t nz = 0;
            for (int z = zb, i = zb * P + u; z < ze; ++z, i += P) nz |= S0[i] | S0[N + i] | S0[2 * N + i];
            int k = 0;
            while (k < most && __syncthreads_or(nz != 0)) {
                nz = apply(false, 0, 0);
                ++k;
            }
            __syncthreads();
            return k;
        };

        if (!kRun) {
            for (int z = zb, i = zb * P + u; z < ze; ++z, i += P) {
#pragma unroll
                for (int n = 0; n < 3; ++n) {
                    S0[n * N + i] = s.at(n * L3 + z * L2 + xy);
                    E0[n * N + i] = 0;
                }
            }
            __syncthreads();
            if (pr.until_clear) {
                const int k = flip_until_clear(pr.n_apply);
                if (pr.sweeps_done && t == 0) atomicMax(pr.sweeps_done, k);
            } else {
                for (int k = 0, letter = 0; k < pr.n_apply; ++k) {
                    apply((pr.sched >> letter) & 1, pr.cycle0, pr.sweep0 + (uint32_t)k);
                    if (++letter == pr.slen) letter = 0;
                    __syncthreads();
                }
            }
            for (int z = zb, i = zb * P + u; z < ze; ++z, i += P) {
#pragma unroll
                for (int n = 0; n < 3; ++n) {
                    s.at(n * L3 + z * L2 + xy) = S0[n * N + i];
                    xor_into(&e.at(n * L3 + z * L2 + xy), E0[n * N + i]);
                }
            }
        } else {
            for (int z = zb, i = zb * P + u; z < ze; ++z, i += P)
#pragma unroll
                for (int k = 0; k < 3; ++k) E0[k * N + i] = e.at(k * L3 + z * L2 + xy);

            auto noise = [&](uint32_t cycle) {
                if (pr.thr_p == 0) return;
                const bool all = pr.thr_p >> 32;
                const BernoulliColumn bc = bernoulli_column(pr.seed, kStreamQubit, cycle, group);
                for (int z = zb, i = zb * P + u; z < ze; ++z, i += P)
#pragma unroll 1
                    for (int k = 0; k < 3; ++k) {
                        const uint64_t f = all ? ~0ULL
                                               : bernoulli_site(bc, (uint32_t)pr.thr_p,
                                                                (uint32_t)(k * L3 + z * L2 + xy));
                        E0[k * N + i] ^= f;
                    }
            };
            auto measure = [&](uint64_t thr, uint32_t cycle) {
                const bool all = thr >> 32, none = thr == 0;
                const BernoulliColumn bc = bernoulli_column(pr.seed, kStreamMeas, cycle, group);
                for (int z = zb, i = zb * P + u; z < ze; ++z, i += P) {
                    const int zz = (z + 1 == L ? 1 - L : 1) * P, site = z * L2 + xy;
                    const uint64_t *px = E0 + i, *py = px + N, *pz = py + N;
                    const uint64_t ex = px[0], exy = px[yp], exz = px[zz], ey = py[0], eyx = py[xp], eyz = py[zz],
                                   ez = pz[0], ezx = pz[xp], ezy = pz[yp];
                    S0[i] = ey ^ eyz ^ ez ^ ezy;
                    S0[N + i] = ex ^ exz ^ ez ^ ezx;
                    S0[2 * N + i] = ex ^ exy ^ ey ^ eyx;
                    if (none) continue;
#pragma unroll 1
                    for (int n = 0; n < 3; ++n)
                        S0[n * N + i] ^= all ? ~0ULL : bernoulli_site(bc, (uint32_t)thr, (uint32_t)(n * L3 + site));
                }
            };

            for (int c = 1; c <= pr.cycles; ++c) {
                const uint32_t cycle = pr.cycle0 + (uint32_t)c;
                noise(cycle);
                __syncthreads();
                measure(pr.thr_q, cycle);
                __syncthreads();
                for (int k = 0, letter = 0; k < pr.n_apply; ++k) {
                    apply((pr.sched >> letter) & 1, cycle, (uint32_t)k);
                    if (++letter == pr.slen) letter = 0;
                    __syncthreads();
                }
            }
            if (pr.perfect >= 0) {
                __syncthreads();
                measure(0, 0);
                __syncthreads();
                flip_until_clear(pr.perfect);
            }
            for (int z = zb, i = zb * P + u; z < ze; ++z, i += P)
#pragma unroll
                for (int k = 0; k < 3; ++k) e.at(k * L3 + z * L2 + xy) = E0[k * N + i];
        }
        __syncthreads();   // the next column overwrites the words
    }
}

// k_column for lattices with at most one site per thread (L <= 10): the site's syndrome, errors and flips
// stay in the thread's registers, and shared memory holds only what neighbours read.  A few columns are a
// chain of dependent applications, whose length halves without the loops and the words' way through
// shared memory; many are bound by the ALUs, which have less to do.  T = 4 cycles with the readout, z-parts
// of several sites -> this: L = 4, 10,000 samples, 32 flips a cycle 100 -> 61 us; FFPFF at L = 6, 300,000
// 822 -> 619 us; L = 8, 10^6 4.41 -> 4.24 ms; L = 10, 300,000 3.72 -> 3.52 ms.
template <bool kRun>
__global__ void __launch_bounds__(kColumnThreads, 1)
k_column_one(const __grid_constant__ ItemDesc d, const __grid_constant__ ColumnProgram pr)
{
    extern __shared__ uint64_t sm[];
    const int L = d.lat.L, L2 = d.lat.L2, L3 = d.lat.L3, Wt = d.tx;
    const int P = L2 * Wt, N = L3 * Wt;   // a z-plane, the lattice
    uint64_t* const S0 = sm;
    uint64_t* const F0 = sm + 3 * N;
    uint64_t* const E0 = sm + 6 * N;

    const int i = threadIdx.x;            // the site's place: word fastest, then x, y, z
    const int z = i / P, u = i - z * P, wl = u % Wt, xy = u / Wt;
    const int y = xy / L, x = xy - y * L, site = z * L2 + xy;
    const int xm = i + (x == 0 ? L - 1 : -1) * Wt, xp = i + (x + 1 == L ? 1 - L : 1) * Wt;
    const int ym = i + (y == 0 ? L - 1 : -1) * L * Wt, yp = i + (y + 1 == L ? 1 - L : 1) * L * Wt;
    const int zm = i + (z == 0 ? L - 1 : -1) * P, zp = i + (z + 1 == L ? 1 - L : 1) * P;

    const int64_t words = d.nw ? d.nw : d.W;
    const int64_t have = d.live ? min(words, *d.live - d.w0) : words;
    for (int64_t w0 = (int64_t)blockIdx.x * Wt; w0 < have; w0 += (int64_t)gridDim.x * Wt) {
        const int64_t w = w0 + wl;
        const bool on = i < N && w < have;
        const uint64_t group = on ? word_group(d, w) : 0;
        const Rows eg{d.e + w, d.W}, sg{d.s + w, d.W};
        uint64_t s[3] = {0, 0, 0}, e[3] = {0, 0, 0};   // the site's faces and edges

        // one application; returns whether this thread's faces keep an unsatisfied check
        auto apply = [&](bool prob, uint32_t cycle, uint32_t sweep) -> uint64_t {
            uint64_t f[3] = {0, 0, 0};
            if (on) {
                const uint64_t s2y = S0[2 * N + ym], s2x = S0[2 * N + xm], s1x = S0[N + xm], s0y = S0[ym],
                               s0z = S0[zm], s1z = S0[N + zm];
                f[0] = at_least_three(s[2], s2y, s[1], s1z);
                f[1] = at_least_three(s[2], s2x, s[0], s0z);
                f[2] = at_least_three(s[1], s1x, s[0], s0y);
                if (prob) {
                    const PhiloxColumn pc = philox_column(pr.seed, kStreamCoin, cycle, sweep, group);
                    const PhiloxSite ps = philox_site(pc, (uint32_t)site);
                    const U32x4 a = philox_finish(pc, ps, philox_block(pc, 0));
                    const U32x4 b = philox_finish(pc, ps, philox_block(pc, 1));
                    f[0] |= exactly_two(s[2], s2y, s[1], s1z) & ((uint64_t)a.v[0] | ((uint64_t)a.v[1] << 32));
                    f[1] |= exactly_two(s[2], s2x, s[0], s0z) & ((uint64_t)a.v[2] | ((uint64_t)a.v[3] << 32));
                    f[2] |= exactly_two(s[1], s1x, s[0], s0y) & ((uint64_t)b.v[0] | ((uint64_t)b.v[1] << 32));
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    F0[k * N + i] = f[k];
                    e[k] ^= f[k];
                }
            }
            __syncthreads();
            if (on) {
                s[0] ^= f[1] ^ F0[N + zp] ^ f[2] ^ F0[2 * N + yp];
                s[1] ^= f[0] ^ F0[zp] ^ f[2] ^ F0[2 * N + xp];
                s[2] ^= f[0] ^ F0[yp] ^ f[1] ^ F0[N + xp];
#pragma unroll
                for (int k = 0; k < 3; ++k) S0[k * N + i] = s[k];
            }
            return s[0] | s[1] | s[2];
        };

        // up to `most` flip applications, stopping once the column is clear: the applications that ran
        auto flip_until_clear = [&](int most) -> int {
            uint64_t nz = s[0] | s[1] | s[2];
            int k = 0;
            while (k < most && __syncthreads_or(nz != 0)) {
                nz = apply(false, 0, 0);
                ++k;
            }
            return k;
        };

        auto schedule = [&](uint32_t cycle, uint32_t sweep0) {
            for (int k = 0, letter = 0; k < pr.n_apply; ++k) {
                __syncthreads();
                apply((pr.sched >> letter) & 1, cycle, sweep0 + (uint32_t)k);
                if (++letter == pr.slen) letter = 0;
            }
        };

        if (!kRun) {
            if (on) {
#pragma unroll
                for (int n = 0; n < 3; ++n) S0[n * N + i] = s[n] = sg.at(n * L3 + site);
            }
            if (pr.until_clear) {
                const int k = flip_until_clear(pr.n_apply);
                if (pr.sweeps_done && threadIdx.x == 0) atomicMax(pr.sweeps_done, k);
            } else {
                schedule(pr.cycle0, pr.sweep0);
            }
            if (on) {
#pragma unroll
                for (int n = 0; n < 3; ++n) {
                    sg.at(n * L3 + site) = s[n];
                    xor_into(&eg.at(n * L3 + site), e[n]);
                }
            }
        } else {
            // the syndrome of e, measured with error rate thr / 2^32
            auto measure = [&](uint64_t thr, uint32_t cycle) {
                __syncthreads();   // the last measurement's reads are done
                if (on) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) E0[k * N + i] = e[k];
                }
                __syncthreads();
                if (on) {
                    s[0] = e[1] ^ E0[N + zp] ^ e[2] ^ E0[2 * N + yp];
                    s[1] = e[0] ^ E0[zp] ^ e[2] ^ E0[2 * N + xp];
                    s[2] = e[0] ^ E0[yp] ^ e[1] ^ E0[N + xp];
                    if (thr != 0) {
                        const BernoulliColumn bc = bernoulli_column(pr.seed, kStreamMeas, cycle, group);
#pragma unroll
                        for (int n = 0; n < 3; ++n)
                            s[n] ^= thr >> 32 ? ~0ULL : bernoulli_site(bc, (uint32_t)thr, (uint32_t)(n * L3 + site));
                    }
#pragma unroll
                    for (int n = 0; n < 3; ++n) S0[n * N + i] = s[n];
                }
            };
            if (on) {
#pragma unroll
                for (int k = 0; k < 3; ++k) e[k] = eg.at(k * L3 + site);
            }
            for (int c = 1; c <= pr.cycles; ++c) {
                const uint32_t cycle = pr.cycle0 + (uint32_t)c;
                if (pr.thr_p != 0 && on) {
                    const BernoulliColumn bc = bernoulli_column(pr.seed, kStreamQubit, cycle, group);
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        e[k] ^= pr.thr_p >> 32 ? ~0ULL
                                               : bernoulli_site(bc, (uint32_t)pr.thr_p, (uint32_t)(k * L3 + site));
                }
                measure(pr.thr_q, cycle);
                schedule(cycle, 0);
            }
            if (pr.perfect >= 0) {
                measure(0, 0);
                flip_until_clear(pr.perfect);
            }
            if (on) {
#pragma unroll
                for (int k = 0; k < 3; ++k) eg.at(k * L3 + site) = e[k];
            }
        }
        __syncthreads();   // the next column overwrites the words
    }
}

// ------------------------------------------------------------------ slabs of a cluster
// Larger lattices (L = 15 .. 32): the lattice of one word is split into z-slabs over the blocks
// of a thread-block cluster, each keeping its slab's syndrome and flip words in shared memory.
// The two phases of an application read one word per (x, y) column from the neighbouring block
// (distributed shared memory): the syndrome below the slab, the flips above it; a cluster barrier
// separates them.  The flips that reach e are gathered in registers, up to 2 kZ sites a thread,
// and XORed into e once at the end.
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The word at this block's shared-memory address `p` in block `rank` of the cluster.
__device__ __forceinline__ uint64_t cluster_load(const uint64_t* p, uint32_t rank)
{
    uint64_t v;
    asm volatile(
        "{\n"
        ".reg .u32 a;\n"
        "mapa.shared::cluster.u32 a, %1, %2;\n"
        "ld.shared::cluster.u64 %0, [a];\n"
        "}\n"
        : "=l"(v)
        : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank)
        : "memory");
    return v;
}

__device__ __forceinline__ void cluster_store(uint32_t* p, uint32_t rank, uint32_t v)
{
    asm volatile(
        "{\n"
        ".reg .u32 a;\n"
        "mapa.shared::cluster.u32 a, %0, %1;\n"
        "st.shared::cluster.u32 [a], %2;\n"
        "}\n" ::"r"((uint32_t)__cvta_generic_to_shared(p)),
        "r"(rank), "r"(v)
        : "memory");
}

constexpr int kMaxCluster = 8;

// Where a word's column lies: row r of word w at p[r * row + w * word].
struct ColumnView {
    uint64_t* p;
    int64_t row, word;
    __device__ __forceinline__ uint64_t& at(int64_t r, int64_t w) const { return p[r * row + w * word]; }
};

// Keeps the compiler from computing what follows from v outside the loop over applications: the
// unrolled sites' shared-memory addresses, kept in registers across it, would push the state
// itself into local memory.
__device__ __forceinline__ int here(int v)
{
    asm volatile("" : "+r"(v));
    return v;
}

// Thread (x, j) of z-part zp owns the sites of rows j and j + ceil(L / 2), z0 <= z < z1 (at most
// kZ planes); the z-neighbours are words it has just read.  Bound by the shared-memory pipe (23
// words read or written per site and application) and, in p-flip, the ALU (the coins).  Measured
// at L = 32, 10^5 samples, one application of a longer schedule: flip 0.43 ms against 0.83 as a
// kernel of its own, p-flip 0.83 against 1.46; the columns' way in and out costs 2.2 ms once (see
// route_schedule).  Keeping the syndrome in registers too (17 words, but 96 registers of state, which
// spill) measured the same, row pairs with shared y-neighbours and prefetched planes slower.
template <int kZ, int kT>
__global__ void __launch_bounds__(kT, 1)
k_slab(const __grid_constant__ ItemDesc d, const __grid_constant__ ColumnProgram pr, int C, const ColumnView sv,
       const ColumnView ev, int e_store)
{
    extern __shared__ uint64_t sm[];
    __shared__ uint32_t left[2][kMaxCluster];   // flip until clear: the blocks' unsatisfied checks
    const int L = d.lat.L, P = d.lat.L2, L3 = d.lat.L3;
    const int rank = (int)(blockIdx.x % (unsigned)C);
    const int zbase = rank * L / C, nz = (rank + 1) * L / C - zbase, most = (L + C - 1) / C;
    const int down = rank == 0 ? C - 1 : rank - 1, up = rank + 1 == C ? 0 : rank + 1;
    const int nz_down = (down + 1) * L / C - down * L / C;
    const int N = most * P;
    uint64_t* const S0 = sm;
    uint64_t* const S1 = sm + N;
    uint64_t* const S2 = sm + 2 * N;
    uint64_t* const Fx = sm + 3 * N;
    uint64_t* const Fy = sm + 4 * N;
    uint64_t* const Fz = sm + 5 * N;

    const int t = threadIdx.x;
    const int half = (L + 1) / 2, H = half * L;    // rows j and j + half of a plane
    const int zp = t / H, u = t - zp * H;
    const int j = u / L, x = u - j * L;
    const bool mine = zp < pr.zt;
    const int rows = !mine ? 0 : j + half < L ? 2 : 1;
    const int z0 = mine ? zp * nz / pr.zt : 0, z1 = mine ? (zp + 1) * nz / pr.zt : 0;
    // offsets of the y-neighbours of the two rows (periodic)
    const int ym0 = j == 0 ? (L - 1) * L : -L, ym1 = -L;
    const int yp0 = j + 1 == L ? -j * L : L, yp1 = j + half + 1 == L ? -(j + half) * L : L;
    const int xm = x == 0 ? L - 1 : -1, xp = x + 1 == L ? 1 - L : 1;

    const int64_t words = d.nw ? d.nw : d.W;
    const int64_t have = d.live ? min(words, *d.live - d.w0) : words;
    for (int64_t w = blockIdx.x / (unsigned)C; w < have; w += gridDim.x / (unsigned)C) {
        const uint64_t group = word_group(d, w);
        const int o0 = here(z0 * P + u), r0 = here((zbase + z0) * P + u);
        uint64_t acc[kZ][2][3];
#pragma unroll
        for (int k = 0; k < kZ; ++k)
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int n = 0; n < 3; ++n) {
                    acc[k][c][n] = 0;
                    if (z0 + k < z1 && c < rows)
                        sm[n * N + o0 + k * P + c * H] = sv.at(n * L3 + r0 + k * P + c * H, w);
                }
        cluster_barrier();

        // the coin words of the thread's edges into F (p-flip; each thread reads its own back)
        auto coins = [&](uint32_t sweep) {
            const PhiloxColumn pc = philox_column(pr.seed, kStreamCoin, pr.cycle0, sweep, group);
            const PhiloxBlock b0 = philox_block(pc, 0), b1 = philox_block(pc, 1);
            for (int c = 0; c < rows; ++c)
                for (int z = z0; z < z1; ++z) {
                    const int i = z * P + u + c * H;
                    const PhiloxSite ps = philox_site(pc, (uint32_t)(zbase * P + i));
                    const U32x4 a = philox_finish(pc, ps, b0);
                    Fx[i] = (uint64_t)a.v[0] | ((uint64_t)a.v[1] << 32);
                    Fy[i] = (uint64_t)a.v[2] | ((uint64_t)a.v[3] << 32);
                    const U32x4 b = philox_finish(pc, ps, b1);
                    Fz[i] = (uint64_t)b.v[0] | ((uint64_t)b.v[1] << 32);
                }
        };
        // decide: flips of the thread's edges into F and acc
        auto decide = [&](auto prob) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (c >= rows) break;
                int i = here(z0 * P + u + c * H);
                uint64_t m0, m1;   // faces 0 and 1 of the plane below
                if (z0 == 0) {
                    m0 = cluster_load(S0 + (nz_down - 1) * P + i, (uint32_t)down);
                    m1 = cluster_load(S1 + (nz_down - 1) * P + i, (uint32_t)down);
                } else {
                    m0 = S0[i - P];
                    m1 = S1[i - P];
                }
                const int im = c ? ym1 : ym0;
#pragma unroll
                for (int k = 0; k < kZ; ++k, i += P) {
                    if (z0 + k >= z1) break;
                    const uint64_t s0 = S0[i], s1 = S1[i], s2 = S2[i];
                    const uint64_t s2y = S2[i + im], s2x = S2[i + xm], s1x = S1[i + xm], s0y = S0[i + im];
                    uint64_t fx = at_least_three(s2, s2y, s1, m1), fy = at_least_three(s2, s2x, s0, m0),
                             fz = at_least_three(s1, s1x, s0, s0y);
                    if (decltype(prob)::value) {
                        fx |= exactly_two(s2, s2y, s1, m1) & Fx[i];
                        fy |= exactly_two(s2, s2x, s0, m0) & Fy[i];
                        fz |= exactly_two(s1, s1x, s0, s0y) & Fz[i];
                    }
                    Fx[i] = fx;
                    Fy[i] = fy;
                    Fz[i] = fz;
                    acc[k][c][0] ^= fx;
                    acc[k][c][1] ^= fy;
                    acc[k][c][2] ^= fz;
                    m0 = s0;
                    m1 = s1;
                }
            }
        };
        // update: the faces take their edges' flips; whether any keeps an unsatisfied check
        auto update = [&]() -> uint64_t {
            uint64_t nz_left = 0;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (c >= rows) break;
                const int top = here(u + c * H);
                uint64_t fxa, fya;   // x- and y-edge flips of the plane above
                if (z1 == nz) {
                    fxa = cluster_load(Fx + top, (uint32_t)up);
                    fya = cluster_load(Fy + top, (uint32_t)up);
                } else {
                    fxa = Fx[z1 * P + top];
                    fya = Fy[z1 * P + top];
                }
                const int ip = c ? yp1 : yp0;
                int i = top + (z0 + kZ - 1) * P;
#pragma unroll
                for (int k = kZ - 1; k >= 0; --k, i -= P) {
                    if (z0 + k >= z1) continue;
                    const uint64_t fx = Fx[i], fy = Fy[i], fz = Fz[i];
                    const uint64_t n0 = S0[i] ^ fy ^ fya ^ fz ^ Fz[i + ip],
                                   n1 = S1[i] ^ fx ^ fxa ^ fz ^ Fz[i + xp],
                                   n2 = S2[i] ^ fx ^ Fx[i + ip] ^ fy ^ Fy[i + xp];
                    S0[i] = n0;
                    S1[i] = n1;
                    S2[i] = n2;
                    nz_left |= n0 | n1 | n2;
                    fxa = fx;
                    fya = fy;
                }
            }
            return nz_left;
        };

        if (pr.until_clear) {
            uint64_t nz_left = 0;
            for (int c = 0; c < rows; ++c)
                for (int z = z0; z < z1; ++z) {
                    const int i = z * P + u + c * H;
                    nz_left |= S0[i] | S1[i] | S2[i];
                }
            int ran = 0;
            for (;;) {
                // every block tells every block; the slots alternate, so a slot is written again
                // only after the barrier that follows its reads
                const uint32_t any = __syncthreads_or(nz_left != 0) ? 1u : 0u;
                if (t < C) cluster_store(&left[ran & 1][rank], (uint32_t)t, any);
                cluster_barrier();
                uint32_t all = 0;
                for (int r = 0; r < C; ++r) all |= left[ran & 1][r];
                if (!all || ran == pr.n_apply) break;
                decide(std::false_type());
                cluster_barrier();
                nz_left = update();
                ++ran;
            }
            if (pr.sweeps_done && rank == 0 && t == 0) atomicMax(pr.sweeps_done, ran);
        } else {
            for (int k = 0, letter = 0; k < pr.n_apply; ++k) {
                if ((pr.sched >> letter) & 1) {
                    coins(pr.sweep0 + (uint32_t)k);
                    decide(std::true_type());
                } else {
                    decide(std::false_type());
                }
                if (++letter == pr.slen) letter = 0;
                cluster_barrier();
                update();
                cluster_barrier();
            }
        }
        const int r1 = here((zbase + z0) * P + u);
#pragma unroll
        for (int k = 0; k < kZ; ++k)
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (z0 + k < z1 && c < rows) {
#pragma unroll
                    for (int n = 0; n < 3; ++n) {
                        const int64_t r = n * L3 + r1 + k * P + c * H;
                        sv.at(r, w) = sm[n * N + o0 + k * P + c * H];
                        if (e_store)
                            ev.at(r, w) = acc[k][c][n];
                        else
                            xor_into(&ev.at(r, w), acc[k][c][n]);
                    }
                }
    }
}

// Word rows <-> contiguous columns: in [R][W] -> out [W][R] and back (kXor: XORed into the
// rows), in 32 x 32 tiles through shared memory, 256-byte runs on both sides.
constexpr int kTurn = 32;

__global__ void __launch_bounds__(256) k_to_columns(int64_t R, int64_t W, const uint64_t* __restrict__ in,
                                                    uint64_t* __restrict__ out)
{
    __shared__ uint64_t tile[kTurn][kTurn + 1];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t r0 = (int64_t)blockIdx.x * kTurn, w0 = (int64_t)blockIdx.y * kTurn;
#pragma unroll
    for (int i = 0; i < kTurn; i += 8)
        if (r0 + ty + i < R && w0 + tx < W) tile[ty + i][tx] = in[(r0 + ty + i) * W + w0 + tx];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kTurn; i += 8)
        if (w0 + ty + i < W && r0 + tx < R) out[(w0 + ty + i) * R + r0 + tx] = tile[tx][ty + i];
}

template <bool kXor>
__global__ void __launch_bounds__(256) k_from_columns(int64_t R, int64_t W, const uint64_t* __restrict__ in,
                                                      uint64_t* __restrict__ out)
{
    __shared__ uint64_t tile[kTurn][kTurn + 1];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t r0 = (int64_t)blockIdx.x * kTurn, w0 = (int64_t)blockIdx.y * kTurn;
    uint64_t was[4] = {0, 0, 0, 0};
#pragma unroll
    for (int i = 0; i < kTurn; i += 8) {
        if (w0 + ty + i < W && r0 + tx < R) tile[ty + i][tx] = __ldcs(&in[(w0 + ty + i) * R + r0 + tx]);
        if (kXor && r0 + ty + i < R && w0 + tx < W) was[i / 8] = out[(r0 + ty + i) * W + w0 + tx];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kTurn; i += 8)
        if (r0 + ty + i < R && w0 + tx < W) out[(r0 + ty + i) * W + w0 + tx] = was[i / 8] ^ tile[tx][ty + i];
}

// Resident blocks by cluster size.
constexpr int kResident[kMaxCluster + 1] = {0, 152, 152, 138, 144, 140, 138, 105, 120};

// Blocks of a cluster for lattice size L: the choice with the most busy SMs, counting the blocks
// that can be resident with about 200 KB each (cudaOccupancyMaxActiveClusters on GB300) and the
// share of them that a split of L planes into unequal slabs leaves waiting.  A thread takes at
// most four planes of its row pair (24 words of flips, 48 registers).  cluster 0: none fits.
struct SlabShape {
    int cluster, zt, z, threads;
    size_t smem;
};

SlabShape slab_shape(int L)
{
    SlabShape best{0, 0, 0, 0, 0};
    double busy = 0.0;
    const int per = (L + 1) / 2 * L;
    for (int c = 1; c <= kMaxCluster && c <= L; ++c) {
        const int most = (L + c - 1) / c;
        const size_t smem = (size_t)48 * L * L * most;
        if (smem + 1024 > kColumnSmem) continue;
        const double b = kResident[c] * (double)L / (c * most);
        if (b <= busy) continue;
        // planes per thread: 4 with up to 512 threads, 3 with up to 640, 2 with up to 896
        for (int z = std::min(4, most); z >= 1; --z) {
            const int zt = (most + z - 1) / z, threads = (per * zt + 31) / 32 * 32;
            if (threads > (z == 4 ? 512 : z == 3 ? 640 : 896)) continue;
            busy = b;
            best = SlabShape{c, zt, z, threads, smem};
            break;
        }
    }
    return best;
}

template <int kZ, int kT>
t3d_status launch_slab_k(const ItemDesc& d, const ColumnProgram& pr, const SlabShape& c, int kind,
                         const ColumnView& sv, const ColumnView& ev, int e_store, cudaStream_t st)
{
    auto kernel = k_slab<kZ, kT>;
    T3D_TRY(allow_dynamic_smem((const void*)kernel, c.smem));
    const int64_t words = d.nw ? d.nw : d.W;
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(c.cluster * std::min<int64_t>(words, 0x7fffffffLL / c.cluster)));
    cfg.blockDim = dim3((unsigned)c.threads);
    cfg.dynamicSmemBytes = c.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)c.cluster;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    ProfScope prof(kind, st);
    T3D_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kernel, d, pr, c.cluster, sv, ev, e_store));
    return T3D_OK;
}

// A word's column is strided by the row length, so a block reads 32-byte sectors for 8-byte words.
// From kTurnWords words on the syndrome is turned into contiguous columns first (in the item's
// scratch array), the gathered flips are written as columns into the syndrome's own array, and both
// are turned back.
constexpr int64_t kTurnWords = 64;

t3d_status launch_slab(const ItemDesc& d, ColumnProgram pr, int kind, cudaStream_t st)
{
    const SlabShape c = slab_shape(d.lat.L);
    pr.zt = c.zt;
    const int64_t R = 3LL * d.lat.L3;
    const bool turn = d.tmp && !d.live && !d.nw && d.W >= kTurnWords && (d.W + kTurn - 1) / kTurn <= 65535;
    ColumnView sv{d.s, d.W, 1}, ev{d.e, d.W, 1};
    const dim3 grid((unsigned)((R + kTurn - 1) / kTurn), (unsigned)((d.W + kTurn - 1) / kTurn));
    if (turn) {
        sv = ColumnView{d.tmp, 1, R};
        ev = ColumnView{d.s, 1, R};
        ProfScope prof(kind, st);
        k_to_columns<<<grid, 256, 0, st>>>(R, d.W, d.s, d.tmp);
        T3D_LAUNCH_CHECK("syndrome columns");
    }
    if (c.z == 4)
        T3D_TRY((launch_slab_k<4, 512>(d, pr, c, kind, sv, ev, turn, st)));
    else if (c.z == 3)
        T3D_TRY((launch_slab_k<3, 640>(d, pr, c, kind, sv, ev, turn, st)));
    else
        T3D_TRY((launch_slab_k<2, 896>(d, pr, c, kind, sv, ev, turn, st)));
    if (turn) {
        ProfScope prof(kind, st);
        k_from_columns<true><<<grid, 256, 0, st>>>(R, d.W, d.s, d.e);
        T3D_LAUNCH_CHECK("flips into the error state");
        k_from_columns<false><<<grid, 256, 0, st>>>(R, d.W, d.tmp, d.s);
        T3D_LAUNCH_CHECK("syndrome rows");
    }
    return T3D_OK;
}

size_t column_bytes(int L) { return (size_t)L * L * L * 72; }

// Words per block and z-parts.  A block should have at least two warps, so tiny lattices take
// several words.  A lattice that fits a block with a thread per site takes one (k_column_one); a larger
// lattice's columns are split into as many z-parts as keep about kColumnTarget threads resident on an SM
// (all the blocks that fit its shared memory together).
constexpr int kColumnTarget = 1024;

struct ColumnShape {
    int wt, zt, threads;
    size_t smem;
};

ColumnShape column_shape(int L, int64_t words)
{
    ColumnShape c;
    c.wt = 1;
    while (L * L * L * c.wt < 64 && c.wt < words) c.wt *= 2;
    c.smem = column_bytes(L) * c.wt;
    const int plane = L * L * c.wt;
    const int64_t columns = (words + c.wt - 1) / c.wt;
    const int fit = (int)std::max<size_t>(1, std::min<size_t>(32, kColumnSmem / (c.smem + 1024)));
    const int per_sm = (int)std::min<int64_t>(fit, std::max<int64_t>(1, (columns + 151) / 152));
    c.zt = plane * L <= kColumnThreads ? L : 1;
    for (int z = 2; z < L; ++z)
        if (c.zt < L && plane * z <= kColumnThreads && plane * z * per_sm <= kColumnTarget) c.zt = z;
    c.threads = (plane * c.zt + 31) / 32 * 32;
    return c;
}

template <bool kRun>
t3d_status launch_column(const ItemDesc& item, ColumnProgram pr, int kind, cudaStream_t st)
{
    ItemDesc d = item;
    const int64_t words = d.nw ? d.nw : d.W;
    const ColumnShape c = column_shape(d.lat.L, words);
    d.tx = c.wt;
    pr.zt = c.zt;
    auto kernel = c.zt == d.lat.L ? k_column_one<kRun> : k_column<kRun>;
    T3D_TRY(allow_dynamic_smem((const void*)kernel, c.smem));
    ProfScope prof(kind, st);
    kernel<<<persistent_grid((const void*)kernel, c.threads, kind, (words + c.wt - 1) / c.wt, false, c.smem),
             c.threads, c.smem, st>>>(d, pr);
    T3D_LAUNCH_CHECK("on-chip column");
    return T3D_OK;
}

uint64_t schedule_bits(const char* schedule, int slen)
{
    uint64_t b = 0;
    for (int i = 0; i < slen; ++i)
        if (schedule[i] == 'P') b |= 1ULL << i;
    return b;
}

// ------------------------------------------------------------------ which form runs
// A schedule runs on chip (one launch per lattice, its columns in and out once, an application between
// two barriers) or step by step (one launch per application over all lattices of a batch, every word
// through L2 or HBM).  Which is faster depends on the lattice, the words, the letters and what else is in
// the batch, so both are estimated, in microseconds.  The constants are fitted to both forms' times at L = 3
// .. 32, 1 .. 1,563 words and the schedules F, FF, 8 F, P, 5 P and FFPFF (1,440 sizes; rms of the estimates 10%
// on chip, 7% step by step).  The form they choose takes 0.25% longer than the faster of the two on
// average, where step by step always takes 35% longer and on chip up to L = 14, below 64 words or from five
// applications on 13%.  Examples, step by
// step / on chip: FFPFF at L = 8, 1,563 words 87 / 50; L = 25, 1,563 words 2,605 / 3,573; L = 32, 1,563 words 5,459 /
// 5,166, 16 words 189 / 96; P alone at L = 16, 16 words 6 / 35; F alone at L = 28, 48 words 48 / 80.
constexpr double kSms = 152.0;
constexpr double kL2Msites = 1.5;     // millions of sites x words whose arrays stay in L2
constexpr int64_t kClearTypical = 8;  // flip until clear: applications that do some work
constexpr double kSkipUs = 2.0;       // ... and what a skipped one costs as a launch
constexpr double kClearUs = 7.0;      // ... and its flags

struct Letters {
    int64_t flips, pflips;
};

// The work of a single on-chip launch: rounds of columns and ns-weighted sites per round.
struct ChipShape {
    double rounds, ksites;   // columns (clusters' words) one SM takes in turn; thousands of sites of a block
    double io, flip, pflip;  // us per thousand sites: columns in and out, one application of each kind
    double each;             // us per application beside that (the cluster's barriers)
};

bool chip_shape(int L, int64_t words, ChipShape& c)
{
    if (column_bytes(L) <= kColumnSmem) {
        const int wt = column_shape(L, words).wt;
        c.rounds = std::ceil(std::ceil((double)words / wt) / kSms);
        c.ksites = 1e-3 * L * L * L * wt;
        c.each = 0.0;
        if (L * L * L <= kColumnThreads) {   // k_column_one
            c.io = 5.0; c.flip = 0.82; c.pflip = 2.05;
        } else {                             // k_column
            c.io = c.rounds > 1.0 ? 4.6 : 6.0; c.flip = 1.23; c.pflip = 2.5;
        }
    } else {
        const SlabShape s = slab_shape(L);
        if (s.cluster == 0) return false;
        c.rounds = std::ceil((double)words / (kResident[s.cluster] / s.cluster));
        c.ksites = 1e-3 * L * L * ((L + s.cluster - 1) / s.cluster);
        // turned columns are cheap while their four arrays stay in L2
        c.io = words < kTurnWords ? 5.0 : (kL2Msites > 1e-6 * L * L * L * (double)words ? 4.4 : 5.6);
        c.flip = 0.8; c.pflip = 1.9;
        c.each = 1.0;
    }
    // a row's words share 32-byte sectors, which the column of every word fetches for itself
    c.io *= std::min(1.0, 0.2 * (double)words);
    return true;
}

constexpr double kLaunchUs = 2.8;

double chip_us(const ChipShape& c, const Letters& n)
{
    const double flip = std::max(0.2, c.rounds * (c.each + c.flip * c.ksites)),
                 pflip = std::max(0.3, c.rounds * (c.each + c.pflip * c.ksites));
    return kLaunchUs + c.rounds * c.io * c.ksites + n.flips * flip + n.pflips * pflip;
}

// Whole runs on chip: a column draws a cycle's noise and measurement on one SM, 12 ns a site (at least
// 3.5 us a cycle), where the noise and measurement kernels spread them over the chip.
double chip_run_us(const ChipShape& c, int cycles, const Letters& n, int perfect)
{
    const Letters all{cycles * n.flips + std::min<int64_t>(std::max(perfect, 0), kClearTypical), cycles * n.pflips};
    return chip_us(c, all) + cycles * std::max(3.5, 12.0 * c.rounds * c.ksites) +
           (perfect >= 0 ? 2.5 * c.rounds * c.ksites : 0.0);
}

int64_t item_words(const ItemDesc& d)
{
    // compacted words: the device knows how many there are, usually few
    return d.live ? std::min<int64_t>(d.W, 16) : (d.nw ? d.nw : d.W);
}

// The step by step form over the items i of tab with !skip[i]: an application's launch takes a
// latency that grows with L (the flip's walk along y) beside the blocks' work; an odd number of flips
// leaves the syndrome in the scratch array and is copied back row by row.
double steps_us(const ItemTable& tab, const bool* skip, const Letters& n, bool until_clear)
{
    int items = 0, maxL = 0;
    bool wide = true;
    for (int i = 0; i < tab.n; ++i)
        if (!skip[i]) {
            ++items;
            maxL = std::max(maxL, tab.it[i].lat.L);
            wide = wide && tab.it[i].lat.L >= 32;
        }
    if (items == 0) return 0.0;
    double work = 0.0, longest = 0.0, blocks = 0.0, waves = 0.0, msites = 0.0, copies = 0.0;
    for (int i = 0; i < tab.n; ++i) {
        if (skip[i]) continue;
        const int L = tab.it[i].lat.L;
        const int64_t words = item_words(tab.it[i]);
        const double m = 1e-6 * L * L * L * (double)words;
        const int wt = flip_tile_words(L, words, wide);
        const double us = 2.5e-3 * L * L * wt, b = L * std::ceil((double)words / wt);
        longest = std::max(longest, us);
        work += us * b / kSms;
        waves += us * std::ceil(b / kSms);
        blocks += b;
        msites += m;
        // below 65,536 rows the copy takes a time per row
        copies += 1.1 + (L < 28 ? std::max(1.6e-3 * L * L * L, 24.0 * m) : std::max(0.55e-3 * L * L * L, 13.0 * m));
    }
    const double turns = items == 1 ? waves : (blocks <= kSms ? longest : work + 0.5 * longest);
    const double flip = std::hypot(1.7 + 0.54 * maxL, turns);
    const double pflip = 3.7 + (msites < kL2Msites ? 20.0 : 26.0 + 0.5 * std::max(0, maxL - 24)) * msites;
    double us = 0.8 + n.pflips * pflip + (n.flips & 1 ? copies : 0.0);
    if (until_clear) {
        const int64_t run = std::min(n.flips, kClearTypical);
        us += run * flip + (double)(n.flips - run) * kSkipUs + items * kClearUs;
    } else {
        us += n.flips * flip;
    }
    return us;
}

// The fastest of: all items step by step, every item that fits on chip, or those whose time on chip is
// below what they add to the shared launches.  chip[i] says which; returns the estimate.
double route_schedule(const ItemTable& tab, const bool* skip, const Letters& n, bool until_clear, bool* chip)
{
    const Letters work{until_clear ? std::min(n.flips, kClearTypical) : n.flips, n.pflips};
    double on[kMaxItems];
    bool fits[kMaxItems], none[kMaxItems], all[kMaxItems], some[kMaxItems];
    double us_all = 0.0;
    for (int i = 0; i < tab.n; ++i) {
        ChipShape c;
        fits[i] = !skip[i] && chip_shape(tab.it[i].lat.L, item_words(tab.it[i]), c);
        on[i] = fits[i] ? chip_us(c, work) : 0.0;
        none[i] = skip[i];
        all[i] = skip[i] || fits[i];
        us_all += on[i];
    }
    const double us_none = steps_us(tab, none, n, until_clear);
    us_all += steps_us(tab, all, n, until_clear);
    double us_some = 0.0;
    for (int i = 0; i < tab.n; ++i) some[i] = none[i];
    for (int i = 0; i < tab.n; ++i) {
        if (!fits[i]) continue;
        none[i] = true;   // without this item
        const bool pays = on[i] < us_none - steps_us(tab, none, n, until_clear);
        none[i] = skip[i];
        some[i] = pays;
        us_some += pays ? on[i] : 0.0;
    }
    us_some += steps_us(tab, some, n, until_clear);
    const bool* best = us_all <= us_none && us_all <= us_some ? all : (us_some < us_none ? some : none);
    for (int i = 0; i < tab.n; ++i) chip[i] = fits[i] && best[i];
    return std::min(us_all, std::min(us_none, us_some));
}

// A run's cycles step by step, its schedules in whichever form is faster.
double step_run_us(const ItemTable& tab, const bool* skip, int cycles, const Letters& n, int perfect)
{
    double msites = 0.0;
    int items = 0;
    for (int i = 0; i < tab.n; ++i)
        if (!skip[i]) {
            const double L = tab.it[i].lat.L;
            msites += 1e-6 * L * L * L * (double)tab.it[i].W;
            ++items;
        }
    if (items == 0) return 0.0;
    bool chip[kMaxItems];
    double us = cycles * (5.5 + 75.0 * msites);
    if (n.flips + n.pflips > 0) us += cycles * route_schedule(tab, skip, n, false, chip);
    if (perfect >= 0) us += 3.0 + 20.0 * msites;
    if (perfect > 0) us += route_schedule(tab, skip, Letters{perfect, 0}, true, chip);
    return us;
}

Letters letters_of(const char* schedule, int slen, int n_apply)
{
    Letters n{0, 0};
    for (int k = 0; k < slen; ++k) {
        const int times = n_apply / slen + (k < n_apply % slen ? 1 : 0);
        (schedule[k] == 'P' ? n.pflips : n.flips) += times;
    }
    return n;
}

}  // namespace

void route_sweeps(const ItemTable& tab, const char* schedule, int slen, int n_apply, bool until_clear, bool* chip)
{
    const bool skip[kMaxItems] = {};
    route_schedule(tab, skip, letters_of(schedule, slen, n_apply), until_clear, chip);
}

void route_run(const ItemTable& tab, int cycles, const char* schedule, int slen, int n_apply, int perfect, bool* whole)
{
    const Letters n = letters_of(schedule, slen, n_apply);
    double on[kMaxItems];
    bool fits[kMaxItems], some[kMaxItems];
    const bool none[kMaxItems] = {};
    double us_all = 0.0;
    for (int i = 0; i < tab.n; ++i) {
        const int L = tab.it[i].lat.L;
        ChipShape c;
        fits[i] = column_bytes(L) <= kColumnSmem && chip_shape(L, tab.it[i].W, c);
        on[i] = fits[i] ? chip_run_us(c, cycles, n, perfect) : 0.0;
        us_all += on[i];
    }
    const double us_none = step_run_us(tab, none, cycles, n, perfect);
    us_all += step_run_us(tab, fits, cycles, n, perfect);
    double us_some = 0.0;
    bool without[kMaxItems] = {};
    for (int i = 0; i < tab.n; ++i) {
        some[i] = false;
        if (!fits[i]) continue;
        without[i] = true;
        some[i] = on[i] < us_none - step_run_us(tab, without, cycles, n, perfect);
        without[i] = false;
        us_some += some[i] ? on[i] : 0.0;
    }
    us_some += step_run_us(tab, some, cycles, n, perfect);
    const bool* best = us_all <= us_none && us_all <= us_some ? fits : (us_some < us_none ? some : none);
    for (int i = 0; i < tab.n; ++i) whole[i] = best[i];
}

t3d_status launch_column_sweeps(const ItemDesc& d, const char* schedule, int slen, int n_apply, uint32_t sweep0,
                                uint64_t seed, uint32_t cycle, cudaStream_t st)
{
    ColumnProgram pr;
    std::memset(&pr, 0, sizeof(pr));
    pr.seed = seed;
    pr.sched = schedule_bits(schedule, slen);
    pr.slen = slen;
    pr.n_apply = n_apply;
    pr.sweep0 = sweep0;
    pr.cycle0 = cycle;
    const int kind = pr.sched ? T3D_K_PFLIP : T3D_K_FLIP;
    return column_bytes(d.lat.L) <= kColumnSmem ? launch_column<false>(d, pr, kind, st) : launch_slab(d, pr, kind, st);
}

t3d_status launch_column_until_clear(const ItemDesc& d, int max_sweeps, int32_t* sweeps_done, cudaStream_t st)
{
    if (sweeps_done) T3D_CUDA_CHECK(cudaMemsetAsync(sweeps_done, 0, sizeof(int32_t), st));
    ColumnProgram pr;
    std::memset(&pr, 0, sizeof(pr));
    pr.slen = 1;
    pr.n_apply = max_sweeps;
    pr.until_clear = 1;
    pr.sweeps_done = sweeps_done;
    return column_bytes(d.lat.L) <= kColumnSmem ? launch_column<false>(d, pr, T3D_K_FLIP, st) : launch_slab(d, pr, T3D_K_FLIP, st);
}

t3d_status launch_column_run(const ItemDesc& d, int cycles, uint32_t cycle0, uint64_t thr_p, uint64_t thr_q,
                             uint64_t seed, const char* schedule, int slen, int n_apply, int perfect, cudaStream_t st)
{
    ColumnProgram pr;
    std::memset(&pr, 0, sizeof(pr));
    pr.seed = seed;
    pr.sched = schedule_bits(schedule, slen);
    pr.slen = slen;
    pr.n_apply = n_apply;
    pr.thr_p = thr_p;
    pr.thr_q = thr_q;
    pr.cycle0 = cycle0;
    pr.cycles = cycles;
    pr.perfect = perfect;
    return launch_column<true>(d, pr, T3D_K_FLIP, st);
}

}  // namespace t3d
