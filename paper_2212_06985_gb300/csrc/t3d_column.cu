// Lattices whose syndrome and flip words fit one SM: a block keeps the whole lattice of one (or
// a few) 64-sample words in shared memory and runs a schedule of flip / p-flip applications
// -- or a whole Monte Carlo run, noise and measurement included -- without going back to global
// memory and without a launch per step.
//
// Samples are independent, so a word's column of the bit-sliced arrays never needs another
// column: what separates two applications is a barrier of one block instead of a kernel
// boundary.  At L <= 16 the syndrome and the flip words (48 bytes per site and word, 196,608
// bytes at L = 16) fit the 227 KB a block can have; at L <= 14 the error words fit as well
// (72 bytes), above that they stay in global memory.
//
// An application is two phases between barriers: every site decides its own three edges from
// the old syndrome (7 shared reads: the z-neighbour's words are the thread's previous ones)
// and writes the flip words; then every site's three faces take the flips of their edges (7
// shared reads, again the z-neighbour's kept in registers).  Each edge is decided once, where
// the one-pass kernel for larger lattices decides nine edges per site.
//
// Thread (xy, word) of z-part zp walks the sites z0 <= z < z1 of one lattice column, so its x
// and y neighbour offsets are fixed for the whole kernel, and a column of random words shares
// the generator's first rounds (PhiloxColumn).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

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

// kRun: whole runs (sweeps otherwise); kESmem: the error words are in shared memory as well.
template <bool kRun, bool kESmem>
__global__ void __launch_bounds__(kColumnThreads, 1)
k_column(const __grid_constant__ ItemDesc d, const __grid_constant__ ColumnProgram pr)
{
    extern __shared__ uint64_t sm[];
    const int L = d.lat.L, L2 = d.lat.L2, L3 = d.lat.L3, Wt = d.tx;
    const int P = L2 * Wt, N = L3 * Wt;   // a z-plane, the lattice
    uint64_t* const S0 = sm;
    uint64_t* const F0 = sm + 3 * N;
    uint64_t* const E0 = sm + 6 * N;      // kESmem

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
                    const int site = z * L2 + xy;
                    if (prob) {
                        const PhiloxSite ps = philox_site(pc, (uint32_t)site);
                        const U32x4 a = philox_finish(pc, ps, b0), b = philox_finish(pc, ps, b1);
                        f[0] |= exactly_two(s2, s2y, s1, s1m) & ((uint64_t)a.v[0] | ((uint64_t)a.v[1] << 32));
                        f[1] |= exactly_two(s2, s2x, s0, s0m) & ((uint64_t)a.v[2] | ((uint64_t)a.v[3] << 32));
                        f[2] |= exactly_two(s1, s1x, s0, s0y) & ((uint64_t)b.v[0] | ((uint64_t)b.v[1] << 32));
                    }
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        F0[k * N + i] = f[k];
                        if (kESmem) {
                            if (f[k]) E0[k * N + i] ^= f[k];
                        } else {
                            xor_into(&e.at(k * L3 + site), f[k]);
                        }
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
                    if (kESmem) E0[n * N + i] = 0;
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
                    if (kESmem) xor_into(&e.at(n * L3 + z * L2 + xy), E0[n * N + i]);
                }
            }
        } else {
            // the error word of edge (k, site z, xy)
            auto E = [&](int k, int z, int i) -> uint64_t& {
                if (kESmem) return E0[k * N + i];
                return e.at(k * L3 + z * L2 + xy);
            };
            if (kESmem)
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
                        if (f) E(k, z, i) ^= f;
                    }
            };
            auto measure = [&](uint64_t thr, uint32_t cycle) {
                const bool all = thr >> 32, none = thr == 0;
                const BernoulliColumn bc = bernoulli_column(pr.seed, kStreamMeas, cycle, group);
                // row offsets of the neighbours in global memory (sites) and in shared memory
                const int gx = kESmem ? xp : (x + 1 == L ? 1 - L : 1), gy = kESmem ? yp : (y + 1 == L ? L - L2 : L);
                for (int z = zb, i = zb * P + u; z < ze; ++z, i += P) {
                    const int gz = (z + 1 == L ? 1 - L : 1) * (kESmem ? P : L2);
                    const int site = z * L2 + xy;
                    uint64_t ex, ey, ez, exy, exz, eyx, eyz, ezx, ezy;
                    if (kESmem) {
                        const uint64_t *px = E0 + i, *py = px + N, *pz = py + N;
                        ex = px[0], exy = px[gy], exz = px[gz];
                        ey = py[0], eyx = py[gx], eyz = py[gz];
                        ez = pz[0], ezx = pz[gx], ezy = pz[gy];
                    } else {
                        ex = e.at(site), exy = e.at(site + gy), exz = e.at(site + gz);
                        ey = e.at(L3 + site), eyx = e.at(L3 + site + gx), eyz = e.at(L3 + site + gz);
                        ez = e.at(2 * L3 + site), ezx = e.at(2 * L3 + site + gx), ezy = e.at(2 * L3 + site + gy);
                    }
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
            if (kESmem)
                for (int z = zb, i = zb * P + u; z < ze; ++z, i += P)
#pragma unroll
                    for (int k = 0; k < 3; ++k) e.at(k * L3 + z * L2 + xy) = E0[k * N + i];
        }
        __syncthreads();   // the next column overwrites the words
    }
}

size_t column_bytes(int L, bool e_smem) { return (size_t)L * L * L * (e_smem ? 72 : 48); }

bool e_fits(int L) { return column_bytes(L, true) <= kColumnSmem; }

// Words per block and z-parts.  A block should have at least two warps, so tiny lattices take
// several words; a lattice column is split into as many z-parts as keep about kColumnTarget
// threads resident on an SM (all the blocks that fit its shared memory together), or, when
// there are fewer columns than that, into one part per site.
constexpr int kColumnTarget = 1024;

struct ColumnShape {
    int wt, zt, threads;
    size_t smem;
};

ColumnShape column_shape(int L, int64_t words)
{
    ColumnShape c;
    const bool es = e_fits(L);
    c.wt = 1;
    while (L * L * L * c.wt < 64 && c.wt < words) c.wt *= 2;
    c.smem = column_bytes(L, es) * c.wt;
    const int plane = L * L * c.wt;
    const int64_t columns = (words + c.wt - 1) / c.wt;
    const int fit = (int)std::max<size_t>(1, std::min<size_t>(32, kColumnSmem / (c.smem + 1024)));
    const int per_sm = (int)std::min<int64_t>(fit, std::max<int64_t>(1, (columns + 151) / 152));
    c.zt = 1;
    for (int z = 2; z <= L; ++z)
        if (plane * z <= kColumnThreads && plane * z * per_sm <= kColumnTarget) c.zt = z;
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
    const bool es = e_fits(d.lat.L);
    auto kernel = es ? k_column<kRun, true> : k_column<kRun, false>;
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

}  // namespace

bool column_fits(int L) { return column_bytes(L, false) <= kColumnSmem; }

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
    return launch_column<false>(d, pr, pr.sched ? T3D_K_PFLIP : T3D_K_FLIP, st);
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
    return launch_column<false>(d, pr, T3D_K_FLIP, st);
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
