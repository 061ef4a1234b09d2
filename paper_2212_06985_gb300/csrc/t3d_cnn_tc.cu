// The learned pre-decoder's convolutions on the fifth-generation tensor cores
// (tcgen05 MMA with TMEM accumulators, operands staged in shared memory): the
// inference forward pass, and for training the forward pass with the loss and
// the backward-data passes (the same kernel with another epilogue).
//
// Each 3x3x3 convolution (16 output channels) is a sum of GEMMs over the input
// sites: for an input site i and every output site o within one step of it,
//   D_o[sample][co] += A_i[sample][ci] . W(i - o)[co][ci],   M = 128, K = 16,
// where A_i is the 128-sample activation tile of site i.  A tcgen05.mma with
// M = 128, K = 16 takes about as long for N = 16 as for N = 64 (the issue
// floor, about 53 cycles; N = 128 takes 64 and N = 256 128, the bf16 peak), so
// one MMA serves every output of a work unit that an input tile reaches: its N
// stacks those outputs' weight blocks (the column kernel below).
//
// Work unit: one 128-sample tile x one 2 x 2 column of output sites running
// through all L planes in z.  The CTA streams the unit's input planes
// z = -1 .. L, each the 4 x 4 input sites around the column (periodic wrap);
// each input tile reaches shared memory once and is multiplied, by one MMA,
// into every column site of the three output planes it touches.  TMEM keeps a
// ring of eight output planes; the epilogue drains a plane once its last
// input plane has been multiplied.
//
// Warp roles (one CTA per SM; each role is warp-uniform code, one elected lane
// issues):
//   warps 0-7  epilogue, in two groups of four that take the output planes in
//              turn: tcgen05.ld of a finished plane (warp w reads TMEM lanes
//              32 (w % 4) .. = samples), then by mode (TcMode): bias + ReLU +
//              BF16 store of the next layer's input; the 16 -> 3 head and the
//              hard decisions; the head with the BCE gradient, the head's
//              gradients and the gradient at the pre-activation; or the
//              backward-data gradient gated by the forward activation;
//   producers  bulk copies of a plane's four rows of four tiles (one copy a row,
//              four where the row wraps) into a ring of shared-memory slots;
//   issuer     the MMAs; commits their completion to the slot's "empty" barrier
//              and to the output plane's "accumulators full" barrier.
// Every wait is bounded (one second; toric3d_cnn_debug_wait_limit shortens the
// waits that may give up, so a test can make them run out); a wait that gives
// up sets the device error flag and the CTA winds down (waiting, again bounded
// but always by the full second, for its copies and MMAs in flight, and
// freeing its TMEM) so the context stays usable.
//
// Shared-memory operand layout ("no swizzle", K-major): core matrices of 8 rows
// x 16 bytes stored contiguously.  Hidden activations in global memory use the
// same layout, [channel/8][128 samples][8 channels] BF16 per tile, and the tile
// of (site, 128-sample tile m) starts at byte (m L^3 + site) 4096, so a tile is
// one contiguous 4 KiB block (K-direction core-matrix stride (LBO) 2 KiB,
// M-direction stride (SBO) 128 B) and a warp of the epilogue writes 512-byte
// runs.  The first layer's input tile (6 of 8 channels used: s_{t-1} then s_t of
// the three faces) is [sample][8], 2 KiB (SBO 128 B); two x-adjacent sites form
// one K = 16 operand as its two K chunks (LBO 2 KiB).  Weight blocks:
// [co/8][ci/8][co%8][ci%8] (512 B, LBO 128 B, SBO 256 B).  The weight gradients
// read the same tiles with samples as K (k_wgrad_tc).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "t3d_cnn.cuh"
#include "t3d_device.cuh"
#include "t3d_host.hpp"

namespace t3d {
namespace cnn {
namespace {

constexpr int kTileM = 128;                         // samples per tile (MMA M)
constexpr uint32_t kTmemCols = 512;
constexpr int kSlotBytes = 4096;                    // one hidden-layer tile
constexpr int kEpiWarps = 4;
constexpr int kProducerWarp = 4;
constexpr int kIssuerWarp = 5;
constexpr int kTcThreads = 32 * (kIssuerWarp + 1);
constexpr uint64_t kWaitNs = 1000000000ull;         // bound of every wait

__device__ unsigned int g_tc_error;   // bit 0: a bounded wait gave up
// bound of the waits that may give up (the wind-down drains always use kWaitNs)
__device__ unsigned long long g_tc_wait_ns = kWaitNs;

// What the epilogue makes of a finished output plane.
enum TcMode {
    kTcRelu = 0,        // bias + ReLU, BF16 activations for the next layer
    kTcHead = 1,        // bias + ReLU, the 16 -> 3 head, hard decisions (and optional logits)
    kTcHeadTrain = 2,   // training: the head, the BCE gradient against the labels, the head's
                        // gradients and the loss, and the gradient at the layer's pre-activation
    kTcMask = 3,        // backward data: the gradient gated by the forward activation's sign
};
__host__ __device__ constexpr bool tc_head(int mode) { return mode == kTcHead || mode == kTcHeadTrain; }

struct TcArgs {
    int L, L3;
    int64_t Sp;                 // padded samples of the activation buffers (multiple of 128)
    int64_t n_samples;
    int64_t W;                  // row stride of the bit-sliced arrays (words)
    int64_t words;              // words of this pass
    int ncx;                    // 2 x 2 columns per axis (ceil(L / 2))
    int64_t n_units;
    const uint8_t* in;          // input activations
    uint8_t* out;               // output activations / gradients (all modes but kTcHead)
    const __nv_bfloat16* w;     // [27][co][ci]
    const float* bias;          // [16]
    const float* w4;            // head [3][16]
    const float* b4;            // [3]
    uint32_t* dec32;            // kTcHead: decision words [word][site][8] 32-bit halves
    float* logits;              // kTcHead: optional [3][L^3][n_samples]
    const uint64_t* label;      // kTcHeadTrain: bit-sliced labels [3][L^3][W]
    float inv_n;                // kTcHeadTrain: 1 / (3 L^3 n_samples)
    float* grad_w4;             // kTcHeadTrain: [3][16], accumulated
    float* grad_b4;             // kTcHeadTrain: [3], accumulated
    float* loss;                // kTcHeadTrain: [1], accumulated
    const uint8_t* mask_act;    // kTcMask: the forward activation at the output sites
};

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Whether the phase of the given parity is complete, without waiting.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase of the given parity.  Gives up after
// g_tc_wait_ns, or early once another role of the CTA has given up (abort
// flag), unless ignore_abort (the final drain of work in flight, bounded by
// kWaitNs whatever the debug limit).
__device__ bool wait_bar(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, bool ignore_abort = false)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    const uint64_t limit = ignore_abort ? kWaitNs : *(volatile unsigned long long*)&g_tc_wait_ns;
    for (;;) {
        for (int i = 0; i < 32; ++i)
            if (mbar_try_wait(bar, parity)) return true;
        if (!ignore_abort && *abort_flag) return false;
        if (global_ns() - t0 > limit) {
            *abort_flag = 1;
            atomicOr(&g_tc_error, 1u);
            return false;
        }
    }
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Ask for [src, src + bytes) in L2 (16-byte aligned, a multiple of 16 bytes).
__device__ __forceinline__ void bulk_prefetch(const void* src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_before()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_after()
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Whole warp: allocate ncols TMEM columns; the base address goes to smem.
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// Shared-memory matrix descriptor: start, leading (K) and stride (M/N) byte
// offsets, descriptor version 1 (bit 46), no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           (1ull << 46);
}

// D += A . B^T with the instruction descriptor of this MMA (N varies).
__device__ __forceinline__ void mma_bf16_n(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc)
{
    asm volatile(
        "{\n"
        ".reg .pred pa;\n"
        "setp.ne.b32 pa, 1, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, pa;\n"
        "}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc)
        : "memory");
}

// D = A . B^T, not accumulating (the first MMA into an accumulator).
__device__ __forceinline__ void mma_bf16_overwrite(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc)
{
    asm volatile(
        "{\n"
        ".reg .pred pa;\n"
        "setp.ne.b32 pa, 0, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, pa;\n"
        "}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc)
        : "memory");
}

// Warp: zero 32 TMEM lanes x 16 consecutive 32-bit columns (one lane per thread).
__device__ __forceinline__ void tmem_zero16(uint32_t taddr)
{
    const uint32_t z = 0;
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};\n" ::"r"(taddr),
        "r"(z)
        : "memory");
}

__device__ __forceinline__ void tmem_wait_st()
{
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// One lane of a converged warp (always the same one).
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "elect.sync _|q, 0xffffffff;\n"
        "selp.u32 %0, 1, 0, q;\n"
        "}\n"
        : "=r"(p));
    return p != 0;
}

// Arrive on the barrier once every MMA this thread issued so far has completed.
__device__ __forceinline__ void mma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// Warp: 32 TMEM lanes x 16 consecutive 32-bit columns, one lane per thread
// (asynchronous: the registers are valid after tmem_wait_ld).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void tmem_wait_ld()
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Four floats of shared memory (volatile: loaded where they are used, not kept in registers).
__device__ __forceinline__ void lds4(uint32_t addr, float (&v)[4])
{
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(addr));
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// ------------------------------------------------------------------ schedule
struct Unit {
    int64_t m0;      // first sample of the tile
    int x0, y;       // column origin (even)
};

// v in [-L, 2L): periodic coordinate
__device__ __forceinline__ int wrap(int v, int L)
{
    return v < 0 ? v + L : (v >= L ? v - L : v);
}

// Activation layout: the tile of (site, 128-sample tile m) starts at byte
// (m L^3 + site) tile_bytes, so a tile is contiguous and so are the tiles of
// x-adjacent sites of one row (bulk copies of whole runs of a row move more
// bytes per clock than one copy per tile).
__device__ __forceinline__ int64_t tile_off(int64_t site, int64_t m0, int L3, uint32_t tile_bytes)
{
    return ((m0 >> 7) * L3 + site) * (int64_t)tile_bytes;
}

// ------------------------------------------------------------------ column kernel
// The convolution with dense operands: a work unit is one 128-sample tile x one
// 2 x 2 column of output sites (x0, x0 + 1) x (y0, y0 + 1) run through all L
// planes in z.  Every input site (xi, yi) of an input plane zi with
// xi = x0 - 1 .. x0 + 2, yi = y0 - 1 .. y0 + 2 feeds the column sites within
// one step of it in x and y, in the three output planes zi - 1, zi, zi + 1;
// TMEM keeps eight output planes of 64 columns (4 sites x 16 channels, site
// j = jx + 2 jy) in a ring, so one MMA covers the input tile's whole reach:
// the columns from (plane zi - 1, its lowest site lo) to (plane zi + 1, its
// highest site hi), N = 16 (4 (P2 - P1) + hi - lo + 1) for the planes P1..P2
// that exist (N = 192 for the four inner sites).  Its B operand is a window of
// one per-position sequence of weight blocks [plane zi - 1: sites lo..3 |
// plane zi: 0..3 | plane zi + 1: 0..hi], W(xi - xo, yi - yo, zi - zo) or zero
// where the site is out of reach; of the blocks multiplied 64% are non-zero
// (108 of 168 per plane).  A window that would cross
// the ring's end is split in two MMAs.  TMEM columns are zeroed by the
// epilogue after it drains a plane (and once at the start), so every MMA
// accumulates.  The first layer pairs x-adjacent input sites in one K = 16
// operand (chunk c = site 2p - 1 + c of the row; LBO 2 KiB steps to the second site).
// Input ring of 128 KiB: two planes of 16 x 4 KiB tiles (hidden layers) or four of 16 x 2 KiB
// (first layer).
constexpr int kColRingBytes = 32 * kSlotBytes;
__host__ __device__ constexpr int col_in_slots(bool bits_in) { return bits_in ? 4 : 2; }
constexpr int kColInMax = 4;
constexpr int kColSlots = 8;                              // output planes resident in TMEM
constexpr int kColPlaneCols = 4 * kC;                     // 64
constexpr int kColWBlocks = 168;                          // windows of the 16 positions (hidden layers)
constexpr int kColOffW = kColRingBytes;
constexpr int kColOffBar = kColOffW + kColWBlocks * 512;
constexpr int kColNumBars = 2 * kColInMax + 2 * kColSlots + 1;   // full, empty, acc_full, acc_empty, done
constexpr int kColOffMisc = kColOffBar + kColNumBars * 8;
constexpr int kColOffPos = kColOffMisc + 16;              // ColPos[16]
constexpr int kColOffHead = kColOffPos + 16 * 12 + 8;     // training's head: w4 [3][16], bias [16]
constexpr int kColSmemBytes = kColOffHead + 4 * kC * 4 + 1024;
static_assert(kColOffHead % 16 == 0, "16-byte loads");
static_assert(kColSmemBytes <= 227 * 1024, "shared memory budget");
static_assert(kColSlots * kColPlaneCols == 512, "TMEM ring");

// Operand position p of a row (hidden: the site x0 - 1 + p; first layer: the
// pair x0 - 1 + 2p, x0 + 2p) at row b (yi = y0 - 1 + b): the column sites in
// reach span lo..hi, and its weight sequence starts at block base.
struct ColPos {
    int base, lo, hi;
};

__host__ __device__ constexpr int col_chunk_dx(bool bits_in, int p, int c) { return bits_in ? 2 * p - 1 + c : p - 1; }

__host__ __device__ constexpr bool col_reach(bool bits_in, int p, int jx)
{
    for (int c = 0; c < 2; ++c) {
        const int dx = col_chunk_dx(bits_in, p, c) - jx;
        if (dx >= -1 && dx <= 1) return true;
    }
    return false;
}

__host__ __device__ constexpr ColPos col_pos(bool bits_in, int p, int b)
{
    const int P = bits_in ? 2 : 4;
    int base = 0;
    ColPos r = {0, 0, 0};
    for (int bb = 0; bb < 4; ++bb)
        for (int pp = 0; pp < P; ++pp) {
            int jx_lo = 2, jx_hi = -1;
            for (int jx = 0; jx < 2; ++jx)
                if (col_reach(bits_in, pp, jx)) {
                    jx_lo = jx < jx_lo ? jx : jx_lo;
                    jx_hi = jx;
                }
            const int jy_lo = bb == 3 ? 1 : 0, jy_hi = bb == 0 ? 0 : 1;   // yi - yo in -1..1
            const int lo = jx_lo + 2 * jy_lo, hi = jx_hi + 2 * jy_hi;
            if (bb == b && pp == p) {
                r.base = base;
                r.lo = lo;
                r.hi = hi;
            }
            base += (4 - lo) + 4 + (hi + 1);
        }
    return r;
}

// The positions' table, evaluated at compile time so the issuer's unrolled loops
// see constants.
struct ColTable {
    ColPos pos[16];
};

__host__ __device__ constexpr ColTable make_col_table(bool bits_in)
{
    ColTable t = {};
    const int P = bits_in ? 2 : 4;
    for (int b = 0; b < 4; ++b)
        for (int p = 0; p < P; ++p) t.pos[b * P + p] = col_pos(bits_in, p, b);
    return t;
}

__device__ __forceinline__ Unit col_unit_of(const TcArgs& a, int64_t u)
{
    const int64_t cols = (int64_t)a.ncx * a.ncx;
    const int64_t tile = u / cols;
    const int rem = (int)(u - tile * cols);
    Unit t;
    t.m0 = tile * kTileM;
    t.y = (rem / a.ncx) * 2;
    t.x0 = (rem % a.ncx) * 2;
    return t;
}

// Warps of the column kernel: two epilogue groups of four (group g drains the output planes of parity
// g), the producers, the issuer.
//
// Roles are warp-uniform (the warp index comes from a shuffle, the issuing lane from elect.sync), so
// descriptors, barriers and addresses stay in uniform registers: from a branch on the lane index an MMA
// took 94 - 112 cycles to issue (the pipe takes one in 53 for N <= 64) and a copy 117 - 190.
//
// Times at L = 24, 4,864 samples (38 tiles, 36 units a CTA), lane-indexed roles -> now: first layer 762 ->
// 591 us, hidden 1250 -> 1130, head 1276 -> 952.  Without the prefetch 600, 1154, 961, and a decode of L =
// 12, 2,048 samples 200 us against 190.  One epilogue group is 1% faster there (581, 1125, 946) and 3%
// slower at L = 12 (195 us against 190).  One producer instead of two 2% slower, four 4%
// slower in the head.  What bounds it: the input tiles' way into shared memory, 16 tiles a plane of four
// output sites, 8.6 GB a hidden layer, at 7.6 TB/s (9.0 for the head, which writes no activations); the
// MMAs of a plane take 1344 of its 2300 cycles.
constexpr int kConvProducers = 2;
constexpr int kConvEpi = 8;
// Training's head has a heavier epilogue (an exponential, a logarithm, a division and about 300 FMAs a
// site and sample, 52 running sums a thread) and takes three groups, its weights from shared memory and
// a plane one site at a time; labels, and the backward pass's gating activations, are requested before
// the wait for the accumulators.  L = 12, 2,048 samples: head 199 -> 108 us, backward data 88 -> 72.
__host__ __device__ constexpr int conv_epi(int mode) { return mode == kTcHeadTrain ? 12 : kConvEpi; }
__host__ __device__ constexpr int conv_threads(int mode) { return 32 * (conv_epi(mode) + kConvProducers + 1); }
constexpr int kAhead = 2;   // planes between the L2 prefetch and the copy

template <int kMode, bool kBitsIn>
__global__ void __launch_bounds__(conv_threads(kMode), 1) k_conv_col(const __grid_constant__ TcArgs a)
{
    constexpr int kProducers = kConvProducers;
    constexpr int kEpi = conv_epi(kMode), kFirstProducer = kEpi, kIssuer = kEpi + kProducers;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t ring = smem_u32(sm);
    const uint32_t wsm = ring + kColOffW;
    const uint32_t bars = ring + kColOffBar;
    constexpr int kColIn = col_in_slots(kBitsIn);
    constexpr uint32_t kColInBytes = (uint32_t)(kColRingBytes / kColIn);
    auto full_bar = [&](int i) { return bars + 8u * (uint32_t)i; };
    auto empty_bar = [&](int i) { return bars + 8u * (uint32_t)(kColInMax + i); };
    auto accf_bar = [&](int i) { return bars + 8u * (uint32_t)(2 * kColInMax + i); };
    auto acce_bar = [&](int i) { return bars + 8u * (uint32_t)(2 * kColInMax + kColSlots + i); };
    const uint32_t done_bar = bars + 8u * (uint32_t)(2 * kColInMax + 2 * kColSlots);
    uint32_t* misc = reinterpret_cast<uint32_t*>(sm + kColOffMisc);   // [0] TMEM base, [1] abort flag
    volatile uint32_t* abort_flag = misc + 1;
    ColPos* s_pos = reinterpret_cast<ColPos*>(sm + kColOffPos);   // [b * P + p]
    constexpr int P = kBitsIn ? 2 : 4;

    // the shuffle makes the warp index uniform for the compiler
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

    if (threadIdx.x < 4 * P) s_pos[threadIdx.x] = col_pos(kBitsIn, threadIdx.x % P, threadIdx.x / P);
    __syncthreads();
    // weight windows: for every position (p, b) and element e of its sequence, block
    // W(dx, dy, dz) in the B-operand layout [co/8][chunk][co%8][ci%8], zero out of reach.  First the
    // offset of every (block, chunk) in a.w or -1 (in the still unused input ring), then rows of eight
    // channels, 16 bytes each.  (Element by element with the search inside a launch took 30 us longer: a
    // decode of L = 12, 2,048 samples 281 us, now 192.)
    int* s_k = reinterpret_cast<int*>(sm);   // [block][chunk]
    {
        const ColPos last = s_pos[4 * P - 1];
        const int n_blocks = last.base + (4 - last.lo) + 4 + (last.hi + 1);
        for (int i = threadIdx.x; i < 2 * n_blocks; i += blockDim.x) {
            const int blk = i >> 1, c = i & 1;
            // the position owning block blk
            int pb = 0;
            while (pb + 1 < 4 * P && s_pos[pb + 1].base <= blk) ++pb;
            const ColPos pos = s_pos[pb];
            const int p = pb % P, b = pb / P;
            const int e = blk - pos.base;
            const int part = (e + pos.lo) >> 2, j = (e + pos.lo) & 3;   // block index = 4 part + j - lo
            const int dx = col_chunk_dx(kBitsIn, p, c) - (j & 1);
            const int dy = (b - 1) - (j >> 1);
            const int dz = 1 - part;
            const bool in_reach = dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1;
            s_k[i] = in_reach ? ((dz + 1) * 9 + (dy + 1) * 3 + (dx + 1)) * kC * kC + (kBitsIn ? 0 : c * 8) : -1;
        }
        __syncthreads();
        auto windows = [&](auto&& row_of) {
#pragma unroll 4
            for (int i = threadIdx.x; i < n_blocks * 32; i += blockDim.x) {
                const int blk = i >> 5, c = (i >> 3) & 1, co = (i >> 1 & 8) | (i & 7);   // in the order of the layout
                const int k = s_k[2 * blk + c];
                uint4 w = make_uint4(0u, 0u, 0u, 0u);
                if (k >= 0) w = row_of(a.w + k + co * kC);
                reinterpret_cast<uint4*>(sm + kColOffW)[i] = w;
            }
        };
        if ((reinterpret_cast<uintptr_t>(a.w) & 15) == 0) {
            windows([](const __nv_bfloat16* p) { return __ldg(reinterpret_cast<const uint4*>(p)); });
        } else {   // training takes weights that are only 4-byte aligned
            windows([](const __nv_bfloat16* p) {
                const uint32_t* r = reinterpret_cast<const uint32_t*>(p);
                return make_uint4(__ldg(r), __ldg(r + 1), __ldg(r + 2), __ldg(r + 3));
            });
        }
    }
    fence_proxy_async_smem();
    if (threadIdx.x == 0) {
        for (int i = 0; i < kColIn; ++i) {
            mbar_init(full_bar(i), kProducers);
            mbar_init(empty_bar(i), 1);
        }
        for (int i = 0; i < kColSlots; ++i) {
            mbar_init(accf_bar(i), 1);
            mbar_init(acce_bar(i), 4);
        }
        mbar_init(done_bar, 1);
        misc[1] = 0;
        fence_mbar_init();
    }
    if (kMode == kTcHeadTrain && threadIdx.x < 4 * kC)
        reinterpret_cast<float*>(sm + kColOffHead)[threadIdx.x] =
            threadIdx.x < 3 * kC ? a.w4[threadIdx.x] : a.bias[threadIdx.x - 3 * kC];
    if (warp == kIssuer) tmem_alloc(smem_u32(misc), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, misc[0], 0);
    // every accumulator starts at zero (the epilogue re-zeroes a plane after draining it)
    if (warp < kEpi) {
#pragma unroll 4
        for (int c = 16 * (warp >> 2); c < kColSlots * kColPlaneCols; c += 4 * kEpi)
            tmem_zero16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + c);
        tmem_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    const int L = a.L;
    const uint32_t in_row = kBitsIn ? 16u : 32u;
    const uint32_t tile_bytes = kTileM * in_row;

    if (warp >= kFirstProducer && warp < kIssuer) {
        // one input plane (the 4 x 4 tiles around the column) per slot, one barrier phase each; producer k
        // of n copies the rows b = k, k + n, .. (y0 - 1 + b)
        const int part = warp - kFirstProducer;
        const bool leader = elect_one();
        uint32_t pseq = 0;
        bool ok = true;
        // The column's own sites (rows y0, y0 + 1) are asked for in L2 kAhead planes before they are
        // copied: all columns of a sample tile walk z together, so without it every plane waits for
        // HBM.  The cursor (pu, pz) runs kAhead planes ahead, into the next unit.
        int64_t pu = blockIdx.x;
        int pz = -1;
        Unit pt = col_unit_of(a, pu);
        auto prefetch = [&]() {
            if (pu >= a.n_units) return;
            for (int b = part; b < 2; b += kProducers)
                if (leader && pt.y + b < L)
                    bulk_prefetch(a.in + tile_off(((int64_t)wrap(pz, L) * L + pt.y + b) * L + pt.x0, pt.m0, a.L3,
                                                  tile_bytes),
                                  (pt.x0 + 1 < L ? 2u : 1u) * tile_bytes);
            if (++pz > L) {
                pz = -1;
                pu += gridDim.x;
                pt = col_unit_of(a, pu);
            }
        };
        for (int k = 0; k < kAhead; ++k) prefetch();
        for (int64_t u = blockIdx.x; u < a.n_units && ok; u += gridDim.x) {
            const Unit t = col_unit_of(a, u);
            const uint8_t* tile0 = a.in + tile_off(0, t.m0, a.L3, tile_bytes);
            // the row's tiles are one run of sites unless it wraps
            const bool run = t.x0 >= 1 && t.x0 + 2 < L;
            for (int zi = -1; zi <= L; ++zi) {
                const int g = (int)(pseq % kColIn);
                const uint32_t use = pseq / kColIn;
                bool good = true;
                if (leader && use > 0) good = wait_bar(empty_bar(g), (use - 1) & 1u, abort_flag);
                ok = __all_sync(0xffffffffu, good);
                if (!ok) break;
                if (leader) mbar_arrive_expect_tx(full_bar(g), (16u / kProducers) * tile_bytes);
#pragma unroll
                for (int k = 0; k < 4 / kProducers; ++k) {
                    const int b = part + k * kProducers;
                    const uint8_t* row = tile0 + (int64_t)((wrap(zi, L) * L + wrap(t.y - 1 + b, L)) * L) * tile_bytes;
                    const uint32_t dst = ring + (uint32_t)g * kColInBytes + (uint32_t)b * 4u * tile_bytes;
                    if (run) {
                        if (leader)
                            bulk_load(dst, row + (int64_t)(t.x0 - 1) * tile_bytes, 4u * tile_bytes, full_bar(g));
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (leader)
                                bulk_load(dst + (uint32_t)i * tile_bytes,
                                          row + (int64_t)wrap(t.x0 - 1 + i, L) * tile_bytes, tile_bytes, full_bar(g));
                    }
                }
                prefetch();
                ++pseq;
            }
        }
        // copies still in flight land before the CTA exits
        if (leader) {
            const uint32_t last = pseq < (uint32_t)kColIn ? pseq : (uint32_t)kColIn;
            for (uint32_t g = 0; g < last; ++g) {
                const uint32_t q = pseq - 1 - ((pseq - 1 - g) % kColIn);
                wait_bar(full_bar((int)g), (q / kColIn) & 1u, abort_flag, true);
            }
        }
        __syncwarp();
    } else if (warp == kIssuer) {
        const bool leader = elect_one();
        // The tensor pipe takes only a few MMAs ahead, so what this thread does between two planes
        // idles it: the next plane's barriers are tested (without waiting) before the current
        // plane's last row is issued, while the pipe still has work.
        constexpr uint32_t a_lbo = 2048u, a_sbo = 128u;
        const uint64_t bdesc0 = smem_desc(wsm, 128u, 256u);   // + 32 per 512-byte block
        const uint64_t adesc_ring = smem_desc(ring, a_lbo, a_sbo);
        constexpr uint32_t kIdescBase = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTileM >> 4) << 24);
        constexpr ColTable kTab = make_col_table(kBitsIn);
        const uint32_t n_planes = (uint32_t)L + 2;   // input planes of a unit, zi = -1 .. L
        uint32_t pseq = 0, qbase = 0;                // input planes done; output planes of finished units
        bool ok = true;
        // barriers of a plane: its copies, and the accumulators of output plane zi + 1, first written by
        // it, drained (use 0 of a slot needs no wait)
        auto full_done = [&](uint32_t seq) { return mbar_test(full_bar((int)(seq % kColIn)), (seq / kColIn) & 1u); };
        auto slot_done = [&](uint32_t q) { return q < 8 || mbar_test(acce_bar((int)(q & 7)), ((q >> 3) - 1) & 1u); };
        bool ready = false;
        for (int64_t u = blockIdx.x; u < a.n_units && ok; u += gridDim.x) {
            for (uint32_t k = 0; k < n_planes; ++k) {   // zi = k - 1; writes output planes k - 2 .. k
                if (!ready) {
                    const uint32_t q = qbase + k;
                    bool good = true;
                    if (leader) {
                        good = k >= (uint32_t)L || q < 8 ||
                               wait_bar(acce_bar((int)(q & 7)), ((q >> 3) - 1) & 1u, abort_flag);
                        good = good && wait_bar(full_bar((int)(pseq % kColIn)), (pseq / kColIn) & 1u, abort_flag);
                    }
                    ok = __all_sync(0xffffffffu, good);
                    if (!ok) break;
                }
                tc_fence_after();
                // parts P1 .. P2 of the windows: output planes k - 2 + P1 .. k - 2 + P2
                const uint32_t P1 = k >= 2 ? 0u : 2u - k, P2 = k < (uint32_t)L ? 2u : (uint32_t)L + 1 - k;
                const uint32_t s1 = (qbase + k - 2 + P1) & 7u, n = P2 - P1;
                // the window of position (b, p): blocks 4 P1 .. 4 P2 + hi - lo of its sequence
                // into TMEM column 64 s1 + 16 lo, N = 16 (4 (P2 - P1) + hi - lo + 1)
                const uint64_t bdesc_plane = bdesc0 + (uint64_t)(128 * P1);
                const uint32_t idesc_plane = kIdescBase + ((8 * n) << 17);
                const uint32_t col_plane = tmem + s1 * kColPlaneCols;
                const uint64_t adesc_plane = adesc_ring + (uint64_t)((pseq % kColIn) * (kColInBytes >> 4));
                auto row_mmas = [&](int b) {
                    const uint64_t adesc0 = adesc_plane + (uint64_t)((uint32_t)b * ((4u * tile_bytes) >> 4));
                    if (s1 + n <= 7) {
#pragma unroll
                        for (int p = 0; p < P; ++p) {
                            const ColPos pos = kTab.pos[b * P + p];
                            if (leader)
                                mma_bf16_n(col_plane + (uint32_t)(pos.lo * kC),
                                           adesc0 + (uint64_t)(p * (kSlotBytes >> 4)),
                                           bdesc_plane + (uint64_t)(32 * pos.base),
                                           idesc_plane + ((uint32_t)(2 * (pos.hi - pos.lo + 1)) << 17));
                        }
                    } else {
                        // the window crosses the ring's end: split at slot 0, part Pw
                        const int Pw = (int)(P1 + 8 - s1);
#pragma unroll
                        for (int p = 0; p < P; ++p) {
                            const ColPos pos = kTab.pos[b * P + p];
                            const uint64_t adesc = adesc0 + (uint64_t)(p * (kSlotBytes >> 4));
                            auto issue = [&](int pa, int ja, int pz, int jz, uint32_t col) {
                                // blocks (pa, ja) .. (pz, jz) of the sequence into TMEM column col
                                const int b0 = 4 * pa + ja - pos.lo, nb = 4 * (pz - pa) + jz - ja + 1;
                                if (leader)
                                    mma_bf16_n(tmem + col, adesc, bdesc0 + (uint64_t)(32 * (pos.base + b0)),
                                               kIdescBase | ((uint32_t)(nb * 2) << 17));
                            };
                            issue((int)P1, pos.lo, Pw - 1, 3, s1 * kColPlaneCols + (uint32_t)(pos.lo * kC));
                            issue(Pw, 0, (int)P2, pos.hi, 0u);
                        }
                    }
                };
#pragma unroll
                for (int b = 0; b < 3; ++b) row_mmas(b);
                // the next plane (of this unit or the next): both barriers, if any, already complete?
                const bool last = k + 1 == n_planes;
                const uint32_t kn = last ? 0 : k + 1, qn = (last ? qbase + (uint32_t)L : qbase) + kn;
                ready = __all_sync(0xffffffffu, full_done(pseq + 1) && (kn >= (uint32_t)L || slot_done(qn)));
                row_mmas(3);
                if (leader) mma_commit(empty_bar((int)(pseq % kColIn)));
                ++pseq;
                // output plane k - 2 has received its last contribution
                if (leader && k >= 2) mma_commit(accf_bar((int)((qbase + k - 2) & 7u)));
            }
            qbase += (uint32_t)L;
        }
        // every MMA issued has completed before TMEM is released
        if (leader) {
            mma_commit(done_bar);
            wait_bar(done_bar, 0, abort_flag, true);
        }
        __syncwarp();
    } else {
        // epilogue: the warp owns TMEM lanes (= tile rows = samples) 32 quad .. 32 quad + 31
        const int quad = warp & 3, r = quad * 32 + lane;
        constexpr bool kHead = tc_head(kMode);
        // training's head keeps its weights in shared memory and takes a plane a site at a time: the sums
        // need the registers
        constexpr bool kLean = kMode == kTcHeadTrain;
        const uint32_t head = smem_u32(sm) + kColOffHead;   // w4 [3][16], bias [16]
        float bias[kC];
#pragma unroll
        for (int c = 0; c < kC; ++c) bias[c] = kMode == kTcMask || kLean ? 0.0f : a.bias[c];
        float w4[kHead && !kLean ? 3 * kC : 1];
        float b4[3] = {0.0f, 0.0f, 0.0f};
        if (kHead) {
#pragma unroll
            for (int i = 0; i < 3 * kC && !kLean; ++i) w4[i] = a.w4[i];
#pragma unroll
            for (int d = 0; d < 3; ++d) b4[d] = a.b4[d];
        }
        // training: this thread's share of the head's gradients and of the loss
        constexpr int kAcc = kMode == kTcHeadTrain ? 3 * kC + 3 + 1 : 1;
        float acc[kAcc];
#pragma unroll
        for (int i = 0; i < kAcc; ++i) acc[i] = 0.0f;
        int64_t q = 0;
        bool ok = true;
        for (int64_t u = blockIdx.x; u < a.n_units && ok; u += gridDim.x) {
            const Unit t = col_unit_of(a, u);
            const int64_t sample = t.m0 + r;
            const bool valid = sample < a.n_samples;
            const int64_t wd = (t.m0 + quad * 32) / 64;   // the warp's word, its half hw
            const int hw = quad & 1;
            for (int zo = 0; zo < L; ++zo, ++q) {
                const int s = (int)(q & 7);
                if ((int)((uint32_t)q % (kEpi / 4)) != warp >> 2) continue;   // another group's plane
                // what the epilogue reads of the plane beside the accumulators, requested before the wait
                uint4 mask[kMode == kTcMask ? 4 : 1][2];
                uint64_t labels = 0;   // lane 4 d + j: edge d's label word of site j
                if (kMode == kTcMask) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int xo = t.x0 + (j & 1), yo = t.y + (j >> 1);
                        if (xo >= L || yo >= L) continue;
                        const uint8_t* p = a.mask_act +
                                           tile_off(((int64_t)zo * L + yo) * L + xo, t.m0, a.L3, 4096) + r * 16;
                        mask[kMode == kTcMask ? j : 0][0] = *reinterpret_cast<const uint4*>(p);
                        mask[kMode == kTcMask ? j : 0][1] = *reinterpret_cast<const uint4*>(p + 2048);
                    }
                } else if (kMode == kTcHeadTrain) {
                    const int xo = t.x0 + (lane & 1), yo = t.y + (lane >> 1 & 1);
                    if (lane < 12 && xo < L && yo < L && wd < a.words)
                        labels = a.label[((int64_t)(lane >> 2) * a.L3 + ((int64_t)zo * L + yo) * L + xo) * a.W + wd];
                }
                int got = 1;
                if (lane == 0) got = wait_bar(accf_bar(s), (uint32_t)(q >> 3) & 1u, abort_flag) ? 1 : 0;
                got = __shfl_sync(0xffffffffu, got, 0);
                if (!got) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(s * kColPlaneCols);
                uint32_t raw[kLean ? 1 : 4][16];
                if (!kLean) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) tmem_ld16(lane_base + (uint32_t)(j * kC), raw[kLean ? 0 : j]);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 4; ++j) tmem_zero16(lane_base + (uint32_t)(j * kC));
                }
#pragma unroll (kLean ? 1 : 4)
                for (int j = 0; j < 4; ++j) {
                    if (kLean) {
                        tmem_ld16(lane_base + (uint32_t)(j * kC), raw[0]);
                        tmem_wait_ld();
                        tmem_zero16(lane_base + (uint32_t)(j * kC));
                    }
                    const int xo = t.x0 + (j & 1), yo = t.y + (j >> 1);
                    if (xo >= L || yo >= L) continue;   // the odd lattice's last column
                    const int64_t site = ((int64_t)zo * L + yo) * L + xo;
                    const int64_t row_off = tile_off(site, t.m0, a.L3, 4096) + r * 16;
                    float v[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) v[c] = __uint_as_float(raw[kLean ? 0 : j][c]);
                    if (kMode == kTcRelu || kMode == kTcMask) {
                        uint32_t pk[8];
                        if (kMode == kTcRelu) {
#pragma unroll
                            for (int c = 0; c < kC; c += 2)
                                pk[c / 2] = pack2(fmaxf(v[c] + bias[c], 0.0f), fmaxf(v[c + 1] + bias[c + 1], 0.0f));
                        } else {
                            // the gradient passes where the forward activation (a ReLU output,
                            // so never negative) is non-zero
                            const uint4 m0v = mask[kMode == kTcMask ? j : 0][0], m1v = mask[kMode == kTcMask ? j : 0][1];
                            const uint32_t mw[8] = {m0v.x, m0v.y, m0v.z, m0v.w, m1v.x, m1v.y, m1v.z, m1v.w};
#pragma unroll
                            for (int c = 0; c < kC; c += 2)
                                pk[c / 2] = pack2((mw[c / 2] & 0x7FFFu) ? v[c] : 0.0f,
                                                  (mw[c / 2] & 0x7FFF0000u) ? v[c + 1] : 0.0f);
                        }
                        uint8_t* dst = a.out + row_off;
                        *reinterpret_cast<uint4*>(dst) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        *reinterpret_cast<uint4*>(dst + 2048) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                    } else {
                        float y3[kC];
                        float z[3] = {b4[0], b4[1], b4[2]};
#pragma unroll
                        for (int c4 = 0; c4 < kC; c4 += 4) {
                            float bw[4][4];   // the three heads' weights and the bias of channels c4 .. c4 + 3
#pragma unroll
                            for (int d = 0; d < 4; ++d) {
                                if (kLean) {
                                    lds4(head + (uint32_t)(d * kC + c4) * 4u, bw[d]);
                                } else {
#pragma unroll
                                    for (int c = 0; c < 4; ++c) bw[d][c] = d < 3 ? w4[kLean ? 0 : d * kC + c4 + c] : bias[c4 + c];
                                }
                            }
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                y3[c4 + c] = fmaxf(v[c4 + c] + bw[3][c], 0.0f);
#pragma unroll
                                for (int d = 0; d < 3; ++d) z[d] = fmaf(y3[c4 + c], bw[d][c], z[d]);
                            }
                        }
                        if (kMode == kTcHead) {
#pragma unroll
                            for (int d = 0; d < 3; ++d) {
                                if (a.logits && valid)
                                    a.logits[((int64_t)d * a.L3 + site) * a.n_samples + sample] = z[d];
                                const uint32_t bits = __ballot_sync(0xffffffffu, valid && z[d] > 0.0f);
                                if (lane == 0 && wd < a.words) a.dec32[(wd * a.L3 + site) * 8 + 2 * d + hw] = bits;
                            }
                        } else {
                            // binary cross-entropy of the logits against the labels (the mean over
                            // edges and samples is what training minimises): dL/dz = (sigmoid(z) - y) / N
                            float dz[3];
#pragma unroll
                            for (int d = 0; d < 3; ++d) {
                                const uint64_t lw = __shfl_sync(0xffffffffu, labels, 4 * d + j);
                                const float yv = (float)((uint32_t)(lw >> (32 * hw + lane)) & 1u);
                                const float ez = expf(-fabsf(z[d])), sig = (z[d] < 0.0f ? ez : 1.0f) / (1.0f + ez);
                                dz[d] = valid ? (sig - yv) * a.inv_n : 0.0f;
                                if (valid) acc[3 * kC + 3] += fmaxf(z[d], 0.0f) - z[d] * yv + log1pf(ez);
                                acc[3 * kC + d] += dz[d];
                            }
                            uint32_t pk[8];
#pragma unroll
                            for (int c4 = 0; c4 < kC; c4 += 4) {
                                float g4[4], hw4[3][4];
#pragma unroll
                                for (int d = 0; d < 3; ++d) lds4(head + (uint32_t)(d * kC + c4) * 4u, hw4[d]);
#pragma unroll
                                for (int h = 0; h < 4; ++h) {
                                    float dy = 0.0f;
#pragma unroll
                                    for (int d = 0; d < 3; ++d) {
                                        dy = fmaf(dz[d], hw4[d][h], dy);
                                        acc[d * kC + c4 + h] = fmaf(y3[c4 + h], dz[d], acc[d * kC + c4 + h]);
                                    }
                                    g4[h] = y3[c4 + h] > 0.0f ? dy : 0.0f;
                                }
                                pk[c4 / 2] = pack2(g4[0], g4[1]);
                                pk[c4 / 2 + 1] = pack2(g4[2], g4[3]);
                            }
                            uint8_t* dst = a.out + row_off;
                            *reinterpret_cast<uint4*>(dst) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                            *reinterpret_cast<uint4*>(dst + 2048) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                        }
                    }
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acce_bar(s));
            }
        }
        if (kMode == kTcHeadTrain) {
            // the warp's sums, then one atomic per value and warp
#pragma unroll
            for (int i = 0; i < kAcc; ++i) {
                float x = acc[i];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                if (lane == 0 && x != 0.0f) {
                    float* dst = i < 3 * kC ? a.grad_w4 + i : (i < 3 * kC + 3 ? a.grad_b4 + (i - 3 * kC) : a.loss);
                    atomicAdd(dst, x);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kIssuer) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// First layer's input: [site][sample][8] BF16, channels s_{t-1}(n) then s_t(n)
// for n = 0..2, then two zeros.  Rows past n_samples are zero.  One warp per
// site and 256 samples (4 words): lanes 0..23 load the 6 channels x 4 words,
// and store j of the warp writes samples 32j .. 32j + 31 (512 contiguous bytes).
__global__ void k_expand_bits(int L3, int64_t Sp, int64_t W, int64_t words, const uint64_t* __restrict__ s_prev,
                              const uint64_t* __restrict__ s_cur, uint4* __restrict__ out)
{
    const int64_t site = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int64_t m0 = (int64_t)blockIdx.y * 256;
    if (site >= L3) return;
    uint64_t v = 0;
    if (lane < 24) {
        const int c = lane >> 2;
        const int64_t w = (m0 >> 6) + (lane & 3);
        if (w < words) {
            const uint64_t* src = c < 3 ? s_prev : s_cur;
            v = __ldg(&src[((int64_t)(c % 3) * L3 + site) * W + w]);
        }
    }
    constexpr uint32_t one = 0x3F80u;   // BF16 1.0
    // tile-major layout: samples m0 .. m0 + 127 in tile m0 / 128 of the site, the next 128 in
    // the next tile (L3 tiles further)
    uint4* dst = out + ((m0 >> 7) * L3 + site) * kTileM + lane;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (m0 + 32 * j >= Sp) break;
        const uint32_t half = (uint32_t)(v >> (32 * (j & 1)));
        uint32_t h[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) h[c] = ((__shfl_sync(0xffffffffu, half, c * 4 + (j >> 1)) >> lane) & 1u) * one;
        dst[(j >> 2) * (int64_t)L3 * kTileM + 32 * (j & 3)] =
            make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), 0u);
    }
}

// ------------------------------------------------------------------ weight gradients
// Weight and bias gradients of one convolution as a GEMM over samples:
//   G[(k, ci)][co] = sum over sites r and samples s of x[r + off_k][s][ci] . d[r][s][co],
// K = 16 samples per MMA.  The reduction runs over samples; both operands are the convolutions'
// own tiles read with the channels as the contiguous dimension (core matrices of 8 samples x 8
// channels, LBO 128 B to the next 8 samples, SBO 2048 B to the next 8 channels, which is also the
// step to the next tile of a run).
//
// Work unit: one 128-sample tile x two rows (y, z), (y + 1, z), walked along x.  The 12 tiles around
// the rows at one x, (dy, dz) = -1..2 x -1..1 with dy fastest, form a column.  A column meets the d tiles
// of a row's three sites x - 1, x, x + 1 as dx = +1, 0, -1 at once: the MMA's M rows are the column's
// tiles (and a tile of ones, whose rows give the bias gradient sum d[r][s][co]), its N = 48 columns those
// three d tiles.  The second row takes the same column from one tile further on, so that dy counts from
// it, into the same accumulators (of every four tiles three are read); the ones are there twice.  So an x
// tile is copied once per two rows: seven tiles a site with the d's, where fetching a site's 27
// neighbours took 29; and a site takes 16 MMAs (first layer: 8) where N = 16 columns per neighbour took
// 32 (16).  M is 128: eight 16-channel tiles, then the other four and the ones in an MMA of their own;
// the first layer's twelve 8-channel tiles and the ones fit one.  Rows past a group's last tile multiply
// whatever follows in shared memory and are never read.
//
// (Both rows' d tiles in one MMA of N = 96, the two rows' sums apart, is faster still, 77 and 55 us.  But
// the tensor cores' sums over half the terms differ from the whole ones by 3e-5.)
//
// The d tiles of each row sit in a ring of slots whose first two are written a second time behind the
// last, so that any three in a row are contiguous.  The accumulators (48 columns of TMEM per group) live
// for the whole launch; at its end they go through shared memory, so that they are added to the gradients
// in runs (every lane adding its own: about 10 us more).
//
// What bounds it: the MMAs (53 cycles each however small N is, 80 us) and the copies to shared memory (29
// KB a site, first layer 17) alike.  L = 12, 2,048 samples: 103 us for a 16-channel layer, 65 us for the
// first; a row at a time (42 KB a site) 113 and 98.  Before, with channel-major copies of x and d written
// first (350 us a step in all), 27 neighbour tiles fetched per site and N = 16: 490 and 330 us.
//
// One elected thread of a converged warp issues the MMAs, and one of each of three producer warps the
// copies: warp and loop state are then uniform, and addresses and descriptors stay in uniform
// registers.  From a branch on the lane index every MMA took 94 - 112 cycles to issue and every copy
// 117 - 190 (164 and 154 us a launch).
constexpr int kWgProducers = 3;
constexpr int kWgThreads = kTcThreads + 32 * (kWgProducers - 1);

template <int kCin>
struct WgShape {
    static constexpr uint32_t kTileB = kCin * 256;               // one x tile
    static constexpr uint32_t kColB = 14 * kTileB;               // twelve tiles and the ones twice
    static constexpr int kCols = kCin == 16 ? 3 : 5;             // column slots
    static constexpr int kGroups = kCin == 16 ? 2 : 1;           // M groups: tiles 0..7 and 8..12
    static constexpr int kD = 5;                                 // a row's d slots (and two mirrors), 4 KiB each
    static constexpr uint32_t kOffD = kCols * kColB;
    static constexpr uint32_t kOffBar = kOffD + 2 * (kD + 2) * 4096;
    static constexpr int kBars = 2 * kCols + kD + 1;             // column full, empty; d empty; done
    static constexpr uint32_t kOffMisc = kOffBar + kBars * 8;
    static constexpr int kSmem = (int)kOffMisc + 16 + 1024;
    static_assert(kSmem <= 227 * 1024, "shared memory budget");
    // a group reads 32 KiB from its first tile on
    static_assert(kOffBar >= (kCols - 1) * kColB + ((kGroups - 1) * 8 + 1) * kTileB + 32768, "group reads stay inside");
};

struct WgArgs {
    int L, L3;
    int64_t n_units;            // 128-sample tiles x L planes x ceil(L / 2) pairs of rows
    const uint8_t* x;           // x tiles (kCin channels)
    const uint8_t* d;           // d tiles (16 channels)
    const uint8_t* ones;        // one x tile of BF16 ones
    int cin;                    // input channels kept in gw (6 for the first layer)
    float* gw;                  // [co][cin][27], accumulated
    float* gb;                  // [16], accumulated
};

template <int kCin>
__global__ void __launch_bounds__(kWgThreads, 1) k_wgrad_tc(const __grid_constant__ WgArgs a)
{
    using Sh = WgShape<kCin>;
    constexpr uint32_t kTileB = Sh::kTileB;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t base = smem_u32(sm);
    const uint32_t bars = base + Sh::kOffBar;
    // use q of a ring of n goes to slot q % n, its phase parity is (q / n) & 1
    constexpr uint32_t kNc = Sh::kCols, kNd = Sh::kD;
    auto col_full = [&](uint32_t q) { return bars + 8u * (q % kNc); };
    auto col_empty = [&](uint32_t q) { return bars + 8u * (kNc + q % kNc); };
    auto d_empty = [&](uint32_t q) { return bars + 8u * (2 * kNc + q % kNd); };
    auto col_at = [&](uint32_t q) { return base + (q % kNc) * Sh::kColB; };
    auto d_at = [&](uint32_t q, int r) { return base + Sh::kOffD + ((uint32_t)r * (kNd + 2) + q % kNd) * 4096u; };
    const uint32_t done_bar = bars + 8u * (2 * kNc + kNd);
    uint32_t* misc = reinterpret_cast<uint32_t*>(sm + Sh::kOffMisc);   // [0] TMEM base, [1] abort
    volatile uint32_t* abort_flag = misc + 1;
    // the shuffle makes the warp index uniform for the compiler
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < Sh::kBars; ++i) mbar_init(bars + 8u * (uint32_t)i, i < Sh::kCols ? kWgProducers : 1);
        misc[1] = 0;
        fence_mbar_init();
    }
    // the ones behind every column's twelve tiles
    constexpr uint32_t kOnes = kTileB / 16;
    for (uint32_t i = threadIdx.x; i < kNc * 2 * kOnes; i += blockDim.x)
        reinterpret_cast<uint4*>(sm + (i / (2 * kOnes)) * Sh::kColB + 12u * kTileB)[i % (2 * kOnes)] =
            reinterpret_cast<const uint4*>(a.ones)[i % kOnes];
    fence_proxy_async_smem();
    if (warp == kIssuerWarp) tmem_alloc(smem_u32(misc), 128);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, misc[0], 0);
    bool finished = true;   // the issuer's: every MMA has completed
    const int L = a.L, pairs = (L + 1) / 2, per_tile = pairs * L;

    if (warp == kProducerWarp || warp > kIssuerWarp) {
        // producer p copies the tiles 4 p .. 4 p + 3 of a column, the last one the d tiles too
        const int part = warp == kProducerWarp ? 0 : warp - kIssuerWarp;
        const bool leader = elect_one();
        uint32_t cq = 0, dq = 0;   // columns and d tiles copied so far
        bool ok = true;
        for (int64_t u = blockIdx.x; u < a.n_units && ok; u += gridDim.x) {
            const int64_t t = u / per_tile;
            const int row = (int)(u - t * per_tile), y = 2 * (row % pairs), z = row / pairs;
            const uint8_t* xt = a.x + t * a.L3 * (int64_t)kTileB;
            const uint8_t* dt = a.d + (t * a.L3 + ((int64_t)z * L + y) * L) * 4096;
            const uint32_t rows = y + 1 < L ? 2 : 1;   // the odd lattice's last row is alone
            // the row of tile i = 4 part + k: (dy, dz) = (i % 4 - 1, i / 4 - 1) = (k - 1, part - 1)
            const uint8_t* xrow[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                xrow[k] = xt + ((int64_t)wrap(z + part - 1, L) * L + wrap(y + k - 1, L)) * L * (int64_t)kTileB;
            for (int c = 0; c < L; ++c) {
                // d tiles in the order L - 1, 0, 1, .., L - 1, 0: the first column brings three of them
                const uint32_t nd = part != 2 ? 0 : (c == 0 ? 3 : 1);
                uint32_t mirrors = 0;
                for (uint32_t k = dq; k < dq + nd; ++k) mirrors += k % kNd < 2 ? 1u : 0u;
                bool good = true;
                if (leader) {
                    if (cq >= kNc) good = wait_bar(col_empty(cq), ((cq / kNc) - 1) & 1u, abort_flag);
                    for (uint32_t k = dq; good && k < dq + nd; ++k)
                        if (k >= kNd) good = wait_bar(d_empty(k), ((k / kNd) - 1) & 1u, abort_flag);
                }
                ok = __all_sync(0xffffffffu, good);
                if (!ok) break;
                if (leader) mbar_arrive_expect_tx(col_full(cq), 4u * kTileB + (nd + mirrors) * rows * 4096u);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (leader)
                        bulk_load(col_at(cq) + (uint32_t)(4 * part + k) * kTileB, xrow[k] + (uint32_t)c * kTileB, kTileB,
                                  col_full(cq));
                for (uint32_t k = dq; k < dq + nd; ++k) {
                    const uint8_t* src = dt + (int64_t)wrap(c + 1 - (int)(dq + nd - 1 - k), L) * 4096;
                    for (uint32_t r = 0; r < rows; ++r, src += (int64_t)L * 4096) {
                        if (leader) bulk_load(d_at(k, (int)r), src, 4096u, col_full(cq));
                        if (leader && k % kNd < 2) bulk_load(d_at(k, (int)r) + kNd * 4096u, src, 4096u, col_full(cq));
                    }
                }
                ++cq;
                dq += nd;
            }
        }
        // copies still in flight land before the CTA exits
        if (leader)
            for (uint32_t k = cq > kNc ? cq - kNc : 0; k < cq; ++k)
                wait_bar(col_full(k), (k / kNc) & 1u, abort_flag, true);
        __syncwarp();
    } else if (warp == kIssuerWarp) {
        const bool leader = elect_one();
        // A and B are read with their channels as the contiguous dimension (bits 15 and 16)
        constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                                    ((uint32_t)(48 >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
        uint32_t cq = 0, dq = 0;   // columns done; the first d tile of the current column's three
        bool ok = true;
        for (int64_t u = blockIdx.x; u < a.n_units && ok; u += gridDim.x) {
            const bool alone = L % 2 != 0 && u % pairs == pairs - 1;   // the odd lattice's last row
            for (int c = 0; c < L; ++c) {
                bool good = true;
                if (leader) good = wait_bar(col_full(cq), (cq / kNc) & 1u, abort_flag);
                ok = __all_sync(0xffffffffu, good);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (r == 1 && alone) break;
                    const uint64_t bdesc = smem_desc(d_at(dq, r), 128u, 2048u);
#pragma unroll
                    for (int grp = 0; grp < Sh::kGroups; ++grp) {
                        const uint64_t adesc = smem_desc(col_at(cq) + (uint32_t)(grp * 8 + r) * kTileB, 128u, 2048u);
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk) {
                            // 16 samples per step: two core matrices (256 B) further along K
                            const uint64_t step = (uint64_t)((kk * 256) >> 4);
                            if (leader) {
                                if (r == 0 && kk == 0 && cq == 0)
                                    mma_bf16_overwrite(tmem + (uint32_t)(grp * 48), adesc + step, bdesc + step, kIdesc);
                                else
                                    mma_bf16_n(tmem + (uint32_t)(grp * 48), adesc + step, bdesc + step, kIdesc);
                            }
                        }
                    }
                }
                if (leader) {
                    mma_commit(col_empty(cq));
                    mma_commit(d_empty(dq));
                    if (c == L - 1) {   // the row's last two d tiles serve no further column
                        mma_commit(d_empty(dq + 1));
                        mma_commit(d_empty(dq + 2));
                    }
                }
                ++cq;
                ++dq;
            }
            dq += 2;
        }
        if (leader) {
            mma_commit(done_bar);
            finished = wait_bar(done_bar, 0, abort_flag, true);
        }
        __syncwarp();
    }
    // every MMA and copy has completed (or the launch gave up): the sums go to shared memory in the
    // gradients' layout, and from there to the gradients in runs
    tc_fence_before();
    const bool good = __syncthreads_and(finished && !*abort_flag);
    tc_fence_after();
    if (good) {
        float* g = reinterpret_cast<float*>(sm);   // [co][cin][27], then [16] of the bias
        const int n_w = kC * a.cin * kOff;
        if (warp < kEpiWarps) {
            const int m = warp * 32 + lane, ci = m % kCin;   // TMEM lane = M row
#pragma unroll
            for (int grp = 0; grp < Sh::kGroups; ++grp) {
                const int i = grp * 8 + m / kCin;            // the tile from the row's first, (dy, dz) = (i % 4, i / 4) - 1
#pragma unroll
                for (int j = 0; j < 3; ++j) {                // the site c - 1 + j: dx = 1 - j
                    uint32_t v[16];
                    tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(grp * 48 + j * 16), v);
                    tmem_wait_ld();
                    if (i < 12 && (i & 3) < 3 && ci < a.cin) {
#pragma unroll
                        for (int co = 0; co < 16; ++co)
                            g[(co * a.cin + ci) * kOff + 3 * (3 * (i >> 2) + (i & 3)) + 2 - j] = __uint_as_float(v[co]);
                    } else if (i == 12 && ci == 0 && j == 1) {
#pragma unroll
                        for (int co = 0; co < 16; ++co) g[n_w + co] = __uint_as_float(v[co]);
                    }
                }
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < n_w + kC; i += blockDim.x) atomicAdd(i < n_w ? a.gw + i : a.gb + (i - n_w), g[i]);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kIssuerWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, 128);
    }
}

__global__ void k_fill_ones(uint16_t* __restrict__ p, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = 0x3F80u;   // BF16 1.0
}

int64_t tc_padded(int64_t n) { return (n + kTileM - 1) / kTileM * kTileM; }
size_t r256(size_t x) { return (x + 255) / 256 * 256; }

int sm_count()
{
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    return n > 0 ? n : 1;
}

template <int kMode, bool kBitsIn>
t3d_status launch_conv_col(const TcArgs& a, cudaStream_t st)
{
    const int grid = (int)std::min<int64_t>(a.n_units, sm_count());
    ProfScope prof(T3D_K_CNN, st);
    k_conv_col<kMode, kBitsIn><<<grid, conv_threads(kMode), kColSmemBytes, st>>>(a);
    T3D_LAUNCH_CHECK("tensor-core convolution");
    return T3D_OK;
}

// Arguments shared by every convolution of a pass over n_samples samples.
TcArgs base_args(int L, int64_t n_samples, int64_t W)
{
    TcArgs a;
    std::memset(&a, 0, sizeof(a));
    const int64_t Sp = tc_padded(n_samples);
    a.L = L;
    a.L3 = L * L * L;
    a.Sp = Sp;
    a.n_samples = n_samples;
    a.W = W;
    a.words = words_for(n_samples);
    a.ncx = (L + 1) / 2;
    a.n_units = (Sp / kTileM) * a.ncx * a.ncx;
    return a;
}

t3d_status expand_bits(const TcArgs& a, const uint64_t* s_prev, const uint64_t* s, uint8_t* x0, cudaStream_t st)
{
    ProfScope prof(T3D_K_CNN, st);
    const dim3 grid((unsigned)((a.L3 + 7) / 8), (unsigned)((a.Sp + 255) / 256));
    k_expand_bits<<<grid, 256, 0, st>>>(a.L3, a.Sp, a.W, a.words, s_prev, s, reinterpret_cast<uint4*>(x0));
    T3D_LAUNCH_CHECK("pre-decoder input expansion");
    return T3D_OK;
}

}  // namespace

t3d_status tc_prepare()
{
    static std::mutex mu;
    static bool configured[64] = {};
    int dev = 0;
    T3D_CUDA_CHECK(cudaGetDevice(&dev));
    T3D_REQUIRE(dev >= 0 && dev < 64, "device %d outside the 64 supported", dev);
    std::lock_guard<std::mutex> lock(mu);
    if (!configured[dev]) {
        const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
        T3D_CUDA_CHECK(cudaFuncSetAttribute(k_conv_col<kTcRelu, true>, attr, kColSmemBytes));
        T3D_CUDA_CHECK(cudaFuncSetAttribute(k_conv_col<kTcRelu, false>, attr, kColSmemBytes));
        T3D_CUDA_CHECK(cudaFuncSetAttribute(k_conv_col<kTcHead, false>, attr, kColSmemBytes));
        T3D_CUDA_CHECK(cudaFuncSetAttribute(k_conv_col<kTcHeadTrain, false>, attr, kColSmemBytes));
        T3D_CUDA_CHECK(cudaFuncSetAttribute(k_conv_col<kTcMask, false>, attr, kColSmemBytes));
        T3D_CUDA_CHECK(cudaFuncSetAttribute(k_wgrad_tc<8>, attr, WgShape<8>::kSmem));
        T3D_CUDA_CHECK(cudaFuncSetAttribute(k_wgrad_tc<kC>, attr, WgShape<kC>::kSmem));
        configured[dev] = true;
    }
    return T3D_OK;
}

size_t tc_act_bytes(int L, int64_t n_samples, int channels)
{
    return r256((size_t)L * L * L * (size_t)tc_padded(n_samples) * 2 * (size_t)channels);
}

size_t tc_workspace_bytes(int L, int64_t n_samples)
{
    return tc_act_bytes(L, n_samples, 8) + 2 * tc_act_bytes(L, n_samples, kC);
}

t3d_status launch_forward_tc(int L, int64_t n_samples, int64_t W, const uint64_t* s_prev, const uint64_t* s,
                             uint64_t* dec, const Blob* blob, float* logits_out, void* work, cudaStream_t st)
{
    uint8_t* in0 = static_cast<uint8_t*>(work);
    uint8_t* act0 = in0 + tc_act_bytes(L, n_samples, 8);
    uint8_t* act1 = act0 + tc_act_bytes(L, n_samples, kC);
    T3D_TRY(tc_prepare());
    TcArgs a = base_args(L, n_samples, W);
    T3D_TRY(expand_bits(a, s_prev, s, in0, st));
    a.in = in0;
    a.out = act0;
    a.w = &blob->wf[0][0][0][0];
    a.bias = blob->bias[0];
    T3D_TRY((launch_conv_col<kTcRelu, true>(a, st)));
    a.in = act0;
    a.out = act1;
    a.w = &blob->wf[1][0][0][0];
    a.bias = blob->bias[1];
    T3D_TRY((launch_conv_col<kTcRelu, false>(a, st)));
    a.in = act1;
    a.out = nullptr;
    a.w = &blob->wf[2][0][0][0];
    a.bias = blob->bias[2];
    a.w4 = &blob->w4[0][0];
    a.b4 = blob->b4;
    a.dec32 = reinterpret_cast<uint32_t*>(dec);
    a.logits = logits_out;
    T3D_TRY((launch_conv_col<kTcHead, false>(a, st)));
    return T3D_OK;
}

t3d_status tc_train_forward(int L, int64_t n_samples, int64_t W, const uint64_t* s_prev, const uint64_t* s,
                            const uint64_t* label, const Blob* blob, uint8_t* x0, uint8_t* y1, uint8_t* y2,
                            uint8_t* g3, float* grad_w4, float* grad_b4, float* loss, cudaStream_t st)
{
    T3D_TRY(tc_prepare());
    TcArgs a = base_args(L, n_samples, W);
    T3D_TRY(expand_bits(a, s_prev, s, x0, st));
    a.in = x0;
    a.out = y1;
    a.w = &blob->wf[0][0][0][0];
    a.bias = blob->bias[0];
    T3D_TRY((launch_conv_col<kTcRelu, true>(a, st)));
    a.in = y1;
    a.out = y2;
    a.w = &blob->wf[1][0][0][0];
    a.bias = blob->bias[1];
    T3D_TRY((launch_conv_col<kTcRelu, false>(a, st)));
    a.in = y2;
    a.out = g3;
    a.w = &blob->wf[2][0][0][0];
    a.bias = blob->bias[2];
    a.w4 = &blob->w4[0][0];
    a.b4 = blob->b4;
    a.label = label;
    a.inv_n = 1.0f / (3.0f * (float)a.L3 * (float)n_samples);
    a.grad_w4 = grad_w4;
    a.grad_b4 = grad_b4;
    a.loss = loss;
    T3D_TRY((launch_conv_col<kTcHeadTrain, false>(a, st)));
    return T3D_OK;
}

t3d_status tc_backward_data(int L, int64_t n_samples, const __nv_bfloat16* wt, const uint8_t* g_in,
                            const uint8_t* mask_act, uint8_t* g_out, cudaStream_t st)
{
    T3D_TRY(tc_prepare());
    TcArgs a = base_args(L, n_samples, words_for(n_samples));
    a.in = g_in;
    a.out = g_out;
    a.w = wt;
    a.mask_act = mask_act;
    return launch_conv_col<kTcMask, false>(a, st);
}

t3d_status tc_fill_ones(uint8_t* tile, cudaStream_t st)
{
    k_fill_ones<<<(2048 + 255) / 256, 256, 0, st>>>(reinterpret_cast<uint16_t*>(tile), 2048);
    T3D_LAUNCH_CHECK("ones tile");
    return T3D_OK;
}

t3d_status tc_weight_grad(int L, int64_t n_samples, int x_ch, int cin_kept, const uint8_t* x, const uint8_t* d,
                          const uint8_t* ones, float* gw, float* gb, cudaStream_t st)
{
    T3D_REQUIRE(x_ch == 8 || x_ch == kC, "weight gradient: %d input channels", x_ch);
    T3D_TRY(tc_prepare());
    const int64_t L3 = (int64_t)L * L * L, n_items = tc_padded(n_samples) / kTileM * L3;
    T3D_REQUIRE(n_items <= 0x7fffffffLL, "weight gradient: %lld (sample tile, site) pairs exceed one grid",
                (long long)n_items);
    ProfScope prof(T3D_K_CNN, st);
    WgArgs a;
    std::memset(&a, 0, sizeof(a));
    a.L = L;
    a.L3 = (int)L3;
    a.n_units = n_items / (L * L) * ((L + 1) / 2);
    a.x = x;
    a.d = d;
    a.ones = ones;
    a.cin = cin_kept;
    a.gw = gw;
    a.gb = gb;
    const int grid = (int)std::min<int64_t>(a.n_units, sm_count());
    if (x_ch == 8)
        k_wgrad_tc<8><<<grid, kWgThreads, WgShape<8>::kSmem, st>>>(a);
    else
        k_wgrad_tc<kC><<<grid, kWgThreads, WgShape<kC>::kSmem, st>>>(a);
    T3D_LAUNCH_CHECK("tensor-core weight gradient");
    return T3D_OK;
}

t3d_status tc_set_wait_limit(uint64_t ns)
{
    const unsigned long long v = ns ? (unsigned long long)ns : (unsigned long long)kWaitNs;
    T3D_REQUIRE(v <= kWaitNs, "the wait limit cannot exceed %llu ns", (unsigned long long)kWaitNs);
    T3D_CUDA_CHECK(cudaDeviceSynchronize());
    T3D_CUDA_CHECK(cudaMemcpyToSymbol(g_tc_wait_ns, &v, sizeof(v)));
    return T3D_OK;
}

t3d_status tc_status()
{
    unsigned int flag = 0, zero = 0;
    T3D_CUDA_CHECK(cudaDeviceSynchronize());
    T3D_CUDA_CHECK(cudaMemcpyFromSymbol(&flag, g_tc_error, sizeof(flag)));
    if (flag) {
        T3D_CUDA_CHECK(cudaMemcpyToSymbol(g_tc_error, &zero, sizeof(zero)));
        set_error("a tensor-core pre-decoder kernel gave up a bounded wait");
        return T3D_ETIMEOUT;
    }
    return T3D_OK;
}

}  // namespace cnn
}  // namespace t3d
