// BP with meta-checks (Sec. 4.1, last paragraph: the paper describes them
// and leaves them out of its simulations).  Every error-free syndrome of the
// 3D toric code is a union of closed loops, so the six faces of every unit
// cube have even parity; a cube whose measured faces have odd parity holds an
// odd number of measurement errors.  The factor graph gets one
// measurement-error variable per face (prior log((1-q)/q), degree 3: its
// face and the face's two cubes) and one meta-check per cube over the
// measurement variables of its six faces, with the measured cube parity as
// its syndrome.  Flooding schedule as in Eqs. 1-4: every iteration computes
// all check -> variable messages from the previous iteration's.
//
// Messages are FP32, sample-innermost ([index][sample], samples of a chunk
// padded to whole 64-sample words), double-buffered, 7 planes of 3L^3 rows:
//   F [face][4]   face -> its four edges (the a-edges at r and r + e_b, then
//                 the b-edges at r and r + e_a; a < b the in-plane axes)
//   Fm[face]      face -> its measurement variable
//   Cl[face]      cube at the face's site (the face is its lower face) -> the face's variable
//   Ch[face]      cube one step down along the face's normal (upper face) -> the variable
// One iteration is one kernel over the sites: the faces (inputs: the edge's total -- prior +
// its four face messages -- minus the face's own message, and the measurement variable's
// prior + both cube messages) and the cube (inputs: prior + face message + the other cube's
// message).  Check nodes use
// the plain BP's cancellation-free (t, d = 1 - t) arithmetic (t3d_bp_math.cuh),
// so magnitudes keep FP32 accuracy up to the +-30 clamp.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "t3d_bp_math.cuh"
#include "t3d_device.cuh"
#include "t3d_host.hpp"

namespace t3d {
namespace meta {
namespace {

using bpm::check_node2;

constexpr int kThreads = 128;
constexpr int kWordsPer = kThreads / 32;   // words per block of the iteration kernel
constexpr int kDecideThreads = 256;        // samples per block of the decision kernel
constexpr int64_t kMaxWords = 65535LL * kWordsPer;   // grid y of both kernels
static_assert(kMaxWords * 64 <= 65535LL * kDecideThreads, "the decision kernel's grid");

struct Bufs {
    float* F;     // [3L^3][4][S]
    float* Fm;    // [3L^3][S]
    float* Cl;    // [3L^3][S]
    float* Ch;    // [3L^3][S]
};

struct Args {
    Lattice lat;
    int64_t S;              // padded samples of this chunk (multiple of 64)
    int64_t W;              // row stride of the bit-sliced arrays (words)
    const uint64_t* s;      // measured syndrome, chunk's first word at column 0
    float l0, lq;
    Bufs in, out;
};

// One flooding iteration in one kernel.  A warp takes the three faces and the cube at one site for
// the 64 samples of a word, two samples a lane, so every message row is one 256-byte access: the
// totals of the nine edges its faces touch are summed from their messages on the spot (36 rows,
// of which 12 are the faces' own), and the cube messages a face needs are the ones its cube reads.
// Each message is read from HBM once and written once, 56 bytes per edge and sample; the earlier
// three kernels (edge totals, faces, cubes) wrote and read the totals as well and read the face
// and cube messages twice, 104 bytes.  kFirst: every message in is zero and nothing is read.
// A block takes four words of one site (1 KB runs of a row).  Bound by the latency of those loads, so by
// the warps in flight: 28 per SM (72 registers) since the check nodes pack their inputs' signs.  At
// L = 18, 1,536 samples 12 iterations with the decision took 4.88 ms with the three kernels, 3.57 at 20
// warps (DRAM at 61% of its peak, issue 55%), 3.49 at 24 and 3.43 now (four sites and one word per block
// 3.70 against 3.49 of that time, 256 threads 3.81).
template <bool kFirst>
__global__ void __launch_bounds__(kThreads, 7) k_iteration(const __grid_constant__ Args a)
{
    const Lattice lat = a.lat;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = (int)blockIdx.x;
    const int64_t w = (int64_t)blockIdx.y * kWordsPer + warp;
    if (w * 64 >= a.S) return;
    const int64_t col = w * 64 + 2 * lane;
    const int L3 = lat.L3;
    const Coord c = site_coord(lat, r);
    const int L = lat.L;
    // steps to the neighbours (periodic); site + plus[] or + minus[]
    const int px = c.x[0] + 1 == L ? 1 - L : 1, mx = c.x[0] == 0 ? L - 1 : -1;
    const int py = c.x[1] + 1 == L ? L - lat.L2 : L, my = c.x[1] == 0 ? lat.L2 - L : -L;
    const int pz = c.x[2] + 1 == L ? lat.L2 - lat.L3 : lat.L2, mz = c.x[2] == 0 ? lat.L3 - lat.L2 : -lat.L2;
    const int rx = r + px, ry = r + py, rz = r + pz;

    // row indices stay below 2^28 and a row below 2^32 bytes: one 32 x 32 -> 64-bit product each
    const uint32_t stride = (uint32_t)a.S * 4u;
    auto row = [&](const float* base, int i) {
        return __ldg(reinterpret_cast<const float2*>(reinterpret_cast<const char*>(base + col) + (uint64_t)(uint32_t)i * stride));
    };
    auto put = [&](float* base, int i, float2 v) {
        __stcs(reinterpret_cast<float2*>(reinterpret_cast<char*>(base + col) + (uint64_t)(uint32_t)i * stride), v);
    };
    // message of face (n, q) to its edge j
    auto F = [&](int n, int q, int j) { return row(a.in.F, (n * L3 + q) * 4 + j); };
    auto add = [](float2 u, float2 v) { return __fadd2_rn(u, v); };
    auto sub = [](float2 u, float2 v) { return __ffma2_rn(v, make_float2(-1.0f, -1.0f), u); };
    const float2 l0 = make_float2(a.l0, a.l0), lq = make_float2(a.lq, a.lq);
    auto sum4 = [&](float2 m0, float2 m1, float2 m2, float2 m3) { return add(add(add(add(l0, m0), m1), m2), m3); };
    auto word = [&](int f) { return a.s[(int64_t)f * a.W + w]; };
    auto bit = [&](uint64_t v, int j) { return (bool)((v >> (2 * lane + j)) & 1ULL); };

    // the faces' own messages, requested before the cube's arithmetic
    float2 f[3][4];
#pragma unroll
    for (int n = 0; n < 3; ++n)
#pragma unroll
        for (int j = 0; j < 4; ++j) f[n][j] = kFirst ? make_float2(0.0f, 0.0f) : F(n, r, j);

    // the cube: its lower faces (n, r), whose variable it reaches through Cl, and its upper faces
    // (n, r + e_n), through Ch
    const int up[3] = {rx, ry, rz};
    uint64_t syn[3], par = 0;
    float2 xm[3];   // the faces' measurement-variable inputs
    {
        float2 x[6], o[6];
#pragma unroll
        for (int n = 0; n < 3; ++n) {
            const int fl = n * L3 + r, fu = n * L3 + up[n];
            syn[n] = word(fl);
            par ^= syn[n] ^ word(fu);
            if (kFirst) {
                x[2 * n] = x[2 * n + 1] = xm[n] = lq;
            } else {
                const float2 ch = row(a.in.Ch, fl);
                x[2 * n] = add(add(lq, row(a.in.Fm, fl)), ch);
                x[2 * n + 1] = add(add(lq, row(a.in.Fm, fu)), row(a.in.Cl, fu));
                xm[n] = add(add(lq, row(a.in.Cl, fl)), ch);
            }
        }
        check_node2<6>(x, bit(par, 0), bit(par, 1), o);
#pragma unroll
        for (int n = 0; n < 3; ++n) {
            put(a.out.Cl, n * L3 + r, o[2 * n]);
            put(a.out.Ch, n * L3 + up[n], o[2 * n + 1]);
        }
    }
    // an edge's four faces in the order of edge_slots: x-edge at q (1, q) 0, (1, q - e_z) 1, (2, q) 0,
    // (2, q - e_y) 1; y-edge (0, q) 0, (0, q - e_z) 1, (2, q) 2, (2, q - e_x) 3; z-edge (0, q) 2,
    // (0, q - e_y) 3, (1, q) 2, (1, q - e_x) 3
    auto face = [&](int n, const float2 (&x)[5]) {
        float2 o[5];
        check_node2<5>(x, bit(syn[n], 0), bit(syn[n], 1), o);
#pragma unroll
        for (int j = 0; j < 4; ++j) put(a.out.F, (n * L3 + r) * 4 + j, o[j]);
        put(a.out.Fm, n * L3 + r, o[4]);
    };
    if (kFirst) {
#pragma unroll
        for (int n = 0; n < 3; ++n) {
            const float2 x[5] = {l0, l0, l0, l0, xm[n]};
            face(n, x);
        }
        return;
    }
    const float2 Ty = sum4(f[0][0], F(0, r + mz, 1), f[2][2], F(2, r + mx, 3));
    const float2 Tz = sum4(f[0][2], F(0, r + my, 3), f[1][2], F(1, r + mx, 3));
    {
        const float2 Tyz = sum4(F(0, rz, 0), f[0][1], F(2, rz, 2), F(2, rz + mx, 3));
        const float2 Tzy = sum4(F(0, ry, 2), f[0][3], F(1, ry, 2), F(1, ry + mx, 3));
        const float2 x[5] = {sub(Ty, f[0][0]), sub(Tyz, f[0][1]), sub(Tz, f[0][2]), sub(Tzy, f[0][3]), xm[0]};
        face(0, x);
    }
    const float2 Tx = sum4(f[1][0], F(1, r + mz, 1), f[2][0], F(2, r + my, 1));
    {
        const float2 Txz = sum4(F(1, rz, 0), f[1][1], F(2, rz, 0), F(2, rz + my, 1));
        const float2 Tzx = sum4(F(0, rx, 2), F(0, rx + my, 3), F(1, rx, 2), f[1][3]);
        const float2 x[5] = {sub(Tx, f[1][0]), sub(Txz, f[1][1]), sub(Tz, f[1][2]), sub(Tzx, f[1][3]), xm[1]};
        face(1, x);
    }
    {
        const float2 Txy = sum4(F(1, ry, 0), F(1, ry + mz, 1), F(2, ry, 0), f[2][1]);
        const float2 Tyx = sum4(F(0, rx, 0), F(0, rx + mz, 1), F(2, rx, 2), f[2][3]);
        const float2 x[5] = {sub(Tx, f[2][0]), sub(Txy, f[2][1]), sub(Ty, f[2][2]), sub(Tyx, f[2][3]), xm[2]};
        face(2, x);
    }
}

// The four (face, slot) pairs of edge (d, r): for each normal n != d with third axis
// c, the faces (n, r) and (n, r - e_c); the edge is slot 0 / 1 of them if d < c, else 2 / 3.
__device__ __forceinline__ void edge_slots(const Lattice& lat, int d, int r, int64_t (&f)[4], int (&slot)[4])
{
    const Coord c = site_coord(lat, r);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int n = i == 0 ? (d == 0 ? 1 : 0) : (d == 2 ? 1 : 2);   // the two normals n != d
        const int ax = 3 - d - n;
        const int lo = d < ax ? 0 : 2;
        f[2 * i] = (int64_t)n * lat.L3 + r;
        slot[2 * i] = lo;
        f[2 * i + 1] = (int64_t)n * lat.L3 + site_index(lat, shifted(lat, c, ax, -1));
        slot[2 * i + 1] = lo + 1;
    }
}

// Posteriors and decisions: qubit v: l = prior + its four face messages (a.in.F nullptr: no
// iteration ran, every message is zero); decision words (one ballot per 32 samples) into
// dec[word][site][4] as 32-bit halves; optional posteriors.
__global__ void __launch_bounds__(kDecideThreads) k_decide(const Args a, int64_t n_samples, uint32_t* __restrict__ dec32,
                                                      float* __restrict__ llr, int64_t llr_stride)
{
    const int64_t smp = (int64_t)blockIdx.y * kDecideThreads + threadIdx.x;
    const int64_t v = blockIdx.x;
    const int64_t L3 = a.lat.L3, n = 3 * L3;
    if (smp >= a.S) return;   // S is a multiple of 64: whole warps
    const int d = (int)(v / L3), r = (int)(v % L3);
    float l = a.l0, m = a.lq;
    if (a.in.F) {
        int64_t f[4];
        int slot[4];
        edge_slots(a.lat, d, r, f, slot);
#pragma unroll
        for (int k = 0; k < 4; ++k) l += __ldcs(&a.in.F[(f[k] * 4 + slot[k]) * a.S + smp]);
        if (llr) m = m + __ldcs(&a.in.Fm[v * a.S + smp]) + __ldcs(&a.in.Cl[v * a.S + smp]) + __ldcs(&a.in.Ch[v * a.S + smp]);
    }
    const bool valid = smp < n_samples;
    const uint32_t bits = __ballot_sync(0xffffffffu, valid && l < 0.0f);
    if ((threadIdx.x & 31) == 0) dec32[((smp >> 6) * L3 + r) * 8 + 2 * d + ((smp >> 5) & 1)] = bits;
    if (llr && valid) {
        llr[v * llr_stride + smp] = l;
        llr[(n + v) * llr_stride + smp] = m;
    }
}

// Messages of one iteration in a contiguous buffer of 7 planes of 3 L^3 x S floats.
Bufs split_messages(float* m, int64_t n, int64_t S)
{
    return Bufs{m, m + 4 * n * S, m + 5 * n * S, m + 6 * n * S};
}

// One flooding iteration: every check -> variable message of `out` from those of `in`
// (in.F nullptr: the first iteration, all zero).
t3d_status launch_iteration(Args& a, const Bufs& in, const Bufs& out, cudaStream_t st)
{
    a.in = in;
    a.out = out;
    ProfScope prof(T3D_K_BP_STEP, st);
    const int64_t words = a.S / 64;
    const dim3 grid((unsigned)a.lat.L3, (unsigned)((words + kWordsPer - 1) / kWordsPer));
    if (in.F)
        k_iteration<false><<<grid, kThreads, 0, st>>>(a);
    else
        k_iteration<true><<<grid, kThreads, 0, st>>>(a);
    T3D_LAUNCH_CHECK("meta-check BP iteration");
    return T3D_OK;
}

Args make_args(const Lattice& lat, int64_t S, int64_t W, const uint64_t* s, double p, double q)
{
    Args a;
    std::memset(&a, 0, sizeof(a));
    a.lat = lat;
    a.S = S;
    a.W = W;
    a.s = s;
    a.l0 = (float)std::log((1.0 - p) / p);
    a.lq = (float)std::log((1.0 - q) / q);
    return a;
}

size_t floats_per_sample(int L)
{
    const size_t n = 3ull * L * L * L;
    // two sets of messages, and a plane that nothing reads (the edge totals of a three-kernel iteration): the
    // size that callers ask for, and the smaller ones refused, stay as they were
    return n + 2 * 7 * n /* F, Fm, Cl, Ch x2 */;
}

}  // namespace

size_t bytes_per_word(int L)
{
    return 64 * floats_per_sample(L) * sizeof(float) + (size_t)L * L * L * 32 /* decision words */ + 4096;
}

// BP with meta-checks on n_samples samples (rows of stride W words), in chunks of
// whole words as large as the workspace allows; e ^= d, s ^= H d.
t3d_status launch_bp_meta(const Lattice& lat, int64_t n_samples, int64_t W, uint64_t* e, uint64_t* s, double p,
                          double q, int iters, void* work, size_t work_bytes, float* llr_out, cudaStream_t st)
{
    const int64_t words = words_for(n_samples);
    const int64_t chunk = std::min<int64_t>({words, (int64_t)(work_bytes / bytes_per_word(lat.L)),
                                             kMaxWords});
    T3D_REQUIRE(chunk >= 1, "workspace too small: %zu bytes < %zu per 64-sample word", work_bytes,
                bytes_per_word(lat.L));
    T3D_REQUIRE(llr_out == nullptr || chunk == words, "llr_out needs a workspace for all samples at once");
    const int64_t n = 3LL * lat.L3;
    for (int64_t w0 = 0; w0 < words; w0 += chunk) {
        const int64_t cw = std::min(chunk, words - w0);
        const int64_t S = cw * 64, ns = std::min<int64_t>(S, n_samples - w0 * 64);
        char* base = static_cast<char*>(work);
        auto take = [&](size_t floats) {
            float* ptr = reinterpret_cast<float*>(base);
            base += (floats * sizeof(float) + 255) / 256 * 256;
            return ptr;
        };
        const Bufs b[2] = {split_messages(take(7 * n * S), n, S), split_messages(take(7 * n * S), n, S)};
        uint64_t* dec = reinterpret_cast<uint64_t*>(base);
        Args a = make_args(lat, S, W, s + w0, p, q);
        for (int it = 0; it < iters; ++it)
            T3D_TRY(launch_iteration(a, it ? b[it & 1] : Bufs{nullptr, nullptr, nullptr, nullptr}, b[(it + 1) & 1], st));
        a.in = iters ? b[iters & 1] : Bufs{nullptr, nullptr, nullptr, nullptr};
        ProfScope prof(T3D_K_BP_DECIDE, st);
        k_decide<<<dim3((unsigned)n, (unsigned)((S + kDecideThreads - 1) / kDecideThreads)), kDecideThreads, 0, st>>>(
            a, ns, reinterpret_cast<uint32_t*>(dec), llr_out, n_samples);
        T3D_LAUNCH_CHECK("meta-check BP decisions");
        T3D_TRY(launch_dec_apply(lat, W, cw, dec, e + w0, s + w0, st));
    }
    return T3D_OK;
}

}  // namespace meta
}  // namespace t3d

using namespace t3d;

extern "C" size_t toric3d_bp_meta_workspace_bytes(int L, int64_t chunk_samples)
{
    if (L < 2 || L > 1024 || chunk_samples < 1) return 0;
    return (size_t)words_for(chunk_samples) * meta::bytes_per_word(L);
}

extern "C" size_t toric3d_bp_meta_message_bytes(int L, int64_t n_samples)
{
    if (L < 2 || L > 1024 || n_samples < 1) return 0;
    return (size_t)7 * 3 * L * L * L * 64 * (size_t)words_for(n_samples) * sizeof(float);
}

extern "C" t3d_status toric3d_bp_meta_step(int L, int64_t n_samples, const uint64_t* s, double p, double q,
                                           const float* msg_in, float* msg_out, void* work, size_t work_bytes,
                                           t3d_stream stream)
{
    clear_error();
    T3D_TRY(check_lattice(L));
    T3D_REQUIRE(n_samples >= 1 && words_for(n_samples) <= meta::kMaxWords, "n_samples out of range");
    T3D_TRY(check_words(s, "s"));
    T3D_REQUIRE(p > 0.0 && p < 1.0, "BP needs 0 < p < 1");
    T3D_REQUIRE(q > 0.0 && q < 1.0, "meta-checks need measurement errors: 0 < q < 1");
    T3D_REQUIRE(msg_in != nullptr && msg_out != nullptr && aligned(msg_in, 16) && aligned(msg_out, 16),
                "msg_in and msg_out must be 16-byte aligned device pointers");
    const size_t mb = toric3d_bp_meta_message_bytes(L, n_samples);
    const char *ib = reinterpret_cast<const char*>(msg_in), *ob = reinterpret_cast<const char*>(msg_out);
    T3D_REQUIRE(ib + mb <= ob || ob + mb <= ib, "msg_in and msg_out must not overlap");
    T3D_REQUIRE(work != nullptr && aligned(work, 16) && work_bytes >= mb / 7, "work: >= %zu bytes, 16-byte aligned",
                mb / 7);
    const Lattice lat = make_lattice_host(L);
    const int64_t n = 3LL * lat.L3, S = 64 * words_for(n_samples);
    meta::Args a = meta::make_args(lat, S, words_for(n_samples), s, p, q);
    return meta::launch_iteration(a, meta::split_messages(const_cast<float*>(msg_in), n, S),
                                  meta::split_messages(msg_out, n, S), as_stream(stream));
}

extern "C" t3d_status toric3d_bp_meta(int L, int64_t n_samples, uint64_t* e, uint64_t* s, double p, double q,
                                      int iters, void* work, size_t work_bytes, float* llr_out, t3d_stream stream)
{
    clear_error();
    T3D_TRY(check_lattice(L));
    T3D_REQUIRE(n_samples >= 1 && words_for(n_samples) <= 65535LL * 32, "n_samples out of range");
    T3D_TRY(check_words(e, "e"));
    T3D_TRY(check_words(s, "s"));
    const size_t state = (size_t)3 * L * L * L * (size_t)words_for(n_samples) * 8;
    T3D_REQUIRE(disjoint(e, state, s, state), "e and s must not overlap");
    T3D_REQUIRE(p > 0.0 && p < 1.0, "BP needs 0 < p < 1");
    T3D_REQUIRE(q > 0.0 && q < 1.0, "meta-checks need measurement errors: 0 < q < 1");
    T3D_REQUIRE(iters >= 0, "negative iteration count");
    T3D_REQUIRE(work != nullptr && aligned(work, 256), "work must be a 256-byte aligned device pointer");
    T3D_REQUIRE(llr_out == nullptr || aligned(llr_out, 4), "llr_out must be 4-byte aligned");
    return meta::launch_bp_meta(make_lattice_host(L), n_samples, words_for(n_samples), e, s, p, q, iters, work,
                                work_bytes, llr_out, as_stream(stream));
}
