// What the kernels at fp32 accuracy share (la_causal_mma.cu, la_linear_mma.cu): parameters, the running state of a sweep in
// registers and shared memory, operand configurations, and the kernel that sums a range of positions into a record.
#pragma once

#include <atomic>
#include <type_traits>

#include "la_mma.cuh"
#include "la_tc.cuh"
#include "la_tc_common.cuh"

namespace la {
namespace sweep {

using namespace mma;

constexpr int T = 64;
constexpr int STRIPS_T = T / 16;

struct Params {
    const void *Q, *K, *V, *G;
    void *O, *dQ, *dK, *dV;
    float* den;
    const float *S0, *Z0;        // state the sweep starts from (forward: S_in, Z_in; reverse: dS_out, dZ_out), each or null
    float *S1, *Z1;              // where the state it ends with goes (S_out, Z_out / dS_in, dZ_in), each or null
    float* rec;                  // [bh][records][D * M + D]: sums of the pieces first_record .. first_record + records - 1
    int records, first_record;
    float* aux;                  // [bh][2][N]: dn_i (a warp per piece: 1 / dn_i), -G_i . O_i
    const int* lengths;
    int64_t N, piece_len;
    int pieces, heads, D, M, phi;
    int chained;                 // launched as a programmatic dependent of the kernel before it in the stream
    int* stamp;                  // kept sums (or null): the plan they were written under, see plan_stamp()
    int* status;                 // device status word (with stamp)
    float eps;
    int parts;                   // records of a piece (causal sums): its sums in that many ranges
    float* rec_out;              // where the dQ sweep leaves the reverse records, or null
};

// positions [lo, hi) of this CTA's piece, of them [lo, end) real
struct Range { int64_t bh, lo, hi, end; int piece; };
__device__ __forceinline__ Range range_of(const Params& p, int piece) {
    Range r;
    r.bh = blockIdx.x;
    r.piece = piece;
    r.lo = piece * p.piece_len;
    r.hi = r.lo + p.piece_len < p.N ? r.lo + p.piece_len : p.N;
    r.end = r.hi;
    if (p.lengths) {
        const int64_t len = p.lengths[r.bh / p.heads];
        if (len < r.end) r.end = len < r.lo ? r.lo : len;
    }
    return r;
}

// Kept sums start with the plan they were written under.  A backward pass that would cut the sequences in another way
// (la_plan_override() in between) would add up the wrong records: it reports that and writes no gradient.
constexpr int kStampBytes = 16;
__device__ __forceinline__ int4 plan_stamp(const Params& p) {
    return make_int4(0x4c414d4d, p.pieces, (int)(p.piece_len / T), p.D * 256 + p.M);
}
__device__ __forceinline__ bool other_plan(const Params& p, const int4& found) {
    const int4 mine = plan_stamp(p);
    if (found.x == mine.x && found.y == mine.y && found.z == mine.z && found.w == mine.w) return false;
    if (threadIdx.x == 0) atomicOr(p.status, sm100::kStatusPlanMismatch);
    return true;
}

template <int THREADS, typename IO>
__device__ void zero_rows(IO* x, int64_t from, int64_t to, int cols) {       // rows from .. to - 1
    for (int64_t i = from * cols + threadIdx.x; i < to * cols; i += THREADS) x[i] = from_f32<IO>(0.f);
}

// u (16 x 8, the same in every column) += A (16 x 16) v, v = elements k0 .. k0 + 15 of a vector held as three planes of
// LEN elements; smallest partial products first
template <int NX, int LEN>
__device__ __forceinline__ void vector_mma(float (&u)[4], const uint32_t (&a)[NX][4], const uint16_t* pl, int k0, int t) {
    uint32_t w[3][2];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        w[k][0] = *reinterpret_cast<const uint32_t*>(pl + k * LEN + k0 + 2 * t);
        w[k][1] = *reinterpret_cast<const uint32_t*>(pl + k * LEN + k0 + 8 + 2 * t);
    }
#pragma unroll
    for (int sum = 2; sum >= 0; --sum)
#pragma unroll
        for (int k = 0; k < NX; ++k)
            if (sum - k >= 0) mma16816(u, a[k], w[sum - k][0], w[sum - k][1]);
}

// The running sums of a warp: rows d = 16 strip + g (+ 8), columns e = 8 (n0 + n) + 2 t (+ 1).  The warps share the DP / 16
// strips out among them: several strips a warp, or several warps a strip with a part of its columns each (at least
// sixteen: with D = M = 32 and eight warps four of them have none).
template <int DP, int MP, int WARPS>
struct State {
    static constexpr int STRIPS = DP / 16, WANT = STRIPS < WARPS ? WARPS / STRIPS : 1;
    static constexpr int SHARE = WANT < MP / 16 ? WANT : MP / 16, SD = STRIPS < WARPS ? 1 : STRIPS / WARPS;
    static constexpr int NC = MP / 8 / SHARE;
    static constexpr bool ALL = STRIPS * SHARE >= WARPS;
    static __device__ __forceinline__ bool owner() { return ALL || ((int)threadIdx.x >> 5) < STRIPS * SHARE; }
    static __device__ __forceinline__ int strip(int i) { return ((int)threadIdx.x >> 5) % STRIPS + WARPS * i; }
    static __device__ __forceinline__ int n0() { return SHARE == 1 ? 0 : ((int)threadIdx.x >> 5) / STRIPS * NC; }
    float s[SD][NC][4];
    float z[SD][2];             // in every warp that shares the strip

    __device__ __forceinline__ void init(const Params& p, const float* S0, const float* Z0, const float* rec, int nrec) {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, c0 = n0();
        const int size = p.D * p.M + p.D;
        if (!owner()) return;
#pragma unroll
        for (int i = 0; i < SD; ++i) {
            const int d = strip(i) * 16 + g;
#pragma unroll
            for (int n = 0; n < NC; ++n)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float2 v = make_float2(0.f, 0.f);
                    if (S0 && d + 8 * h < p.D && (c0 + n) * 8 < p.M) v = load_pair(S0 + (d + 8 * h) * p.M + (c0 + n) * 8 + 2 * t);
                    s[i][n][2 * h] = v.x;
                    s[i][n][2 * h + 1] = v.y;
                }
#pragma unroll
            for (int h = 0; h < 2; ++h) z[i][h] = Z0 && d + 8 * h < p.D ? Z0[d + 8 * h] : 0.f;
#pragma unroll 4
            for (int r = 0; r < nrec; ++r) {        // (several records in flight)
                const float* q = rec + (int64_t)r * size;
#pragma unroll
                for (int n = 0; n < NC; ++n)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if (d + 8 * h < p.D && (c0 + n) * 8 < p.M) {
                            const float2 v = *reinterpret_cast<const float2*>(q + (d + 8 * h) * p.M + (c0 + n) * 8 + 2 * t);
                            s[i][n][2 * h] += v.x;
                            s[i][n][2 * h + 1] += v.y;
                        }
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (d + 8 * h < p.D) z[i][h] += q[p.D * p.M + d + 8 * h];
            }
        }
    }
    __device__ __forceinline__ void write(const Params& p, float* S1, float* Z1) const {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, c0 = n0();
        if (!owner()) return;
#pragma unroll
        for (int i = 0; i < SD; ++i) {
            const int d = strip(i) * 16 + g;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (d + 8 * h < p.D) {
#pragma unroll
                    for (int n = 0; n < NC; ++n)
                        if (S1 && (c0 + n) * 8 < p.M) store_pair<float>(S1 + (d + 8 * h) * p.M + (c0 + n) * 8 + 2 * t, s[i][n][2 * h], s[i][n][2 * h + 1]);
                    if (Z1 && t == 0 && c0 == 0) Z1[d + 8 * h] = z[i][h];
                }
        }
    }
    // the operand planes [DP][MP] of the matrix; the vector in fp32 and as three planes of DP elements
    template <int NS>
    __device__ __forceinline__ void publish(uint8_t* tile, float* vec, uint16_t* vpl) const {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, c0 = n0();
        if (!owner()) return;
#pragma unroll
        for (int i = 0; i < SD; ++i) {
            const int d = strip(i) * 16 + g;
#pragma unroll
            for (int n = 0; n < NC; ++n)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t o[NS];
                    split2<NS>(s[i][n][2 * h], s[i][n][2 * h + 1], o);
#pragma unroll
                    for (int k = 0; k < NS; ++k)
                        *reinterpret_cast<uint32_t*>(tile + k * (DP * MP * 2) + tile_at<MP>(d + 8 * h, c0 + n) + t * 4) = o[k];
                }
            if (t == 0 && c0 == 0) {
                uint32_t o[3];
                split2<3>(z[i][0], z[i][1], o);
                vec[d] = z[i][0];
                vec[d + 8] = z[i][1];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    vpl[k * DP + d] = (uint16_t)o[k];
                    vpl[k * DP + d + 8] = (uint16_t)(o[k] >> 16);
                }
            }
        }
    }
    // s += X^T Y, z += X^T w over the rows of the tiles X [ROWS][DP] (NX planes), Y [ROWS][MP] (NY);
    // w: ones, or the vector whose three planes of ROWS elements are at wpl
    // (a chunk that is not full has zeros in the tiles' other rows)
    template <int NX, int NY, bool ONES, int ROWS = T>
    __device__ __forceinline__ void update(uint32_t X, uint32_t Y, const uint16_t* wpl) {
        const int lane = threadIdx.x & 31, t = lane & 3, c0 = n0();
        if (!owner()) return;
#pragma unroll
        for (int i = 0; i < SD; ++i) {
            uint32_t a[ROWS / 16][NX][4];
            float zs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int b = 0; b < ROWS / 16; ++b) {
                load_rows_t<NX, DP>(a[b], X, ROWS * DP * 2, b * 16, strip(i) * 2, lane);
                float u[4] = {0.f, 0.f, 0.f, 0.f};
                if constexpr (ONES) {
#pragma unroll
                    for (int k = NX - 1; k >= 0; --k) mma16816(u, a[b][k], 0x3f803f80u, 0x3f803f80u);
                } else {
                    vector_mma<NX, ROWS>(u, a[b], wpl, b * 16, t);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) zs[j] += u[j];
            }
            z[i][0] += zs[0];
            z[i][1] += zs[2];
#pragma unroll
            for (int n = 0; n < NC / 2; ++n) {
                Chain c;
#pragma unroll
                for (int b = 0; b < ROWS / 16; ++b) {
                    uint32_t y[NY][4];
                    load_cols_t<NY, MP>(y, Y, ROWS * MP * 2, b * 16, c0 + n * 2, lane);
                    c.step<NX, NY>(a[b], y);
                }
                c.add_to(s[i][2 * n], s[i][2 * n + 1]);
            }
        }
    }
};

// I/O type and planes of each kind of operand: feature-mapped rows (NQ), value rows V, G (NV), scores (NP), state (NS),
// q / dn (NR).  Everything computed in fp32 has three planes; bf16 values, and features that are bf16 as given, one.
struct Fp32 {
    using IO = float;
    static constexpr int NQ = 3, NV = 3, NP = 3, NS = 3, NR = 3, WPS = 2;
    static constexpr bool MAPPED = true, ALONE = false;
};
struct Bf16Wide {
    using IO = __nv_bfloat16;
    static constexpr int NQ = 3, NV = 1, NP = 3, NS = 3, NR = 3, WPS = 2;
    static constexpr bool MAPPED = true, ALONE = false;
};
struct Bf16Features {
    using IO = __nv_bfloat16;
    static constexpr int NQ = 1, NV = 1, NP = 3, NS = 3, NR = 3, WPS = 2;
    static constexpr bool MAPPED = false, ALONE = false;
};
// ... with one warp per strip, at twice the registers: where a machine full of CTAs keeps the schedulers busy anyway, the
// hand-overs cost more than they give.  Forward + backward, us, one / two warps: fp32 B32 H8 N4096 D64 2690 / 2930,
// B4 H8 N4096 477 / 472; Fourier B8 H8 N1000 C128 272 / 288.  (The smallest grids run the kernels that follow or clusters.)
struct Fp32One : Fp32 { static constexpr int WPS = 1; };
struct Bf16FeaturesOne : Bf16Features { static constexpr int WPS = 1; };
// ... and with an SM to itself: a grid of at most 148 CTAs has that anyway, and the backward kernels then have 255 registers
// instead of 128 and up to 2.2 KB spilled.  Forward + backward, us, before / after: Fourier B1 H8 N4000 C128 282 / 234, B3 H8
// N2666 341 / 327; fp32 D = 64 B1 H8 N2000 110 / 100, B16 H8 N100 67 / 59 (but 160 CTAs, B20 H8 N99, 95 / 100).
struct Fp32Alone : Fp32 { static constexpr bool ALONE = true; };
struct Bf16FeaturesAlone : Bf16Features { static constexpr bool ALONE = true; };
// bf16 operands throughout (with fp32 sums), as the tcgen05 kernels have them (la_cluster.cu)
struct Bf16 {
    using IO = __nv_bfloat16;
    static constexpr int NQ = 1, NV = 1, NP = 1, NS = 1, NR = 1, WPS = 1;
    static constexpr bool MAPPED = true, ALONE = false;
};

// Shared memory: tiles X [T][DP] and Y [T][MP]; with two warps per strip the tile that holds the strips' own operand
// (RC columns, NRW planes); the state planes, later the partial results of the strips (EX columns); the vectors.
template <int WPS, int DP, int MP, int NX, int NY, int NRW, int RC, int NS, int EX> struct Layout {
    static constexpr int X = 0, Y = X + NX * T * DP * 2, R = Y + NY * T * MP * 2, S = R + (WPS == 2 ? NRW * T * RC * 2 : 0),
                         PLANES = NS * DP * MP * 2, PART = WPS == 2 ? T * EX * 4 : 0,
                         Z = S + (PLANES > PART ? PLANES : PART), ZP = Z + DP * 4, W = ZP + 3 * DP * 2, WP = W + T * 4,
                         BYTES = (WP + 3 * T * 2 + 127) / 128 * 128;
};
// Where q and G are bf16 and q / dn and G / dn need three planes, the division goes to G, of which there are fewer columns, and in the
// reverse scores to their columns: (k q^T) / dn, ((G V^T + dl) / dn) q instead of k (q / dn)^T, (G V^T + dl) (q / dn).  Per sixteen
// keys and queries that is 96 products where it was 176.  Fourier B8 H8 N1000 C128 dK and dV 84 -> 77 us.
template <typename C> constexpr bool kScaled = C::NQ == 1 && C::NV == 1 && C::NR == 3;
// (all but 128 features by 64 columns have one record of a piece: known when compiled, it is 1 to 4 % of a step of a small grid)
template <typename C, bool EXACT> __device__ __forceinline__ int parts_of(const Params& p) { return kScaled<C> && EXACT ? p.parts : 1; }
template <typename C, int DP, int MP, bool REVERSE>
using SumLayout = Layout<1, DP, MP, REVERSE && !kScaled<C> ? C::NR : C::NQ, REVERSE && kScaled<C> ? C::NR : C::NV, 0, 0, 0, 0>;

template <typename C> constexpr int kThreads = 128 * C::WPS;
// CTAs of an SM that the registers are shared out for: as many as shared memory holds, at most two (or `most`)
template <typename Sh> constexpr int resident(int most = 2) {
    const int fit = 227 * 1024 / (Sh::BYTES + 1024);
    return fit < most ? fit : most;
}

template <int NT8> __device__ __forceinline__ void clear(float (&x)[NT8][4]) {
#pragma unroll
    for (int n = 0; n < NT8; ++n)
#pragma unroll
        for (int j = 0; j < 4; ++j) x[n][j] = 0.f;
}

// rows n0 .. n0 + T - 1, those before `end`, on their way to L2
template <typename C, typename IO>
__device__ __forceinline__ void prefetch_rows(const IO* x, int64_t n0, int64_t end, int cols) {
    constexpr int THREADS = kThreads<C>;
    if (n0 < 0 || n0 >= end) return;
    const int64_t rows = end - n0 < T ? end - n0 : T;
    const char* p = reinterpret_cast<const char*>(x + n0 * cols);
    for (int64_t o = threadIdx.x * 128; o < rows * cols * (int64_t)sizeof(IO); o += THREADS * 128) prefetch_l2(p + o);
}

// feature-mapped pairs in registers: bf16 where features have one plane
template <int NQ> struct FeatureType { using type = float; };
template <> struct FeatureType<1> { using type = __nv_bfloat16; };

// ---- sums over a piece: the forward records [k^T V | k^T 1], or the reverse ones [q^^T G | q^^T dl] -----------------
// Reverse tiles: q^ = phi(Q) / dn and the planes of dl, from the parked dn_i, dl_i.
template <typename IO, int DP, int MP, int THREADS>
struct ReverseRows {
    RawTile<IO, T, DP, THREADS> rq;
    RawTile<IO, T, MP, THREADS> rg;
    float inv[RawTile<IO, T, DP, THREADS>::GROUPS];
    float dl;
    __device__ __forceinline__ void load(const IO* Q, const IO* G, const float* dn, const float* delta, int64_t n0, int cn, int D, int M,
                                         float pad) {
        rq.load(Q + n0 * D, cn, D, pad);
        rg.load(G + n0 * M, cn, M, 0.f);
#pragma unroll
        for (int u = 0; u < RawTile<IO, T, DP, THREADS>::GROUPS; ++u) {
            const int row = ((int)threadIdx.x + u * THREADS) / (DP / 8);
            inv[u] = row < cn ? dn[n0 + row] : 1.f;
        }
        dl = (int)threadIdx.x < cn ? delta[n0 + threadIdx.x] : 0.f;
    }
    template <int NR, int NV>
    __device__ __forceinline__ void store(uint8_t* tq, uint8_t* tg, float* w, uint16_t* wpl, int phi) {
#pragma unroll
        for (int u = 0; u < RawTile<IO, T, DP, THREADS>::GROUPS; ++u) inv[u] = 1.f / inv[u];
        with_phi<NR>(phi, [&](auto f) { rq.template store<NR>(tq, [&](int u, float x) { return f(x) * inv[u]; }); });
        rg.template values<NV>(tg);
        if (threadIdx.x < T) {
            w[threadIdx.x] = dl;
            uint32_t o[3];
            split2<3>(dl, 0.f, o);
#pragma unroll
            for (int k = 0; k < 3; ++k) wpl[k * T + threadIdx.x] = (uint16_t)o[k];
        }
    }
};

// The same for kScaled: q and (tg, if given) G as they are, G / dn in three planes, the planes of dl / dn; dl and 1 / dn in fp32.
template <typename IO, int DP, int MP, int THREADS>
struct ScaledRows {
    RawTile<IO, T, DP, THREADS> rq;
    RawTile<IO, T, MP, THREADS> rg;
    float inv[RawTile<IO, T, MP, THREADS>::GROUPS];
    float dl, dn;
    __device__ __forceinline__ void load(const IO* Q, const IO* G, const float* dns, const float* delta, int64_t n0, int cn, int D, int M, float) {
        rq.load(Q + n0 * D, cn, D, 0.f);
        rg.load(G + n0 * M, cn, M, 0.f);
#pragma unroll
        for (int u = 0; u < RawTile<IO, T, MP, THREADS>::GROUPS; ++u) {
            const int row = ((int)threadIdx.x + u * THREADS) / (MP / 8);
            inv[u] = row < cn ? dns[n0 + row] : 1.f;
        }
        dl = (int)threadIdx.x < cn ? delta[n0 + threadIdx.x] : 0.f;
        dn = (int)threadIdx.x < cn ? dns[n0 + threadIdx.x] : 1.f;
    }
    __device__ __forceinline__ void store(uint8_t* tq, uint8_t* tg, uint8_t* th, float* w, float* winv, uint16_t* wpl) {
#pragma unroll
        for (int u = 0; u < RawTile<IO, T, MP, THREADS>::GROUPS; ++u) inv[u] = 1.f / inv[u];
        rq.copy(tq);
        if (tg) rg.copy(tg);
        rg.template store<3>(th, [&](int u, float x) { return x * inv[u]; });
        if (threadIdx.x < T) {
            const float i = 1.f / dn;
            w[threadIdx.x] = dl;
            if (winv) winv[threadIdx.x] = i;
            uint32_t o[3];
            split2<3>(dl * i, 0.f, o);
#pragma unroll
            for (int k = 0; k < 3; ++k) wpl[k * T + threadIdx.x] = (uint16_t)o[k];
        }
    }
};

template <typename C, int DP, int MP, bool EXACT, bool REVERSE>
__global__ void __launch_bounds__(kThreads<C>, 2)
causal_mma_sum_kernel(const Params p) {
    using IO = typename C::IO;
    using Sh = SumLayout<C, DP, MP, REVERSE>;
    constexpr bool SCALED = REVERSE && kScaled<C>;
    constexpr int NX = REVERSE && !SCALED ? C::NR : C::NQ, NY = SCALED ? C::NR : C::NV, THREADS = kThreads<C>;
    extern __shared__ __align__(128) uint8_t smem[];
    const int D = EXACT ? DP : p.D, M = EXACT ? MP : p.M, phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    wait_for_stream();
    release_next();
    const int parts = parts_of<C, EXACT>(p);
    Range r = range_of(p, (int)blockIdx.y / parts + p.first_record);
    if (parts > 1) {            // the CTA's part of the piece
        const int64_t chunks = (r.hi - r.lo + T - 1) / T, each = (chunks + parts - 1) / parts * T, lo = r.lo + (int)blockIdx.y % parts * each;
        r.lo = lo < r.hi ? lo : r.hi;
        if (r.lo + each < r.hi) r.hi = r.lo + each;
        r.end = r.end < r.lo ? r.lo : r.end < r.hi ? r.end : r.hi;
    }
    const IO* X = (const IO*)(REVERSE ? p.Q : p.K) + r.bh * p.N * D;
    const IO* Y = (const IO*)(REVERSE ? p.G : p.V) + r.bh * p.N * M;
    const float* dn = REVERSE ? p.aux + r.bh * 2 * p.N : nullptr;
    const float* delta = REVERSE ? dn + p.N : nullptr;
    float* w = reinterpret_cast<float*>(smem + Sh::W);
    uint16_t* wpl = reinterpret_cast<uint16_t*>(smem + Sh::WP);
    if (!REVERSE && p.stamp && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *reinterpret_cast<int4*>(p.stamp) = plan_stamp(p);
    struct ForwardRows {
        RawTile<IO, T, DP, THREADS> rx;
        RawTile<IO, T, MP, THREADS> ry;
    };
    // bf16 rows of a chunk are requested before the products of the one before (fp32 ones have no registers for that)
    constexpr bool AHEAD = sizeof(IO) == 2 && C::WPS == 2;
    std::conditional_t<SCALED, ScaledRows<IO, DP, MP, THREADS>, std::conditional_t<REVERSE, ReverseRows<IO, DP, MP, THREADS>, ForwardRows>> rows;
    auto load = [&](int64_t n0) {
        const int cn = (int)(r.end - n0 < T ? r.end - n0 : T);
        if constexpr (REVERSE) {
            rows.load(X, Y, dn, delta, n0, cn, D, M, pad);
        } else {
            rows.rx.load(X + n0 * D, cn, D, pad);
            rows.ry.load(Y + n0 * M, cn, M, 0.f);
        }
    };
    if (AHEAD && r.lo < r.end) load(r.lo);
    State<DP, MP, 4 * C::WPS> st;
    st.init(p, nullptr, nullptr, nullptr, 0);
    for (int64_t n0 = r.lo; n0 < r.end; n0 += T) {
        if constexpr (!AHEAD) {
            load(n0);
            __syncthreads();        // the planes of the chunk before are no longer read
        }
        if constexpr (SCALED) rows.store(smem + Sh::X, nullptr, smem + Sh::Y, w, nullptr, wpl);
        else if constexpr (REVERSE) rows.template store<NX, NY>(smem + Sh::X, smem + Sh::Y, w, wpl, phi);
        else {
            rows.rx.template features<NX>(smem + Sh::X, phi);
            rows.ry.template values<NY>(smem + Sh::Y);
        }
        if constexpr (!AHEAD) {
            prefetch_rows<C>(X, n0 + T, r.end, D);
            prefetch_rows<C>(Y, n0 + T, r.end, M);
        }
        __syncthreads();
        if constexpr (AHEAD) {
            if (n0 + T < r.end) load(n0 + T);
            prefetch_rows<C>(X, n0 + 2 * T, r.end, D);
            prefetch_rows<C>(Y, n0 + 2 * T, r.end, M);
        }
        st.template update<NX, NY, !REVERSE>(smem_u32(smem + Sh::X), smem_u32(smem + Sh::Y), wpl);
        if constexpr (AHEAD) __syncthreads();
    }
    float* dst = p.rec + (r.bh * p.records + blockIdx.y) * (int64_t)(D * M + D);
    st.write(p, dst, dst + D * M);
}

template <auto KERNEL>
inline int launch(ProfKernel prof, int threads, unsigned bh, unsigned y, int smem, const Params& a, cudaStream_t st) {
    static std::atomic<uint64_t> opted_in{0};           // devices on which the kernel may use that much shared memory
    if (smem > 48 * 1024)
        if (int rc = tc::opt_in_smem_once(KERNEL, (uint32_t)smem, opted_in)) return rc;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(bh, y);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = a.chained ? 1 : 0;
    prof_begin(prof, st);
    LA_CUDA_TRY(cudaLaunchKernelEx(&cfg, KERNEL, a));
    note_launch();
    prof_end(prof, st);
    return LA_OK;
}

}  // namespace sweep
}  // namespace la
