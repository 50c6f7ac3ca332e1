// Causal form (Eq. 8-15) of bf16 problems with D = M = 32, a warp per piece of a sequence.
//
// The running sums of such a problem are 32 x 33 numbers: a warp holds them in its registers, walks its piece in chunks of
// sixteen positions and needs no other warp.  Every product is mma.sync m16n8k16 (tcgen05 wants 128 rows: at D = 32 that is four
// times as many scores as sums, and a start-up of three chunks per piece).  Operands do not pass through shared memory from lane to lane
// (of the rows only their two weights do, and once per piece the sums are turned there):
//   * Rows arrive and leave in loads and stores of sixteen bytes, the columns in the order of la_warp.cuh.  With the fragments as they
//     lie, pair by pair, the L1 pipe was 70 % busy.
//   * The transposes that sums over positions need come from movmatrix.
//   * The accumulators of the sums, rounded to bf16, are the operand of the next chunk's products as they lie.
// Chunks of sixteen: one diagonal block of scores and no others, and loops of 440 to 620 instructions (twice as many, in chunks of 32, made
// the fetch of the loop, not its issue, set the pace).
//
// What is rounded: features, phi(q) / dn, scores and the copy of the sums that a chunk reads are bf16 operands, each rounded once; the sums, the normaliser
// (its state in fp32 throughout) and everything per row are fp32.  A chunk's sums start from zero and are added with rounding:
// the tensor cores truncate.
//
// What bounds it: two warps on a scheduler and what they wait for of their own instructions (0.56 issued per cycle), then HBM.  The next
// two chunks are on their way to shared memory (cp.async, each lane its own bytes), so that no load is waited for.
// Measured, B128 H8 N784, forward / dQ / dK, dV, us: 45 / 62 / 57 where the kernels with a CTA of four warps per sequence, a chunk of 64
// and tiles in shared memory took 72 / 95 / 129; instructions of a warp per sixteen rows 440 / 620 / 555 for 660 / 950 / 1140.
#pragma once

#include <type_traits>

#include "la_warp.cuh"

namespace la {
namespace warp32 {

using namespace warp;
using sweep::Params;
using sweep::Range;

constexpr int C = 32, NT = C / 8;           // columns of a row, and their tiles
constexpr int RECORD_FLOATS = C * C + C;
using Rows = warp::Rows<C>;
template <int T, bool WEIGHTS> using Ring = warp::Ring<C, T, WEIGHTS>;

// ---- the running sums -------------------------------------------------------------------------------------------
// s[i][n]: rows 16 i + g (+ 8), columns 2 t, 2 t + 1 of tile n of the matrix X^T Y, rows and columns in the order of the tiles
// (or Y^T X); v[n]: the vector at columns 2 t, 2 t + 1 of tile n, the same in every row of lanes.
struct Sums {
    float s[2][NT][4];
    float v[NT][2];

    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int j = 0; j < 4; ++j) s[i][n][j] = 0.f;
#pragma unroll
        for (int n = 0; n < NT; ++n) v[n][0] = v[n][1] = 0.f;
    }
    // s += rows of a^T times rows of b
    __device__ __forceinline__ void add(const Rows& a, const Rows& b) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                float t[4];
                mma_first(t, a.x[0][2 * i], a.x[0][2 * i + 1], a.x[1][2 * i], a.x[1][2 * i + 1], b.x[0][n], b.x[1][n]);
                add_pair(s[i][n][0], s[i][n][1], t[0], t[1]);
                add_pair(s[i][n][2], s[i][n][3], t[2], t[3]);
            }
    }
    // v += sum of the rows of b (transposed)
    __device__ __forceinline__ void add_ones(const Rows& b) {
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            float t[4];
            mma_first(t, kOnes, kOnes, kOnes, kOnes, b.x[0][n], b.x[1][n]);
            add_pair(v[n][0], v[n][1], t[0], t[1]);
        }
    }
    // v += sum of the rows of b times w (w0: rows 2 t, 2 t + 1; w1: 8 + 2 t, ...), w in its three planes: the first two in the
    // upper and the lower eight rows of one operand
    __device__ __forceinline__ void add_weighted(const Rows& b, float2 w0, float2 w1) {
        uint32_t p0[3], p1[3];
        split2<3>(w0.x, w0.y, p0);
        split2<3>(w1.x, w1.y, p1);
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            float t[4];
            mma_first(t, p0[2], 0u, p1[2], 0u, b.x[0][n], b.x[1][n]);
            mma_add(t, p0[0], p0[1], p1[0], p1[1], b.x[0][n], b.x[1][n]);
            add_pair(t[0], t[1], t[2], t[3]);
            add_pair(v[n][0], v[n][1], t[0], t[1]);
        }
    }
    // bf16 pairs of rows 8 r .. 8 r + 7 (lane g: row 8 r + g), columns of tile n
    __device__ __forceinline__ void rounded(uint32_t (&p)[4][NT]) const {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int n = 0; n < NT; ++n) p[r][n] = pack_rn(s[r >> 1][n][(r & 1) * 2], s[r >> 1][n][(r & 1) * 2 + 1]);
    }

    // ... and what that leaves of them
    __device__ __forceinline__ void rounding(uint32_t (&p)[4][NT]) const {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                const float x = s[r >> 1][n][(r & 1) * 2], y = s[r >> 1][n][(r & 1) * 2 + 1];
                const uint32_t w = pack_rn(x, y);
                p[r][n] = pack_rn(x - sm100::bf16_lo(w), y - sm100::bf16_hi(w));
            }
    }

    // Records, in the order of the lanes; the vector in the order of the tensor's columns.
    __device__ __forceinline__ void add_records(const float* rec, int64_t count) {
        const int lane = threadIdx.x & 31, t = lane & 3;
#pragma unroll 2
        for (int64_t r = 0; r < count; ++r) {
            const float4* q = reinterpret_cast<const float4*>(rec + r * RECORD_FLOATS);
            float4 a[8], z[2];
#pragma unroll
            for (int i = 0; i < 8; ++i) a[i] = q[i * 32 + lane];
            z[0] = q[256 + 2 * t];
            z[1] = q[256 + 2 * t + 1];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float (&d)[4] = s[i / NT][i % NT];
                d[0] += a[i].x; d[1] += a[i].y; d[2] += a[i].z; d[3] += a[i].w;
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                v[2 * i][0] += z[i].x; v[2 * i][1] += z[i].y; v[2 * i + 1][0] += z[i].z; v[2 * i + 1][1] += z[i].w;
            }
        }
    }
    __device__ __forceinline__ void put_record(float* rec) const {
        const int lane = threadIdx.x & 31, t = lane & 3;
        float4* q = reinterpret_cast<float4*>(rec);
#pragma unroll
        for (int i = 0; i < 8; ++i) q[i * 32 + lane] = make_float4(s[i / NT][i % NT][0], s[i / NT][i % NT][1], s[i / NT][i % NT][2], s[i / NT][i % NT][3]);
        if (lane < 4)
#pragma unroll
            for (int i = 0; i < 2; ++i) q[256 + 2 * t + i] = make_float4(v[2 * i][0], v[2 * i][1], v[2 * i + 1][0], v[2 * i + 1][1]);
    }
    // the matrix transposed; buf: 4 KB that no lane uses
    __device__ __forceinline__ void turn(float* buf) {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
        auto at = [](int row, int col) { return row * C + (col ^ ((row & 7) << 2)); };
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int j = 0; j < 4; ++j) buf[at(16 * i + 8 * (j >> 1) + g, 8 * n + 2 * t + (j & 1))] = s[i][n][j];
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int j = 0; j < 4; ++j) s[i][n][j] = buf[at(8 * n + 2 * t + (j & 1), 16 * i + 8 * (j >> 1) + g)];
        __syncwarp();
    }
    // The caller's matrix [D][M] and vector [D], in loads and stores of sixteen bytes.  A lane has of s every
    // second one of eight rows, and of the matrix its own two columns of each tile: columns 8 t .. 8 t + 7 of rows 8 (g / 2) + g % 2 + 2 k.
    // TURNED (s holds the matrix transposed): rows and columns change places, and lanes g and g ^ 1 load (store) half a row each and
    // exchange what the other wants.
    static __device__ __forceinline__ int first_row() { const int g = (threadIdx.x & 31) >> 2; return 8 * (g >> 1) + (g & 1); }
    template <bool TURNED> __device__ __forceinline__ void add_state(const float* S, const float* z) {
        const int lane = threadIdx.x & 31, t = lane & 3;
        const bool odd = lane & 4;
        if (S && !TURNED)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4* q = reinterpret_cast<const float4*>(S + (first_row() + 2 * k) * C + 8 * t);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float4 v = q[u];
                    float (&a)[4] = s[k >> 1][2 * u], (&b)[4] = s[k >> 1][2 * u + 1];
                    const int e = (k & 1) * 2;
                    a[e] += v.x; a[e + 1] += v.y; b[e] += v.z; b[e + 1] += v.w;
                }
            }
        if (S && TURNED)
#pragma unroll
            for (int u = 0; u < 8; ++u) {           // element u & 1 of tile u / 2
                const float4 v = *reinterpret_cast<const float4*>(S + (8 * t + u) * C + 8 * (lane >> 3) + (odd ? 4 : 0));
                const float x = __shfl_xor_sync(0xffffffffu, odd ? v.x : v.y, 4), y = __shfl_xor_sync(0xffffffffu, odd ? v.z : v.w, 4);
                const int n = u >> 1, e = u & 1;
                s[0][n][e] += odd ? x : v.x;
                s[0][n][2 + e] += odd ? y : v.z;
                s[1][n][e] += odd ? v.y : x;
                s[1][n][2 + e] += odd ? v.w : y;
            }
        if (z)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float4 w = reinterpret_cast<const float4*>(z + 8 * t)[u];
                v[2 * u][0] += w.x; v[2 * u][1] += w.y; v[2 * u + 1][0] += w.z; v[2 * u + 1][1] += w.w;
            }
    }
    template <bool TURNED> __device__ __forceinline__ void put_state(float* S, float* z) const {
        const int lane = threadIdx.x & 31, t = lane & 3;
        const bool odd = lane & 4;
        if (S && !TURNED)
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float (&a)[4] = s[k >> 1][2 * u], (&b)[4] = s[k >> 1][2 * u + 1];
                    const int e = (k & 1) * 2;
                    reinterpret_cast<float4*>(S + (first_row() + 2 * k) * C + 8 * t)[u] = make_float4(a[e], a[e + 1], b[e], b[e + 1]);
                }
        if (S && TURNED)
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int n = u >> 1, e = u & 1;
                const float a0 = s[0][n][e], a1 = s[0][n][2 + e], a2 = s[1][n][e], a3 = s[1][n][2 + e];
                const float x = __shfl_xor_sync(0xffffffffu, odd ? a0 : a2, 4), y = __shfl_xor_sync(0xffffffffu, odd ? a1 : a3, 4);
                *reinterpret_cast<float4*>(S + (8 * t + u) * C + 8 * (lane >> 3) + (odd ? 4 : 0)) = odd ? make_float4(x, a2, y, a3) : make_float4(a0, x, a1, y);
            }
        if (z && lane < 4)
#pragma unroll
            for (int u = 0; u < 2; ++u) reinterpret_cast<float4*>(z + 8 * t)[u] = make_float4(v[2 * u][0], v[2 * u][1], v[2 * u + 1][0], v[2 * u + 1][1]);
    }
};

// ---- chunks on their way ------------------------------------------------------------------------------------------
// Positions [lo, hi) of the sequence, of them [lo, end) real (la_causal_mma.cu leaves longer sequences to other kernels than
// an int can count).
struct Span {
    int lo, hi, end, piece;
    int64_t bh;
    __device__ __forceinline__ Span(const Params& p, int at) {
        const Range r = sweep::range_of(p, at);
        lo = (int)r.lo; hi = (int)r.hi; end = (int)r.end; piece = at; bh = r.bh;
    }
};

// features of sixteen rows, two at a time
template <bool ELU> __device__ __forceinline__ void map_features(Rows& r) {
    if constexpr (ELU)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int n = 0; n < NT; ++n) r.x[h][n] = tc::phi_pair<true>(r.x[h][n]);
}
// the larger of two bf16 pairs, NaN where one of them is
__device__ __forceinline__ uint32_t max_nan_bf16x2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// phi(q) / dn, rounded once
template <bool ELU> __device__ __forceinline__ void map_weighted(Rows& r, float inv0, float inv1) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const sm100::f32x2 inv = h ? sm100::pair(inv1, inv1) : sm100::pair(inv0, inv0);
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const uint32_t w = r.x[h][n];
            sm100::f32x2 x = sm100::pair_bf16(w);
            if constexpr (ELU) {          // exp(min(x, 0)) + max(x, 0); the square of the exponential of half the number, as phi_pair: the smallest features are kept
                float t0, t1, e0, e1;
                sm100::unpair(sm100::mul2(sm100::pair_bf16(sm100::min_bf16x2(w, 0u)), sm100::pair(0.72134752044448170f, 0.72134752044448170f)), t0, t1);
                asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(t0));
                asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(t1));
                const sm100::f32x2 e = sm100::pair(e0, e1);
                x = sm100::fma2(e, e, sm100::pair_bf16(max_nan_bf16x2(w, 0u)));
            }
            r.x[h][n] = sm100::pack_bf16x2(sm100::mul2(x, inv));
        }
    }
}

// pairs of columns 2 t, 2 t + 1 of an 8 x 8 diagonal block: those up to row g (UPPER: from row g on)
template <bool UPPER> __device__ __forceinline__ uint32_t diagonal_mask() {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const bool lo = UPPER ? 2 * t >= g : 2 * t <= g, hi = UPPER ? 2 * t + 1 >= g : 2 * t + 1 <= g;
    return (lo ? 0xffffu : 0u) | (hi ? 0xffff0000u : 0u);
}

template <typename F> __device__ __forceinline__ float row_sum(const uint32_t (&a)[NT], F b) { return sm100::pair_sum(row_part(a, b)); }
// the lane's bytes of a result's row g; row g + 8 is 512 further
__device__ __forceinline__ uint8_t* rows_at(void* tensor, const Span& r, int64_t N, int n0) {
    return (uint8_t*)tensor + (r.bh * N + n0) * (C * 2) + (threadIdx.x & 31) * 16;
}
__device__ __forceinline__ void put_row(uint8_t* at, int h, const uint32_t (&o)[NT]) {
    *reinterpret_cast<uint4*>(at + h * 512) = make_uint4(o[0], o[1], o[2], o[3]);
}
__device__ __forceinline__ void zero_rows(void* tensor, const Span& r, int64_t N) {
    sweep::zero_rows<32>((__nv_bfloat16*)tensor + r.bh * N * C, r.end, r.hi, C);
}

// ---- forward ------------------------------------------------------------------------------------------------------
template <bool ELU>
__device__ __forceinline__ void forward(const Params& p, uint8_t* smem) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const Span r(p, blockIdx.y);
    uint8_t* O = rows_at(p.O, r, p.N, r.lo);
    float* den = p.den ? p.den + r.bh * p.N : nullptr;
    Ring<3, false> in;
    in.start(smem, r.bh, p.N, r.end, {p.Q, p.K, p.V}, nullptr);
    for (int i = 0; i < in.AHEAD; ++i) in.request(r.lo + i * ROWS);

    Sums st;                // S^T: rows are the columns of V
    st.clear();
    st.add_records(p.rec + r.bh * p.records * (int64_t)RECORD_FLOATS, r.piece);
    st.add_state<true>(p.S0 ? p.S0 + r.bh * C * C : nullptr, p.Z0 ? p.Z0 + r.bh * C : nullptr);
    const uint32_t lower = diagonal_mask<false>();
#pragma unroll 1
    for (int n0 = r.lo; n0 < r.end; n0 += ROWS) {
        const int cn = r.end - n0;              // (of them sixteen at most)
        in.request(n0 + in.AHEAD * ROWS);
        in.arrived(1, r.end - n0, ELU ? kMinusInf : 0u);
        Rows q = in.rows(0), k = in.rows(1);
        const Rows v = in.rows(2);
        map_features<ELU>(q);
        map_features<ELU>(k);
        const Rows vt = transposed(v);
        float o[NT][4], d0, d1;
        {
            uint32_t sb[4][NT];
            st.rounded(sb);
#pragma unroll
            for (int n = 0; n < NT; ++n) columns_mma<true>(o[n], q, [&](int kk, int h) { return sb[n][2 * kk + h]; });
        }
        {
            float s0[4], s1[4], u[4];
            columns_mma<true>(s0, q, [&](int kk, int h) { return k.x[0][2 * kk + h]; });
            columns_mma<true>(s1, q, [&](int kk, int h) { return k.x[1][2 * kk + h]; });
            const uint32_t a0 = pack_rn(s0[0], s0[1]) & lower, a1 = pack_rn(s0[2], s0[3]), a3 = pack_rn(s1[2], s1[3]) & lower;
            mma_first(u, a0, a1, 0u, a3, kOnes, kOnes);            // numerator and normaliser see the same rounded scores
#pragma unroll
            for (int n = 0; n < NT; ++n) mma_add(o[n], a0, a1, 0u, a3, vt.x[0][n], vt.x[1][n]);
            d0 = u[0] + quad_sum(row_sum(q.x[0], [&](int n) { return sm100::pair(st.v[n][0], st.v[n][1]); }));
            d1 = u[2] + quad_sum(row_sum(q.x[1], [&](int n) { return sm100::pair(st.v[n][0], st.v[n][1]); }));
        }
        {
            const Rows kt = transposed(k);
            st.add(vt, kt);
            st.add_ones(kt);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = g + 8 * h;
            const float d = h ? d1 : d0, i = reciprocal(d + p.eps);
            const sm100::f32x2 inv = sm100::pair(i, i);
            uint32_t w[NT];
#pragma unroll
            for (int n = 0; n < NT; ++n) w[n] = sm100::pack_bf16x2(sm100::mul2(sm100::pair(o[n][2 * h], o[n][2 * h + 1]), inv));
            if (row < cn) {
                put_row(O, h, w);
                if (den && t == 0) den[n0 + row] = d;
            }
        }
        in.next();
        O += ROWS * C * 2;
    }
    zero_rows(p.O, r, p.N);
    if (den) sweep::zero_rows<32>(den, r.end, r.hi, 1);
    if (r.piece == p.pieces - 1) st.put_state<true>(p.S1 ? p.S1 + r.bh * C * C : nullptr, p.Z1 ? p.Z1 + r.bh * C : nullptr);
}

// ---- sums of a piece: V^T k, 1^T k ----------------------------------------------------------------------------------
template <bool ELU>
__device__ __forceinline__ void sums(const Params& p, uint8_t* smem) {
    const Span r(p, (int)blockIdx.y + p.first_record);
    if (p.stamp && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *reinterpret_cast<int4*>(p.stamp) = sweep::plan_stamp(p);
    Ring<2, false> in;
    in.start(smem, r.bh, p.N, r.end, {p.K, p.V}, nullptr);
    for (int i = 0; i < in.AHEAD; ++i) in.request(r.lo + i * ROWS);
    Sums st;
    st.clear();
#pragma unroll 1
    for (int n0 = r.lo; n0 < r.end; n0 += ROWS) {
        in.request(n0 + in.AHEAD * ROWS);
        in.arrived(0, r.end - n0, ELU ? kMinusInf : 0u);
        Rows k = in.rows(0);
        const Rows v = in.rows(1);
        map_features<ELU>(k);
        const Rows kt = transposed(k), vt = transposed(v);
        st.add(vt, kt);
        st.add_ones(kt);
        in.next();
    }
    st.put_record(p.rec + (r.bh * p.records + blockIdx.y) * (int64_t)RECORD_FLOATS);
}

// ---- dQ sweep -----------------------------------------------------------------------------------------------------
// REVERSE: and the sums q^^T [G | dl] of the piece, q^ = phi(q) / dn, for the sweep that follows.
template <bool ELU, bool REVERSE>
__device__ __forceinline__ void dq(const Params& p, uint8_t* smem) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    if (p.stamp && sweep::other_plan(p, *reinterpret_cast<const int4*>(p.stamp))) return;
    const Span r(p, blockIdx.y);
    uint8_t* dQ = rows_at(p.dQ, r, p.N, r.lo);
    float* inv_all = p.aux + 2 * r.bh * p.N;         // 1 / dn_i, which every later use of it takes
    float* dl_all = inv_all + p.N;
    Ring<4, false> in;
    in.start(smem, r.bh, p.N, r.end, {p.Q, p.K, p.V, p.G}, nullptr);
    for (int i = 0; i < in.AHEAD; ++i) in.request(r.lo + i * ROWS);

    Sums st;                // S: rows are features
    st.clear();
    if (r.piece > 0) {
        st.add_records(p.rec + r.bh * p.records * (int64_t)RECORD_FLOATS, r.piece);
        st.turn(reinterpret_cast<float*>(smem + in.write));
    }
    Sums back;
    if constexpr (REVERSE) back.clear();
    st.add_state<false>(p.S0 ? p.S0 + r.bh * C * C : nullptr, p.Z0 ? p.Z0 + r.bh * C : nullptr);
    const uint32_t lower = diagonal_mask<false>();
    // The first 64 positions of a sequence go through twice, the second time with the G_i . O_i they found taken off the scores
    // and off the sums' part: where few terms make up a row, h and (q . h / dn) Zc cancel almost entirely (in row 0 completely).  The first
    // 192 have the sums in two bf16 parts: their rounding, once for sixteen positions, is what dQ loses most by where the weights are
    // near-uniform.  dQ's error against 64 bits with 64 / 128 / 192 / 256 positions, inputs scaled by 1/8: B16 H8 N3072 1.83e-2 / 1.79e-2 /
    // 1.76e-2 / 1.73e-2, where tcgen05 chunks of 128 positions have 1.76e-2; B50 H8 N1000 1.79e-2 / 1.73e-2 / 1.69e-2 / 1.66e-2 for 1.71e-2 (the
    // features' own rounding: 1.5e-2).  A step of B128 H8 N784 159.7 / 160.1 / 161.7 / 162.3 us when it was measured.
    constexpr int TWICE = 4 * ROWS, PRECISE = 12 * ROWS;
    auto chunk = [&](int n0, auto first) {
        const bool twice = decltype(first)::value && n0 < TWICE;
        const int cn = r.end - n0;              // (of them sixteen at most)
        in.request(n0 + in.AHEAD * ROWS);
        in.arrived(1, cn, ELU ? kMinusInf : 0u);
        Rows q = in.rows(0), k = in.rows(1);
        const Rows v = in.rows(2), G = in.rows(3);
        map_features<ELU>(q);
        map_features<ELU>(k);
        const Rows kt = transposed(k);
        float c[2] = {0.f, 0.f}, dn[2], inv[2], go[2];          // c: G_i . O_i of rows g, g + 8, as far as it is known
        float h[NT][4], zc[NT][4];
#pragma unroll 1
        for (int pass = twice ? 0 : 1; pass < 2; ++pass) {
            {
                uint32_t sb[4][NT];
                st.rounded(sb);
#pragma unroll
                for (int n = 0; n < NT; ++n) columns_mma<true>(h[n], G, [&](int kk, int i) { return sb[n][2 * kk + i]; });
            }
            float s0[4], s1[4];
            columns_mma<true>(s0, G, [&](int kk, int i) { return v.x[0][2 * kk + i]; });
            columns_mma<true>(s1, G, [&](int kk, int i) { return v.x[1][2 * kk + i]; });
            if constexpr (decltype(first)::value) {
                uint32_t sb[4][NT];
                st.rounding(sb);
#pragma unroll
                for (int n = 0; n < NT; ++n) columns_mma<false>(h[n], G, [&](int kk, int i) { return sb[n][2 * kk + i]; });
            }
            if (twice && pass == 1) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    s0[j] -= c[j >> 1];
                    s1[j] -= c[j >> 1];
#pragma unroll
                    for (int n = 0; n < NT; ++n) h[n][j] = fmaf(-c[j >> 1], st.v[n][j & 1], h[n][j]);
                }
            }
            const uint32_t a0 = pack_rn(s0[0], s0[1]) & lower, a1 = pack_rn(s0[2], s0[3]), a3 = pack_rn(s1[2], s1[3]) & lower;
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                mma_add(h[n], a0, a1, 0u, a3, kt.x[0][n], kt.x[1][n]);
                zc[n][0] = zc[n][2] = st.v[n][0];
                zc[n][1] = zc[n][3] = st.v[n][1];
                mma_add(zc[n], kOnes & lower, kOnes, 0u, kOnes & lower, kt.x[0][n], kt.x[1][n]);
            }
            if (pass == 1) {            // (the sums are not needed any more; their products run beside the row sums)
                st.add(kt, transposed(v));
                st.add_ones(kt);
            }
            float d[2], e[2];
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                d[b] = row_sum(q.x[b], [&](int n) { return sm100::pair(zc[n][2 * b], zc[n][2 * b + 1]); });
                e[b] = row_sum(q.x[b], [&](int n) { return sm100::pair(h[n][2 * b], h[n][2 * b + 1]); });
            }
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                dn[b] = quad_sum(d[b]) + p.eps;
                inv[b] = reciprocal(dn[b]);
                go[b] = (quad_sum(e[b]) - c[b] * p.eps) * inv[b];        // what is left of G_i . O_i
                c[b] += go[b];
            }
        }
        if (REVERSE && r.piece > 0) {
            Rows w = in.rows(0);            // (again: rounded once, as the sweep that takes these sums has its own)
            float i[2], dl[2];
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const bool real = g + 8 * b < cn;           // (rows that are not there may have a normaliser of zero)
                i[b] = real ? inv[b] : 0.f;
                dl[b] = real ? -c[b] : 0.f;
            }
            map_weighted<ELU>(w, i[0], i[1]);
            w = transposed(w);
            back.add(w, transposed(G));
            auto of_row = [&](float x, int row) { return __shfl_sync(0xffffffffu, x, row * 4); };
            back.add_weighted(w, make_float2(of_row(dl[0], 2 * t), of_row(dl[0], 2 * t + 1)), make_float2(of_row(dl[1], 2 * t), of_row(dl[1], 2 * t + 1)));
        }
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const sm100::f32x2 inv2 = sm100::pair(inv[b], inv[b]), go2 = sm100::pair(-go[b], -go[b]);
            uint32_t w[NT];
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                sm100::f32x2 x = sm100::fma2(go2, sm100::pair(zc[n][2 * b], zc[n][2 * b + 1]), sm100::pair(h[n][2 * b], h[n][2 * b + 1]));
                x = sm100::mul2(x, inv2);
                if constexpr (ELU) x = sm100::mul2(x, sm100::pair_bf16(sm100::min_bf16x2(q.x[b][n], kOnes)));
                w[n] = sm100::pack_bf16x2(x);
            }
            if (g + 8 * b < cn) {
                put_row(dQ, b, w);
                if (t == 0) {
                    inv_all[n0 + g + 8 * b] = inv[b];
                    dl_all[n0 + g + 8 * b] = -c[b];
                }
            }
        }
        in.next();
        dQ += ROWS * C * 2;
    };
    int n0 = r.lo;
#pragma unroll 1
    for (; n0 < PRECISE && n0 < r.end; n0 += ROWS) chunk(n0, std::true_type());
#pragma unroll 1
    for (; n0 < r.end; n0 += ROWS) chunk(n0, std::false_type());
    if (REVERSE && r.piece > 0) back.put_record(p.rec_out + (r.bh * p.records + r.piece - 1) * (int64_t)RECORD_FLOATS);
    zero_rows(p.dQ, r, p.N);
}

// ---- sums of a piece: q^^T [G | dl], q^ = phi(q) / dn -----------------------------------------------------------------------
template <bool ELU>
__device__ __forceinline__ void reverse_sums(const Params& p, uint8_t* smem) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const Span r(p, (int)blockIdx.y + p.first_record);
    Ring<2, true> in;
    in.start(smem, r.bh, p.N, r.end, {p.Q, p.G}, p.aux);
    for (int i = 0; i < in.AHEAD; ++i) in.request(r.lo + i * ROWS);
    Sums st;
    st.clear();
#pragma unroll 1
    for (int n0 = r.lo; n0 < r.end; n0 += ROWS) {
        in.request(n0 + in.AHEAD * ROWS);
        in.arrived(0, r.end - n0, ELU ? kMinusInf : 0u);
        Rows q = in.rows(0);
        const Rows G = in.rows(1);
        const float* w = in.weights();
        const float2 l0 = load_pair(w + 16 + 2 * t), l1 = load_pair(w + 24 + 2 * t);
        map_weighted<ELU>(q, w[g], w[g + 8]);
        const Rows qt = transposed(q);
        st.add(qt, transposed(G));
        st.add_weighted(qt, l0, l1);
        in.next();
    }
    st.put_record(p.rec + (r.bh * p.records + blockIdx.y) * (int64_t)RECORD_FLOATS);
}

// ---- dK, dV sweep ---------------------------------------------------------------------------------------------------
template <bool ELU>
__device__ __forceinline__ void dkv(const Params& p, uint8_t* smem) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    if (p.stamp && sweep::other_plan(p, *reinterpret_cast<const int4*>(p.stamp))) return;
    const Span r(p, (int)(gridDim.y - 1 - blockIdx.y));
    const int last = r.lo + (r.end - r.lo - 1) / ROWS * ROWS;           // (an empty piece: its end is its start)
    uint8_t *dK = rows_at(p.dK, r, p.N, last), *dV = rows_at(p.dV, r, p.N, last);
    Ring<4, true> in;
    in.start(smem, r.bh, p.N, r.end, {p.Q, p.K, p.V, p.G}, p.aux);
    auto at = [&](int n0) { return n0 >= r.lo ? n0 : -1; };
    for (int i = 0; i < in.AHEAD; ++i) in.request(at(last - i * ROWS));

    Sums st;                // R: rows are features; record i is the sum of piece i + 1
    st.clear();
    st.add_records(p.rec + (r.bh * p.records + r.piece) * (int64_t)RECORD_FLOATS, p.pieces - 1 - r.piece);
    st.add_state<false>(p.S0 ? p.S0 + r.bh * C * C : nullptr, p.Z0 ? p.Z0 + r.bh * C : nullptr);
    const uint32_t upper = diagonal_mask<true>();
#pragma unroll 1
    for (int n0 = last; n0 >= r.lo && n0 < r.end; n0 -= ROWS) {
        const int cn = r.end - n0;              // (of them sixteen at most)
        in.request(at(n0 - in.AHEAD * ROWS));
        in.arrived(0, r.end - n0, ELU ? kMinusInf : 0u);
        Rows q = in.rows(0), k = in.rows(1);
        const Rows v = in.rows(2), G = in.rows(3);
        const float* w = in.weights();
        const float2 l0 = load_pair(w + 16 + 2 * t), l1 = load_pair(w + 24 + 2 * t);
        map_weighted<ELU>(q, w[g], w[g + 8]);
        map_features<ELU>(k);
        const Rows qt = transposed(q), gt = transposed(G);
        uint32_t rb[4][NT];
        st.rounded(rb);
        {
            float gv[NT][4], s0[4], s1[4];
#pragma unroll
            for (int n = 0; n < NT; ++n) columns_mma<true>(gv[n], k, [&](int kk, int h) { return transposed(rb[2 * kk + h][n]); });
            columns_mma<true>(s0, k, [&](int kk, int h) { return q.x[0][2 * kk + h]; });
            columns_mma<true>(s1, k, [&](int kk, int h) { return q.x[1][2 * kk + h]; });
            const uint32_t a0 = pack_rn(s0[0], s0[1]) & upper, a2 = pack_rn(s1[0], s1[1]), a3 = pack_rn(s1[2], s1[3]) & upper;
#pragma unroll
            for (int n = 0; n < NT; ++n) mma_add(gv[n], a0, 0u, a2, a3, gt.x[0][n], gt.x[1][n]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t o[NT];
#pragma unroll
                for (int n = 0; n < NT; ++n) o[n] = pack_rn(gv[n][2 * h], gv[n][2 * h + 1]);
                if (g + 8 * h < cn) put_row(dV, h, o);
            }
        }
        {
            float gk[NT][4], s0[4] = {l0.x, l0.y, l0.x, l0.y}, s1[4] = {l1.x, l1.y, l1.x, l1.y};
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                gk[n][0] = gk[n][2] = st.v[n][0];
                gk[n][1] = gk[n][3] = st.v[n][1];
                columns_mma<false>(gk[n], v, [&](int kk, int h) { return rb[n][2 * kk + h]; });
            }
            columns_mma<false>(s0, v, [&](int kk, int h) { return G.x[0][2 * kk + h]; });
            columns_mma<false>(s1, v, [&](int kk, int h) { return G.x[1][2 * kk + h]; });
            const uint32_t a0 = pack_rn(s0[0], s0[1]) & upper, a2 = pack_rn(s1[0], s1[1]), a3 = pack_rn(s1[2], s1[3]) & upper;
#pragma unroll
            for (int n = 0; n < NT; ++n) mma_add(gk[n], a0, 0u, a2, a3, qt.x[0][n], qt.x[1][n]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t o[NT];
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    sm100::f32x2 x = sm100::pair(gk[n][2 * h], gk[n][2 * h + 1]);
                    if constexpr (ELU) x = sm100::mul2(x, sm100::pair_bf16(sm100::min_bf16x2(k.x[h][n], kOnes)));
                    o[n] = sm100::pack_bf16x2(x);
                }
                if (g + 8 * h < cn) put_row(dK, h, o);
            }
        }
        st.add(qt, gt);
        st.add_weighted(qt, l0, l1);
        in.next();
        dK -= ROWS * C * 2;
        dV -= ROWS * C * 2;
    }
    zero_rows(p.dK, r, p.N);
    zero_rows(p.dV, r, p.N);
    if (r.piece == 0) st.put_state<false>(p.S1 ? p.S1 + r.bh * C * C : nullptr, p.Z1 ? p.Z1 + r.bh * C : nullptr);
}

}  // namespace warp32
}  // namespace la
