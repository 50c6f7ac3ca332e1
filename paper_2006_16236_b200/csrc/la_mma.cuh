// Products at fp32 accuracy on the warp-level tensor instructions (mma.sync m16n8k16, bf16 operands, fp32 sums).
//
// An fp32 number is the exact sum of three bf16 numbers: x = x0 + x1 + x2 with x0 = x rounded to bf16, x1 the next
// eight bits and x2 what is left of the 24-bit significand.  A product of two such numbers keeps the six partial
// products x_i y_j with i + j <= 2; the three that are dropped are below 2^-24 of it.  An operand that is bf16 to
// begin with has one plane, so its products cost three instructions (against a three-plane operand) or one.
//
// The tensor cores round their running sums toward zero (measured: 1 + 0.75 ulp stays 1).  Every 16-term block
// therefore starts from zero, smallest partial products first, and is added to the running sum with an ordinary
// round-to-nearest addition: no truncation accumulates over a sum.
//
// Why these instructions and not tcgen05: three planes of every operand of one chunk (Q, K, V, G and the state) do
// not fit shared memory beside each other at the 128-row tiles tcgen05 wants, the score blocks would have to go out
// to shared or tensor memory in three planes, and half of a triangular block would be multiplied for nothing.
// From registers, blocks right of the diagonal are skipped at a grain of 16 and the scores of a row strip turn
// into the operand of the next product without leaving the warp.
#pragma once

#include "la_common.cuh"
#include "la_tc_common.cuh"

namespace la {
namespace mma {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// four 8x8 bf16 matrices; lane i of each group of eight gives the address of row i of its matrix
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// acc0 | acc1 (16 x 16) += A (16 x 16, NA planes) B (16 x 16, NB planes; registers 0,1: columns 0..7, 2,3: 8..15)
template <int NA, int NB>
__device__ __forceinline__ void block_mma(float (&acc0)[4], float (&acc1)[4], const uint32_t (&a)[NA][4],
                                          const uint32_t (&b)[NB][4]) {
    if constexpr (NA == 1 && NB == 1) {
        mma16816(acc0, a[0], b[0][0], b[0][1]);
        mma16816(acc1, a[0], b[0][2], b[0][3]);
        return;
    }
    float t0[4] = {0.f, 0.f, 0.f, 0.f}, t1[4] = {0.f, 0.f, 0.f, 0.f};
    constexpr int top = NA + NB - 2 < 2 ? NA + NB - 2 : 2;
#pragma unroll
    for (int s = top; s >= 0; --s)
#pragma unroll
        for (int i = 0; i < NA; ++i)
            if (s - i >= 0 && s - i < NB) {
                mma16816(t0, a[i], b[s - i][0], b[s - i][1]);
                mma16816(t1, a[i], b[s - i][2], b[s - i][3]);
            }
#pragma unroll
    for (int j = 0; j < 4; ++j) { acc0[j] += t0[j]; acc1[j] += t1[j]; }
}

// The same for longer sums: the partial products of the leading planes and all the others run in two chains (the
// others are below 2^-8 of the first: truncating the long sum is done once per step, not once per instruction).
struct Chain {
    float hi0[4] = {0.f, 0.f, 0.f, 0.f}, hi1[4] = {0.f, 0.f, 0.f, 0.f}, lo0[4] = {0.f, 0.f, 0.f, 0.f}, lo1[4] = {0.f, 0.f, 0.f, 0.f};
    template <int NA, int NB>
    __device__ __forceinline__ void step(const uint32_t (&a)[NA][4], const uint32_t (&b)[NB][4]) {
        constexpr int top = NA + NB - 2 < 2 ? NA + NB - 2 : 2;
        mma16816(hi0, a[0], b[0][0], b[0][1]);
        mma16816(hi1, a[0], b[0][2], b[0][3]);
#pragma unroll
        for (int s = top; s >= 1; --s)
#pragma unroll
            for (int i = 0; i < NA; ++i)
                if (s - i >= 0 && s - i < NB) {
                    mma16816(lo0, a[i], b[s - i][0], b[s - i][1]);
                    mma16816(lo1, a[i], b[s - i][2], b[s - i][3]);
                }
    }
    __device__ __forceinline__ void add_to(float (&acc0)[4], float (&acc1)[4]) const {
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc0[j] += hi0[j] + lo0[j]; acc1[j] += hi1[j] + lo1[j]; }
    }
    __device__ __forceinline__ void put(float (&acc0)[4], float (&acc1)[4]) const {
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc0[j] = hi0[j] + lo0[j]; acc1[j] = hi1[j] + lo1[j]; }
    }
};

// x, y -> NP planes of packed pairs (x in the low half)
__device__ __forceinline__ uint32_t pack_rn(float x, float y) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(y), "f"(x));
    return r;
}
__device__ __forceinline__ uint32_t pack_rn_finite(float x, float y) {        // numbers beyond the largest bf16 become that
    uint32_t r;
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(y), "f"(x));
    return r;
}
template <int NP>
__device__ __forceinline__ void split2(float x, float y, uint32_t (&p)[NP]) {
    if constexpr (NP == 1) {
        p[0] = pack_rn(x, y);
    } else {
        // (finite: an fp32 number above 3.39e38 keeps its value, the rest of it in plane 1; an infinity becomes a NaN)
        p[0] = pack_rn_finite(x, y);
        // (both differences are exact; the rounding of plane 0 leaves planes 1 and 2 with a sign of their own, so
        // that the dropped partial products have no common sign and truncating them costs no bias)
        const float rx = x - __uint_as_float(p[0] << 16), ry = y - __uint_as_float(p[0] & 0xffff0000u);
        p[1] = __byte_perm(__float_as_uint(rx), __float_as_uint(ry), 0x7632);
        const float sx = rx - __uint_as_float(p[1] << 16), sy = ry - __uint_as_float(p[1] & 0xffff0000u);
        p[2] = __byte_perm(__float_as_uint(sx), __float_as_uint(sy), 0x7632);
    }
}
// A bf16 plane of a shared-memory tile: rows of C columns, the 16-byte group c of row r stored at c ^ (r & 7), so
// that the eight rows of an ldmatrix fall into different banks (C = 32: two rows per 128 bytes, at c ^ (r / 2 & 3)).
template <int C> __device__ __forceinline__ uint32_t tile_at(int row, int group) {
    if constexpr (C == 32) return (uint32_t)(row * 64 + ((group ^ ((row >> 1) & 3)) << 4));
    return (uint32_t)(row * (C * 2) + ((group ^ (row & 7)) << 4));
}

// Lane address patterns of a 16 x 16 block (row, group of eight columns) inside a tile:
//   Rows: the tile's rows are the rows/columns of the operand (B[n][k] as it lies; A^T[k][m] with .trans)
//   Cols: the tile's rows are the k index (B[k][n] with .trans) or the rows of A (as it lies)
__device__ __forceinline__ int rows_row(int lane) { return (lane & 7) + ((lane >> 4) << 3); }
__device__ __forceinline__ int rows_grp(int lane) { return (lane >> 3) & 1; }
__device__ __forceinline__ int cols_row(int lane) { return lane & 15; }
__device__ __forceinline__ int cols_grp(int lane) { return lane >> 4; }

// NP planes of the 16 x 16 block at rows r0.., groups g0.. of a tile whose planes are `pitch` bytes apart
template <int NP, int C>
__device__ __forceinline__ void load_rows(uint32_t (&f)[NP][4], uint32_t tile, uint32_t pitch, int r0, int g0, int lane) {
    const uint32_t a = tile + tile_at<C>(r0 + rows_row(lane), g0 + rows_grp(lane));
#pragma unroll
    for (int p = 0; p < NP; ++p) ldsm4(f[p], a + p * pitch);
}
template <int NP, int C>
__device__ __forceinline__ void load_rows_t(uint32_t (&f)[NP][4], uint32_t tile, uint32_t pitch, int r0, int g0, int lane) {
    const uint32_t a = tile + tile_at<C>(r0 + rows_row(lane), g0 + rows_grp(lane));
#pragma unroll
    for (int p = 0; p < NP; ++p) ldsm4t(f[p], a + p * pitch);
}
template <int NP, int C>
__device__ __forceinline__ void load_cols(uint32_t (&f)[NP][4], uint32_t tile, uint32_t pitch, int r0, int g0, int lane) {
    const uint32_t a = tile + tile_at<C>(r0 + cols_row(lane), g0 + cols_grp(lane));
#pragma unroll
    for (int p = 0; p < NP; ++p) ldsm4(f[p], a + p * pitch);
}
template <int NP, int C>
__device__ __forceinline__ void load_cols_t(uint32_t (&f)[NP][4], uint32_t tile, uint32_t pitch, int r0, int g0, int lane) {
    const uint32_t a = tile + tile_at<C>(r0 + cols_row(lane), g0 + cols_grp(lane));
#pragma unroll
    for (int p = 0; p < NP; ++p) ldsm4t(f[p], a + p * pitch);
}

// ---- global memory -> registers -> operand planes ------------------------------------------------------------
// Ordinary loads throughout, not __ldg: a kernel that was launched as a programmatic dependent is resident while the kernel
// before it still writes what it will read (the state of the piece before, the features of a map).  The read-only path asks
// for data that nobody writes while the kernel runs, and the compiler may move such a load ahead of griddepcontrol.wait.

// A group of eight consecutive elements of a row.
template <typename IO> struct Group8;
template <> struct Group8<float> {
    float4 a, b;
    __device__ __forceinline__ void fill(float v) { a = b = make_float4(v, v, v, v); }
    __device__ __forceinline__ void load(const float* p) {
        a = *reinterpret_cast<const float4*>(p);
        b = reinterpret_cast<const float4*>(p)[1];
    }
    __device__ __forceinline__ void get(float (&x)[8]) const {
        x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
    }
};
template <> struct Group8<__nv_bfloat16> {
    uint4 a;
    __device__ __forceinline__ void fill(float v) { const uint32_t w = __byte_perm(__float_as_uint(v), 0u, 0x3232); a = make_uint4(w, w, w, w); }
    __device__ __forceinline__ void load(const __nv_bfloat16* p) { a = *reinterpret_cast<const uint4*>(p); }
    __device__ __forceinline__ void get(float (&x)[8]) const {
        const uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) { x[2 * j] = __uint_as_float(w[j] << 16); x[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u); }
    }
};

// What rows and columns that do not exist are read as: a number whose feature is zero.
__device__ __forceinline__ float pad_value(int phi) { return phi == LA_PHI_IDENTITY ? 0.f : -INFINITY; }

// f(x) over a range of registers with the feature map chosen once; NQ = 1: the values are rounded to bf16 afterwards,
// the approximate exponential (2^-21, the square of that of half the number: no feature that bf16 holds is lost) will do
template <int NQ, typename F>
__device__ __forceinline__ void with_phi(int phi, F f) {
    if (phi == LA_PHI_IDENTITY) f([](float x) { return x; });
    else if constexpr (NQ == 1) f([](float x) {
        float e;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x * 0.72134752044448170f));
        return x > 0.f ? x + 1.f : e * e;
    });
    else f([](float x) { const float e = expf(x); return x > 0.f ? x + 1.f : e; });
}

// Whole strips without a predicate and padding per group: where they are never wider than the problem and the kernels small,
// that is bf16 with 32 columns (D = M = 32, la_cluster.cu); the others lost 5 to 8 % to the second copy of their loads.
template <typename IO, int C> constexpr bool kPlainLoads = sizeof(IO) == 2 && C == 32;

// T rows of `cols` columns (padded to C), contiguous in global memory; rows cn.. and columns cols.. hold `pad`.
template <typename IO, int T, int C, int THREADS>
struct RawTile {
    static constexpr int GROUPS = T * (C / 8) / THREADS;
    Group8<IO> r[GROUPS];
    __device__ __forceinline__ void load(const IO* src, int cn, int cols, float pad) {
#pragma unroll
        for (int u = 0; u < GROUPS; ++u) {
            const int idx = (int)threadIdx.x + u * THREADS, row = idx / (C / 8), c = idx % (C / 8) * 8;
            r[u].fill(pad);
            if (row < cn && c < cols) r[u].load(src + row * cols + c);
        }
    }
    // the one plane of bf16 values
    __device__ __forceinline__ void copy(uint8_t* tile) const {
        static_assert(sizeof(IO) == 2, "one plane");
#pragma unroll
        for (int u = 0; u < GROUPS; ++u) {
            const int idx = (int)threadIdx.x + u * THREADS, row = idx / (C / 8), g = idx % (C / 8);
            *reinterpret_cast<uint4*>(tile + tile_at<C>(row, g)) = r[u].a;
        }
    }
    // planes of the features
    template <int NP>
    __device__ __forceinline__ void features(uint8_t* tile, int phi) const {
        if constexpr (NP == 1) {            // features as they are given
            copy(tile);
        } else {
            with_phi<NP>(phi, [&](auto f) { store<NP>(tile, [&](int, float x) { return f(x); }); });
        }
    }
    template <int NP>
    __device__ __forceinline__ void values(uint8_t* tile) const {
        if constexpr (sizeof(IO) == 2) copy(tile);
        else store<NP>(tile, [](int, float x) { return x; });
    }
    // planes of f(u, x), u the group's index in r
    template <int NP, typename F>
    __device__ __forceinline__ void store(uint8_t* tile, F f) const {
#pragma unroll
        for (int u = 0; u < GROUPS; ++u) {
            const int idx = (int)threadIdx.x + u * THREADS, row = idx / (C / 8), g = idx % (C / 8);
            float x[8];
            r[u].get(x);
            uint32_t o[NP][4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t p[NP];
                split2<NP>(f(u, x[2 * j]), f(u, x[2 * j + 1]), p);
#pragma unroll
                for (int k = 0; k < NP; ++k) o[k][j] = p[k];
            }
#pragma unroll
            for (int k = 0; k < NP; ++k)
                *reinterpret_cast<uint4*>(tile + k * (T * C * 2) + tile_at<C>(row, g)) = make_uint4(o[k][0], o[k][1], o[k][2], o[k][3]);
        }
    }
};

__device__ __forceinline__ float2 load_pair(const float* p) { return *reinterpret_cast<const float2*>(p); }
template <typename IO> __device__ __forceinline__ void store_pair(IO* p, float x, float y);
template <> __device__ __forceinline__ void store_pair<float>(float* p, float x, float y) { *reinterpret_cast<float2*>(p) = make_float2(x, y); }
template <> __device__ __forceinline__ void store_pair<__nv_bfloat16>(__nv_bfloat16* p, float x, float y) {
    *reinterpret_cast<uint32_t*>(p) = pack_rn(x, y);
}

// Sixteen rows as A operands straight from global memory: element pairs (row g or g + 8, columns 16 kk + 2t (+ 8)),
// which are also the positions of the thread's elements in a 16 x C result.
template <typename IO> struct Pair;
template <> struct Pair<float> {
    float2 v;
    __device__ __forceinline__ void load(const float* p) { v = *reinterpret_cast<const float2*>(p); }
    __device__ __forceinline__ void fill(float x) { v = make_float2(x, x); }
    __device__ __forceinline__ float lo() const { return v.x; }
    __device__ __forceinline__ float hi() const { return v.y; }
    __device__ __forceinline__ void set(float x, float y) { v = make_float2(x, y); }
    template <int NP> __device__ __forceinline__ void planes(uint32_t (&p)[NP]) const { split2<NP>(v.x, v.y, p); }
};
template <> struct Pair<__nv_bfloat16> {        // as loaded: one plane
    uint32_t w;
    __device__ __forceinline__ void load(const __nv_bfloat16* p) { w = *reinterpret_cast<const uint32_t*>(p); }
    __device__ __forceinline__ void fill(float x) { w = __byte_perm(__float_as_uint(x), 0u, 0x3232); }
    __device__ __forceinline__ float lo() const { return __uint_as_float(w << 16); }
    __device__ __forceinline__ float hi() const { return __uint_as_float(w & 0xffff0000u); }
    __device__ __forceinline__ void set(float x, float y) { w = pack_rn(x, y); }
    template <int NP> __device__ __forceinline__ void planes(uint32_t (&p)[NP]) const {
        static_assert(NP == 1, "a bf16 pair has one plane");
        p[0] = w;
    }
};

template <typename IO, int C>
struct RawStrip {
    static constexpr int KS = C / 16;
    Pair<IO> r[KS][4];
    __device__ __forceinline__ void load(const IO* src, int row0, int cn, int cols, float pad) {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
        if constexpr (kPlainLoads<IO, C>) {
            if (cn >= row0 + 16) {
                src += (row0 + g) * C + t * 2;
#pragma unroll
                for (int kk = 0; kk < KS; ++kk)
#pragma unroll
                    for (int j = 0; j < 4; ++j) r[kk][j].load(src + (j & 1) * (8 * C) + kk * 16 + (j >> 1) * 8);
                return;
            }
        }
#pragma unroll
        for (int kk = 0; kk < KS; ++kk)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int row = row0 + g + (j & 1) * 8, c = kk * 16 + t * 2 + (j >> 1) * 8;
                r[kk][j].fill(pad);
                if (row < cn && c < cols) r[kk][j].load(src + row * cols + c);
            }
    }
    // features: as fp32 pairs, or (To = bf16) rounded
    template <int NQ, bool kSubnormal = true, typename To>
    __device__ __forceinline__ void map(int phi, RawStrip<To, C>& out) const {
        if constexpr (sizeof(To) == 2) {        // two at a time, from bf16 to bf16
            if (phi == LA_PHI_IDENTITY) {
                out = *this;
                return;
            }
#pragma unroll
            for (int kk = 0; kk < KS; ++kk)
#pragma unroll
                for (int j = 0; j < 4; ++j) out.r[kk][j].w = tc::phi_pair<kSubnormal>(r[kk][j].w);
        } else with_phi<NQ>(phi, [&](auto f) {
#pragma unroll
            for (int kk = 0; kk < KS; ++kk)
#pragma unroll
                for (int j = 0; j < 4; ++j) out.r[kk][j].set(f(r[kk][j].lo()), f(r[kk][j].hi()));
        });
    }
    template <int NP>
    __device__ __forceinline__ void planes(uint32_t (&a)[KS][NP][4]) const {
#pragma unroll
        for (int kk = 0; kk < KS; ++kk)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t p[NP];
                r[kk][j].template planes<NP>(p);
#pragma unroll
                for (int k = 0; k < NP; ++k) a[kk][k][j] = p[k];
            }
    }
};

// a 16 x 16 block of results (two 16 x 8 accumulators) as the planes of an A operand
template <int NP>
__device__ __forceinline__ void operand_of(uint32_t (&a)[NP][4], const float (&c0)[4], const float (&c1)[4]) {
    const float* c[2] = {c0, c1};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t p[NP];
        split2<NP>(c[j >> 1][(j & 1) * 2], c[j >> 1][(j & 1) * 2 + 1], p);
#pragma unroll
        for (int k = 0; k < NP; ++k) a[k][j] = p[k];
    }
}

__device__ __forceinline__ float quad_sum(float v) {       // over the four lanes that share a result row
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    return v;
}

// Kernels that follow each other on a stream start early (programmatic dependent launch): nothing of the kernels before
// is read or written ahead of the wait; the next kernel may be scheduled once every CTA of this one has released it.
__device__ __forceinline__ void wait_for_stream() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void release_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

}  // namespace mma
}  // namespace la
