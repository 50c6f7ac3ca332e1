// What kernels share whose warps hold their operands in registers (la_causal_warp.cuh, la_linear_warp.cuh): sixteen rows as operands of
// mma.sync m16n8k16, and chunks of sixteen rows on their way to a warp.
//
// A lane loads sixteen bytes of a row, columns 8 t .. 8 t + 7 (and 32 + 8 t ..), and takes the four pairs as columns 2 t, 2 t + 1
// of four 8-column tiles.  Tiles therefore hold the columns in another order (column 2 t + e of tile n is column
// 32 (n / 4) + 8 t + 2 (n % 4) + e of the tensor), the same one for every operand, so that all sums over columns agree and a result row
// leaves as sixteen bytes again.
#pragma once

#include "la_mma_sweep.cuh"

namespace la {
namespace warp {

using namespace mma;

constexpr int ROWS = 16;                    // positions of a chunk

// Sixteen rows: x[h][n] = columns 2 t, 2 t + 1 of tile n in row g + 8 h.  As an A operand (rows x columns) and as a B operand
// (columns x rows) it serves as it lies; transposed, t[h][n] = rows 8 h + 2 t, 2 t + 1 of column g of tile n, it is
// an A operand (columns x rows) and a B operand (rows x columns).
template <int W> struct Rows { uint32_t x[2][W / 8]; };

__device__ __forceinline__ uint32_t transposed(uint32_t v) {
    uint32_t r;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}
template <int W> __device__ __forceinline__ Rows<W> transposed(const Rows<W>& r) {
    Rows<W> o;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int n = 0; n < W / 8; ++n) o.x[h][n] = transposed(r.x[h][n]);
    return o;
}

__device__ __forceinline__ void mma_add(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_first(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
// c (rows of a x eight rows or columns) = or += the columns of a times b, b's operand pairs given by f(kk, half)
template <bool FIRST, int W, typename F>
__device__ __forceinline__ void columns_mma(float (&c)[4], const Rows<W>& a, F f) {
#pragma unroll
    for (int kk = 0; kk < W / 16; ++kk) {
        if (FIRST && kk == 0) mma_first(c, a.x[0][0], a.x[1][0], a.x[0][1], a.x[1][1], f(0, 0), f(0, 1));
        else mma_add(c, a.x[0][2 * kk], a.x[1][2 * kk], a.x[0][2 * kk + 1], a.x[1][2 * kk + 1], f(kk, 0), f(kk, 1));
    }
}

// two additions in one instruction
__device__ __forceinline__ void add_pair(float& x, float& y, float a, float b) {
    sm100::unpair(sm100::add2(sm100::pair(x, y), sm100::pair(a, b)), x, y);
}

// 1 / x as a division gives it, without the branch of one, at which these loops would be cut in two (B128 H8 N784 161.7 -> 155.7 us a
// step): the approximation and one Newton-Raphson step in fused multiply-adds, which rounds correctly but for mantissas of all ones
// (Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", 1990); of all 2^32 numbers ten, with reciprocals
// below 1.2e-38, differ from 1.f / x, of the approximation alone 13 %.  Where the residual is no small number (x zero, infinite, NaN, or its
// reciprocal too large) the approximation is the answer.
__device__ __forceinline__ float reciprocal(float x) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    const float e = fmaf(-x, r, 1.f);
    return fabsf(e) < 0.5f ? fmaf(r, e, r) : r;
}

// the lane's part of a row's dot product: a (bf16 pairs) with b (fp32 pairs at the same columns)
template <int NT, typename F>
__device__ __forceinline__ sm100::f32x2 row_part(const uint32_t (&a)[NT], F b) {
    sm100::f32x2 d = sm100::mul2(sm100::pair_bf16(a[0]), b(0));
#pragma unroll
    for (int n = 1; n < NT; ++n) d = sm100::fma2(sm100::pair_bf16(a[n]), b(n), d);
    return d;
}

constexpr uint32_t kOnes = 0x3f803f80u, kMinusInf = 0xff80ff80u;

// T tensors of sixteen rows each, a lane's own sixteen bytes of rows g and g + 8; WEIGHTS: and two fp32 numbers per row.
// STAGES: the chunk at hand and those on their way.
template <int W, int T, bool WEIGHTS, int STAGES = 3>
struct Ring {
    static constexpr int AHEAD = STAGES - 1, TILE = ROWS * W * 2, PARTS = W / 32;        // a row's parts of 64 bytes
    static constexpr int STAGE_BYTES = T * TILE + (WEIGHTS ? 128 : 0), BYTES = STAGES * STAGE_BYTES;
    const uint8_t* src[T];          // the lane's bytes of the sequence's first chunk
    const float* w;                 // the lane's weight of it: 1 / dn in lanes 0 .. 15, dl in lanes 16 .. 31
    uint8_t* base;                  // slot 0
    uint8_t* mine;                  // the lane's bytes of it (rows of 64 bytes, the four sixteens of row g in another order: an
                                    // ldmatrix that reads one of eight rows finds them in different banks)
    int read, write;                // offsets of the slot at hand and of the next one to be filled
    int end;                        // rows from `end` on are not there: zeros

    // of sequence bh of N positions, those before `stop`; aux: two rows of N weights per sequence
    __device__ __forceinline__ void start(uint8_t* smem, int64_t bh, int64_t N, int stop, const void* const (&tensors)[T], const float* aux) {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int i = 0; i < T; ++i) src[i] = (const uint8_t*)tensors[i] + bh * N * (W * 2) + (lane >> 2) * (W * 2) + (lane & 3) * 16;
        if constexpr (WEIGHTS) w = aux + 2 * bh * N + (lane < 16 ? lane : N + lane - 16);
        base = smem;
        mine = smem + (lane >> 2) * 64 + (((lane & 3) ^ ((lane >> 3) & 3)) << 4);
        end = stop;
        read = write = 0;
    }
    __device__ __forceinline__ void request(int n0) {
        if constexpr (WEIGHTS) __syncwarp();            // every lane has read what is overwritten
        if (n0 >= 0 && n0 < end) {
            const int lane = threadIdx.x & 31, left = end - n0;
            const uint32_t dst = smem_u32(mine + write);
            const int64_t at = (int64_t)n0 * (W * 2);
            if (left >= ROWS) {
#pragma unroll
                for (int i = 0; i < T; ++i)
#pragma unroll
                    for (int j = 0; j < 2 * PARTS; ++j)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i * TILE + j * 512),
                                     "l"(src[i] + at + j / PARTS * (16 * W) + j % PARTS * 64) : "memory");
                if constexpr (WEIGHTS) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(base + write + T * TILE) + lane * 4), "l"(w + n0) : "memory");
            } else {                // (a size of zero reads nothing; the address stays inside the tensor)
#pragma unroll
                for (int i = 0; i < T; ++i)
#pragma unroll
                    for (int j = 0; j < 2 * PARTS; ++j) {
                        const bool real = (lane >> 2) + j / PARTS * 8 < left;
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + i * TILE + j * 512),
                                     "l"(real ? src[i] + at + j / PARTS * (16 * W) + j % PARTS * 64 : src[i] - (lane >> 2) * (W * 2)), "r"(real ? 16 : 0) : "memory");
                    }
                if constexpr (WEIGHTS) {
                    const bool real = (lane & 15) < left;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(base + write + T * TILE) + lane * 4), "l"(real ? w + n0 : w - (lane & 15)),
                                 "r"(real ? 4 : 0) : "memory");
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        write = write == (STAGES - 1) * STAGE_BYTES ? 0 : write + STAGE_BYTES;
    }
    __device__ __forceinline__ void next() { read = read == (STAGES - 1) * STAGE_BYTES ? 0 : read + STAGE_BYTES; }
    // The chunk STAGES - 1 behind the one that was just requested has arrived.  If not all of its rows are real, the others of
    // tensor `i` are filled.
    __device__ __forceinline__ void arrived(int i, int real, uint32_t fill) const { arrived_of<STAGES - 1>(i, real, fill); }
    // ... all but the last PENDING requests
    template <int PENDING> __device__ __forceinline__ void arrived_of(int i, int real, uint32_t fill) const {
        asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
        if (real < ROWS) {
            const int lane = threadIdx.x & 31;
#pragma unroll
            for (int j = 0; j < 2 * PARTS; ++j)
                if ((lane >> 2) + j / PARTS * 8 >= real) *reinterpret_cast<uint4*>(mine + read + i * TILE + j * 512) = make_uint4(fill, fill, fill, fill);
            if constexpr (WEIGHTS)
                if (lane < 16 && lane >= real) *reinterpret_cast<float*>(base + read + T * TILE + lane * 4) = 1.f;
        }
        if constexpr (WEIGHTS) __syncwarp();
    }
    __device__ __forceinline__ Rows<W> rows(int i) const {
        Rows<W> r;
#pragma unroll
        for (int j = 0; j < 2 * PARTS; ++j) {
            const uint4 v = *reinterpret_cast<const uint4*>(mine + read + i * TILE + j * 512);
            uint32_t* x = r.x[j / PARTS] + j % PARTS * 4;
            x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
        }
        return r;
    }
    // the lane's rows of tensor i, for the other warps
    __device__ __forceinline__ void put_rows(int i, const Rows<W>& r) const {
#pragma unroll
        for (int j = 0; j < 2 * PARTS; ++j) {
            const uint32_t* x = r.x[j / PARTS] + j % PARTS * 4;
            *reinterpret_cast<uint4*>(mine + read + i * TILE + j * 512) = make_uint4(x[0], x[1], x[2], x[3]);
        }
    }
    __device__ __forceinline__ const float* weights() const { return reinterpret_cast<const float*>(base + read + T * TILE); }
};

}  // namespace warp
}  // namespace la
