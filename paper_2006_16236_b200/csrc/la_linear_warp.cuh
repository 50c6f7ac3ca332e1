// Non-causal form (Eq. 5-6 and its gradient) of bf16 problems with D = M = 32 or 64 on mma.sync: the kernels of la_tc_linear.cu, where
// the formulas and the centred operands are.  A CTA of sixteen warps per split of a sequence (or eight, two on an SM, where nothing is summed); a warp takes sixteen positions at a time
// past the sums of the whole sequence, with its next positions on their way (la_warp.cuh).  Where sums over the positions are formed,
// every warp has sixteen rows and sixteen columns of them (W = 64) and adds up over the chunks of all warps, which lie in shared memory
// as they came or were mapped: a barrier per 256 positions.  (All of the sums in the registers of every warp, transposes by movmatrix and
// an addition over the warps at the end: the same 23 us for the forward sums of B8 H8 N4096 D = 64, but no room for those of the dQ
// pass, 27 us on top.)  tcgen05 tiles of 128 positions have the same products behind a chain of mapping, product, read-out and
// exchanges between the halves of a row: 2000 to 3500 cycles a tile.
// What bounds it: instruction issue (a row of 32 columns costs half of one of 64, at the same bytes per number), and a CTA's start: two
// trips to L2 and four barriers, 4 us, beside the first positions.  Figures at of_warps() in la_tc_linear.cu.
#pragma once

#include "la_warp.cuh"

namespace la {
namespace tc {
namespace lin {

using namespace warp;
using sm100::f32x2;

constexpr int WARPS = 16, THREADS = 32 * WARPS, CHUNK = WARPS * ROWS;

// Record of one split: [A' (64x64) | a' (64) | ysum (64) | w0 (1) | pad | stamp (4)]:
//   forward sums: A' = sum k'_j V_j^T, a' = sum k'_j, ysum = sum V_j,                    w0 unused
//   reverse sums: A' = sum qh'_i G_i^T, a' = sum qh'_i dl_i, ysum = sum G_i / dn_i,      w0 = sum dl_i / dn_i
constexpr int kRecFloats = kDim * kDim + kDim + kDim + 8;
// The last four words of a record: the split plan it was written under.  A backward pass that is given kept records and
// would split the sequences in another way (la_plan_override() in between) reports that and writes nothing.  The CTAs of
// sequence i look at record i, which every plan has: all of them at the first one took 0.5 us longer a step.
constexpr int kRecStamp = kRecFloats - 4;
__device__ __forceinline__ int4 split_stamp(int nseg, int chunks_per_seg, int dim) {
    return make_int4(0x4c414c53, nseg, chunks_per_seg, dim);
}

struct Params {
    const void *X, *Y;          // sums: K, V (reverse: Q, G);  forward: Q;  backward Q: Q, G;  backward K/V: K, V
    void *out0, *out1;          // forward: O;  backward Q: dQ;  backward K/V: dK, dV
    float* records;             // [BH][nseg][kRecFloats]: written by the sums, added up by every CTA of the others
    float* rec_out;             // backward Q: [BH][nseg][kRecFloats], the reverse sums of its rows
    float* den;                 // forward: q . Z (optional)
    float *state_out, *vec_out; // forward: KV [BH][D][M], Zs [BH][D] (optional)
    const float* kept;          // backward: the forward's kept records, whose stamp has to be this plan's, or null
    const int* lengths;         // [B] real positions per batch element (right-padded ragged batch), or null
    int* status;
    int64_t N;
    int heads, nseg, chunks_per_seg;            // records of a sequence, written by a CTA each
    int parts;                  // CTAs of a sequence
    float eps;
    int early;                  // a kernel of the same call runs in front: the first positions are requested before the wait
};

// Of a sequence's `len` positions a split takes [lo, end), whole chunks but the last; of the padding behind them it
// fills [zero_lo, zero_hi).  By its real length: a sequence half as long is half the work for each of its CTAs.
struct Span { int64_t bh; int lo, end, zero_lo, zero_hi, len; };
__device__ __forceinline__ Span span_of(const Params& p) {
    Span s;
    const int parts = p.parts, part = (int)(blockIdx.x % parts);
    s.bh = blockIdx.x / parts;
    s.len = (int)(p.lengths ? min((int64_t)max(p.lengths[s.bh / p.heads], 0), p.N) : p.N);
    const int chunks = (s.len + ROWS - 1) / ROWS, each = (chunks + parts - 1) / parts;
    s.lo = min(part * each * ROWS, s.len);
    s.end = min(s.lo + each * ROWS, s.len);
    const int pad = (int)p.N - s.len, fill = (pad + parts - 1) / parts;
    s.zero_lo = s.len + min(part * fill, pad);
    s.zero_hi = s.len + min(part * fill + fill, pad);
    return s;
}

// element (8-column tile n, column c of it, in the order of la_warp.cuh) -> column of the tensor
__device__ __forceinline__ int column(int n, int c) { return 32 * (n >> 2) + 8 * (c >> 1) + 2 * (n & 3) + (c & 1); }

// elu(x) = phi(x) - 1 of a bf16 pair, rounded (x > 0: x itself)
template <bool ELU> __device__ __forceinline__ uint32_t centred_pair(uint32_t w) {
    const f32x2 x = sm100::pair_bf16(w);
    if constexpr (!ELU) return sm100::pack_bf16x2(sm100::add2(x, sm100::pair(-1.f, -1.f)));
    float t0, t1, e0, e1;
    sm100::unpair(sm100::mul2(x, sm100::pair(1.4426950408889634f, 1.4426950408889634f)), t0, t1);
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(t0));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(t1));
    const uint32_t ex = sm100::pack_bf16x2(sm100::add2(sm100::pair(e0, e1), sm100::pair(-1.f, -1.f)));
    uint32_t mask, res;
    asm("prmt.b32 %0, %1, %1, 0xBB99;" : "=r"(mask) : "r"(w));
    asm("lop3.b32 %0, %1, %2, %3, 0xCA;" : "=r"(res) : "r"(mask), "r"(ex), "r"(w));    // mask ? ex : w
    return res;
}
template <bool ELU, int W> __device__ __forceinline__ void centre(Rows<W>& r) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int n = 0; n < W / 8; ++n) r.x[h][n] = centred_pair<ELU>(r.x[h][n]);
}

// Dot products of rows with fp32 vectors are products with one tile of columns: the three planes of a' (0 .. 2), ones (3), the three
// planes of nu (4 .. 6).  Lane t of a row then has columns 2 t, 2 t + 1 of the result, and the others get theirs by shuffles.
template <int W> __device__ __forceinline__ void vector_product(float (&u)[4], const Rows<W>& a, const uint2* vectors) {
#pragma unroll
    for (int kk = 0; kk < W / 16; ++kk) {
        const uint2 b = vectors[kk * 32 + (threadIdx.x & 31)];
        if (kk == 0) mma_first(u, a.x[0][0], a.x[1][0], a.x[0][1], a.x[1][1], b.x, b.y);
        else mma_add(u, a.x[0][2 * kk], a.x[1][2 * kk], a.x[0][2 * kk + 1], a.x[1][2 * kk + 1], b.x, b.y);
    }
}
// the lane with column `col` of row g (h = 0) or g + 8
__device__ __forceinline__ float from_column(const float (&u)[4], int h, int col) {
    return __shfl_sync(0xffffffffu, u[2 * h + (col & 1)], (threadIdx.x & 28) | (col >> 1));
}
__device__ __forceinline__ float across(f32x2 part) { return quad_sum(sm100::pair_sum(part)); }

template <int W> __device__ __forceinline__ void put_row(void* tensor, int64_t row, const uint32_t (&o)[W / 8]) {
    uint8_t* at = (uint8_t*)tensor + row * (W * 2) + (threadIdx.x & 3) * 16;
#pragma unroll
    for (int q = 0; q < W / 32; ++q) *reinterpret_cast<uint4*>(at + q * 64) = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
}
template <int W, int THREADS> __device__ __forceinline__ void zero_rows(void* tensor, int64_t from, int64_t to) {
    uint4* x = reinterpret_cast<uint4*>((uint8_t*)tensor + from * (W * 2));
    for (int64_t i = threadIdx.x; i < (to - from) * (W / 8); i += THREADS) x[i] = make_uint4(0u, 0u, 0u, 0u);
}

// ---- sums of a split -----------------------------------------------------------------------------------------------
// Of X^T Y, 1^T X and 1^T Y (or with weights) a warp has rows 16 i .., columns 16 c .. and adds up over every GROUPS-th chunk.
template <int W> struct Sums {
    static constexpr int SIDE = W / 16, GROUPS = WARPS / (SIDE * SIDE), FLOATS = W * W + 2 * W;
    float s[2][4], x[4], y[2][4];

    static __device__ __forceinline__ int block_row() { return (int)(threadIdx.x >> 5) % SIDE; }
    static __device__ __forceinline__ int block_col() { return (int)(threadIdx.x >> 5) / SIDE % SIDE; }
    static __device__ __forceinline__ int group() { return (int)(threadIdx.x >> 5) / (SIDE * SIDE); }
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int j = 0; j < 4; ++j) s[0][j] = s[1][j] = x[j] = y[0][j] = y[1][j] = 0.f;
    }
    // The chunks of `warps` warps: X and Y at tx, ty, their shared addresses for the first warp, `pitch` bytes apart.  wx, wy: the
    // weights' planes, [chunk][plane 0 .. 3 (zeros)][16] bf16, or null for ones.
    template <bool WEIGHTED>
    __device__ __forceinline__ void add(uint32_t tx, uint32_t ty, uint32_t pitch, int warps, const uint16_t* wx, const uint16_t* wy) {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, m = lane >> 3, row = lane & 7;
        auto at = [&](int tile, int h) {
            return (uint32_t)(h * (W / 32) * 512 + (tile >> 2) * 512 + row * 64 + (((tile & 3) ^ ((row >> 1) & 3)) << 4));
        };
        const uint32_t ax = at(2 * block_row() + (m & 1), m >> 1), ay = at(2 * block_col() + (m >> 1), m & 1);
        const bool rows = block_col() == 0, cols = block_row() == 0;
#pragma unroll 4
        for (int w = group(); w < warps; w += GROUPS) {
            uint32_t a[4], b[4];
            ldsm4t(a, tx + w * pitch + ax);
            ldsm4t(b, ty + w * pitch + ay);
            mma_add(s[0], a[0], a[1], a[2], a[3], b[0], b[1]);
            mma_add(s[1], a[0], a[1], a[2], a[3], b[2], b[3]);
            // a vector's planes (or ones) are columns of a B operand, rows of an A operand
            uint32_t v0 = g == 0 ? kOnes : 0u, v1 = v0;
            if (rows) {
                if constexpr (WEIGHTED) {
                    const uint16_t* p = wx + w * 64 + min(g, 3) * 16 + 2 * t;
                    v0 = *reinterpret_cast<const uint32_t*>(p);
                    v1 = *reinterpret_cast<const uint32_t*>(p + 8);
                }
                mma_add(x, a[0], a[1], a[2], a[3], v0, v1);
            }
            if (cols) {
                if constexpr (WEIGHTED) {
                    const uint16_t* p = wy + w * 64 + min(g, 3) * 16 + 2 * t;
                    v0 = *reinterpret_cast<const uint32_t*>(p);
                    v1 = *reinterpret_cast<const uint32_t*>(p + 8);
                }
                mma_add(y[0], v0, 0u, v1, 0u, b[0], b[1]);
                mma_add(y[1], v0, 0u, v1, 0u, b[2], b[3]);
            }
        }
    }
    // smem: GROUPS * FLOATS floats that nobody uses any more
    __device__ __forceinline__ void put_record(float* smem, float* rec, float w0) const {
        const int tid = threadIdx.x, lane = tid & 31, g = lane >> 2, t = lane & 3;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        float* mine = smem + group() * FLOATS;
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const int col = 16 * block_col() + 8 * n + 2 * t;
#pragma unroll
            for (int h = 0; h < 2; ++h) *reinterpret_cast<float2*>(mine + (16 * block_row() + 8 * h + g) * W + col) = make_float2(s[n][2 * h], s[n][2 * h + 1]);
            if (block_row() == 0) {
                float v[2] = {y[n][0], y[n][1]};
#pragma unroll
                for (int o = 4; o < 32; o <<= 1)
#pragma unroll
                    for (int e = 0; e < 2; ++e) v[e] += __shfl_xor_sync(0xffffffffu, v[e], o);
                if (g == 0) *reinterpret_cast<float2*>(mine + W * W + W + col) = make_float2(v[0], v[1]);
            }
        }
        if (block_col() == 0)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float v = quad_sum(x[2 * h] + x[2 * h + 1]);
                if (t == 0) mine[W * W + 16 * block_row() + 8 * h + g] = v;
            }
        __syncthreads();
        for (int at = tid; at < FLOATS / 4; at += THREADS) {
            float4 a = reinterpret_cast<const float4*>(smem)[at];
#pragma unroll
            for (int k = 1; k < GROUPS; ++k) {
                const float4 b = reinterpret_cast<const float4*>(smem + k * FLOATS)[at];
                a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
            }
            const int row = at / (W / 4), col = at % (W / 4) * 4;
            *reinterpret_cast<float4*>(rec + (row < W ? row * kDim : kDim * kDim + (row - W) * kDim) + col) = a;
        }
        if (tid == 0) rec[kDim * kDim + 2 * kDim] = w0;
    }
};

template <int W> constexpr int kSumRing = Ring<W, 2, false>::BYTES;
template <int W> constexpr int kSumSmem = WARPS * kSumRing<W>;

// wait(): for the kernel before this one, then the next may be scheduled
template <int W, bool ELU, typename Wait>
__device__ __forceinline__ void sums(const Params& p, uint8_t* smem, Wait wait) {
    static_assert(kSumSmem<W> >= Sums<W>::GROUPS * Sums<W>::FLOATS * 4, "room for the sums");
    const int warp = threadIdx.x >> 5;
    // (Wait first, then let the next kernel be scheduled: a kernel behind this one requests its first positions before it waits in
    // turn, which is safe only if everything before this kernel is complete by then.)
    wait();
    const Span r = span_of(p);
    float* rec = p.records + (int64_t)blockIdx.x * kRecFloats;
    if (threadIdx.x == THREADS - 1) *reinterpret_cast<int4*>(rec + kRecStamp) = split_stamp(p.nseg, p.chunks_per_seg, W);
    Ring<W, 2, false> in;
    in.start(smem + warp * kSumRing<W>, r.bh, p.N, r.end, {p.X, p.Y}, nullptr);
    int n0 = r.lo + warp * ROWS;
    for (int i = 0; i < in.AHEAD; ++i) in.request(n0 + i * CHUNK);
    Sums<W> st;
    st.clear();
#pragma unroll 1
    for (int c0 = r.lo; c0 < r.end; c0 += CHUNK, n0 += CHUNK) {
        in.template arrived_of<in.AHEAD - 1>(0, r.end - n0, ELU ? 0u : kOnes);        // x' = 0 where there is no row (and y = 0)
        Rows<W> x = in.rows(0);
        centre<ELU>(x);
        in.put_rows(0, x);
        __syncthreads();
        in.request(n0 + in.AHEAD * CHUNK);          // into the slot that every warp has left by now
        st.template add<false>(smem_u32(smem + in.read), smem_u32(smem + in.read + in.TILE), kSumRing<W>, min(WARPS, (r.end - c0 + ROWS - 1) / ROWS), nullptr, nullptr);
        in.next();
    }
    st.put_record(reinterpret_cast<float*>(smem), rec, 0.f);
}

// ---- apply ---------------------------------------------------------------------------------------------------------
enum ApplyMode { kApplyForward = 0, kApplyBackwardQ = 1, kApplyBackwardKV = 2 };

// Shared memory: the centred matrix S'' as B operands in the order of the lanes ([kk][n / 2][lane], sixteen bytes), as it lies (rows
// summed over) and / or transposed; the vectors a' and nu; scratch for their making, later the chunks on their way
template <int W, int MODE, int WARPS> struct ApplyLayout {
    static constexpr int TENSORS = MODE == kApplyForward ? 1 : 2;
    using Chunks = Ring<W, TENSORS, false, MODE == kApplyForward ? 3 : 2>;          // (three of two tensors do not fit)
    static constexpr int OPERAND = W * W * 2;
    static constexpr int ROWWISE = 0, COLWISE = MODE == kApplyBackwardQ ? 0 : OPERAND,        // K/V has both
                         VECTORS = MODE == kApplyBackwardKV ? 2 * OPERAND : OPERAND, VEC = VECTORS + W / 16 * 32 * 8,
                         SCRATCH = VEC + (2 * kDim + 4 + WARPS) * 4,
                         PLANES = SCRATCH + (kDim * W + 9 * kDim) * 4,          // backward Q: the weights' planes, twice two per warp
                         RING = PLANES + (MODE == kApplyBackwardQ ? 2 * WARPS * 256 : 0), BYTES = RING + WARPS * Chunks::BYTES;
    static_assert(BYTES <= 227 * 1024, "shared memory");
};

// c (sixteen rows, tiles n, n + 1) = rows of a times the operand
template <int W> __device__ __forceinline__ void product(float (&c)[W / 8][4], const Rows<W>& a, const uint8_t* operand) {
    const uint4* b = reinterpret_cast<const uint4*>(operand) + (threadIdx.x & 31);
#pragma unroll
    for (int n = 0; n < W / 16; ++n)
#pragma unroll
        for (int kk = 0; kk < W / 16; ++kk) {
            const uint4 f = b[(kk * (W / 16) + n) * 32];
            if (kk == 0) {
                mma_first(c[2 * n], a.x[0][0], a.x[1][0], a.x[0][1], a.x[1][1], f.x, f.y);
                mma_first(c[2 * n + 1], a.x[0][0], a.x[1][0], a.x[0][1], a.x[1][1], f.z, f.w);
            } else {
                mma_add(c[2 * n], a.x[0][2 * kk], a.x[1][2 * kk], a.x[0][2 * kk + 1], a.x[1][2 * kk + 1], f.x, f.y);
                mma_add(c[2 * n + 1], a.x[0][2 * kk], a.x[1][2 * kk], a.x[0][2 * kk + 1], a.x[1][2 * kk + 1], f.z, f.w);
            }
        }
}

template <int W, int MODE, int WARPS, bool ELU, typename Wait>
__device__ __forceinline__ void apply(const Params& p, uint8_t* smem, Wait wait) {
    using L = ApplyLayout<W, MODE, WARPS>;
    constexpr int NT = W / 8, THREADS = 32 * WARPS, CHUNK = WARPS * ROWS;
    static_assert(MODE != kApplyBackwardQ || WARPS == lin::WARPS, "the sums are shared out over that many");
    constexpr bool kHasY = MODE != kApplyForward;
    float* sA = reinterpret_cast<float*>(smem + L::VEC);         // a': Z' (forward, backward Q) or r' (backward K/V)
    float* sNu = sA + kDim;                                      // rank-one part along 1: ysum + mu  /  gsum + rho
    float* sScal = sA + 2 * kDim;                                // [0] = sum_d a'_d, [1] = w0
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    // The rows of this pass are inputs of the call.  Behind another kernel of the same call (which waited for everything before it and
    // only then let this one be scheduled) the first of them are requested before the wait; as the first kernel of a call everything
    // waits first.
    const bool early = p.early != 0;
    if (!early) wait();
    const Span r = span_of(p);
    const float* rec = p.records + r.bh * p.nseg * (int64_t)kRecFloats;
    typename L::Chunks in;
    if constexpr (kHasY) in.start(smem + L::RING + warp * L::Chunks::BYTES, r.bh, p.N, r.end, {p.X, p.Y}, nullptr);
    else in.start(smem + L::RING + warp * L::Chunks::BYTES, r.bh, p.N, r.end, {p.X}, nullptr);
    int n0 = r.lo + warp * ROWS;
    for (int i = 0; i < in.AHEAD; ++i) in.request(n0 + i * CHUNK);
    if (early) wait();
    if (kHasY && p.kept) {
        const int4 a = *reinterpret_cast<const int4*>(p.kept + r.bh * kRecFloats + kRecStamp), b = split_stamp(p.nseg, p.chunks_per_seg, W);
        if (a.x != b.x || a.y != b.y || a.z != b.z || a.w != b.w) {     // (the same for every thread)
            if (tid == 0) atomicOr(p.status, sm100::kStatusPlanMismatch);
            asm volatile("cp.async.wait_all;" ::: "memory");
            return;
        }
    }
    // state of this head: add the split records (fp32), remove the column means, round the centred remainder to operands
    {
        float* sF = reinterpret_cast<float*>(smem + L::SCRATCH);                // fp32 [W][64], means [64], partial sums [8][64]
        float* sMu = sF + kDim * W;
        constexpr int PER = W * kDim / 4 / THREADS;
        float4 acc[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
        for (int n = 0; n < p.nseg; ++n) {
            const float4* src = reinterpret_cast<const float4*>(rec + (int64_t)n * kRecFloats);
#pragma unroll
            for (int u = 0; u < PER; ++u) {
                const float4 a = load_global(src + tid + u * THREADS);
                acc[u].x += a.x; acc[u].y += a.y; acc[u].z += a.z; acc[u].w += a.w;
            }
        }
#pragma unroll
        for (int u = 0; u < PER; ++u) reinterpret_cast<float4*>(sF)[tid + u * THREADS] = acc[u];
        if (tid < 2 * kDim + 1) {       // a' (64), ysum (64), w0 (1)
            float z = 0.f;
            for (int n = 0; n < p.nseg; ++n) z += load_global(rec + (int64_t)n * kRecFloats + kDim * kDim + tid);
            if (tid < kDim) sA[tid] = tid < W ? z : 0.f;
            else if (tid < 2 * kDim) sNu[tid - kDim] = z;
            else sScal[1] = z;
        }
        __syncthreads();
        constexpr int PARTS = THREADS / kDim;
        {                               // column sums: every PARTS-th row a thread
            const int col = tid & (kDim - 1), part = tid >> 6;
            float m = 0.f;
            if (col < W)
                for (int d = part; d < W; d += PARTS) m += sF[d * kDim + col];
            sMu[kDim + part * kDim + col] = m;
        }
        __syncthreads();
        if (tid < W) {                  // column tid: mean over the rows; nu = ysum + mu
            float m = 0.f;
#pragma unroll
            for (int k = 1; k <= PARTS; ++k) m += sMu[k * kDim + tid];
            m *= 1.f / W;
            const float ysum = sNu[tid];
            sNu[tid] = ysum + m;
            sMu[tid] = m;
            if (MODE == kApplyForward && blockIdx.x % p.parts == 0) {
                // true sums for the caller: S = 1 ysum^T + A', Z = N 1 + a'
                if (p.vec_out) p.vec_out[r.bh * W + tid] = (float)r.len + sA[tid];
                if (p.state_out)
                    for (int d = 0; d < W; ++d) p.state_out[r.bh * (int64_t)(W * W) + d * W + tid] = sF[d * kDim + tid] + ysum;
            }
        }
        if (warp == 2) {                // sum of a' (64 values, two per lane, then a butterfly: the same order in every CTA)
            float z = sA[lane] + sA[lane + 32];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) z += __shfl_xor_sync(0xffffffffu, z, off);
            if (lane == 0) sScal[0] = z;
        }
        __syncthreads();
        for (int at = tid; at < W * W / 8; at += THREADS) {        // operand registers of tiles 2 n, 2 n + 1 and rows 16 kk ..
            const int l = at & 31, n = at / 32 % (W / 16), kk = at / (2 * W), lg = l >> 2, lt = l & 3;
            if (MODE != kApplyBackwardQ) {              // summed over the rows of S'': columns are its columns
                uint32_t f[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int m = column(2 * n + (j >> 1), lg), d = column(2 * kk + (j & 1), 2 * lt);
                    f[j] = pack_rn(sF[d * kDim + m] - sMu[m], sF[(d + 1) * kDim + m] - sMu[m]);
                }
                reinterpret_cast<uint4*>(smem + (MODE == kApplyForward ? L::ROWWISE : L::COLWISE))[at] = make_uint4(f[0], f[1], f[2], f[3]);
            }
            if (MODE != kApplyForward) {                // summed over the columns
                uint32_t f[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int d = column(2 * n + (j >> 1), lg), m = column(2 * kk + (j & 1), 2 * lt);
                    const float2 v = load_pair(sF + d * kDim + m), u = load_pair(sMu + m);
                    f[j] = pack_rn(v.x - u.x, v.y - u.y);
                }
                reinterpret_cast<uint4*>(smem + L::ROWWISE)[at] = make_uint4(f[0], f[1], f[2], f[3]);
            }
        }
        if (tid < W / 16 * 32) {        // the vectors' tile: rows (columns of x) 16 kk .., column lane / 4
            const int kk = tid >> 5;
            uint32_t f[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int d = column(2 * kk + j, 2 * t);
                const float* v = g < 4 ? sA : sNu;
                uint32_t pl[3];
                split2<3>(v[d], v[d + 1], pl);
                f[j] = g == 3 ? kOnes : g == 7 ? 0u : (g & 3) == 0 ? pl[0] : (g & 3) == 1 ? pl[1] : pl[2];
            }
            reinterpret_cast<uint2*>(smem + L::VECTORS)[tid] = make_uint2(f[0], f[1]);
        }
        __syncthreads();
    }
    const uint2* vectors = reinterpret_cast<const uint2*>(smem + L::VECTORS);
    const float fD = (float)W, fN = (float)r.len, a_sum = sScal[0], w0 = sScal[1];
    const float* aH = sA + t * 8;               // the lane's columns of tile n at 32 (n / 4) + 2 (n % 4)
    const float* nuH = sNu + t * 8;
    auto of = [](const float* v, int n) { return sm100::pair_ld(v + 32 * (n >> 2) + 2 * (n & 3)); };
    const int64_t base = r.bh * p.N;
    constexpr bool kSums = MODE == kApplyBackwardQ;         // the warps meet once per chunk, and have one request less under way
    Sums<W> st;
    float w_sum = 0.f;
    if constexpr (kSums) {
        st.clear();
        for (int i = tid; i < 2 * WARPS * 64; i += THREADS) reinterpret_cast<uint32_t*>(smem + L::PLANES)[i] = 0u;
        __syncthreads();
    }
    bool odd = false;
#pragma unroll 1
    for (int c0 = r.lo; kSums ? c0 < r.end : n0 < r.end; c0 += CHUNK, n0 += CHUNK) {
        if constexpr (!kSums) in.request(n0 + in.AHEAD * CHUNK);
        in.template arrived_of<kSums ? in.AHEAD - 1 : in.AHEAD>(0, ROWS, 0u);
        Rows<W> x = in.rows(0);
        centre<ELU>(x);
        float acc[NT][4];
        float x1[2], xa[2], ynu[2];                 // (1 + x') . 1, x' . a', Y . nu of rows g, g + 8
        {
            float u[4];
            vector_product<W>(u, x, vectors);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                x1[h] = fD + from_column(u, h, 3);
                if (MODE != kApplyBackwardKV) xa[h] = (from_column(u, h, 2) + from_column(u, h, 1)) + from_column(u, h, 0);
            }
        }
        if constexpr (MODE == kApplyForward) {
            product<W>(acc, x, smem + L::ROWWISE);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                // den = (1 + q') . (N 1 + Z');  num = (1 + q').1 nu + q' S''
                const float den = fN * x1[h] + a_sum + xa[h];
                const float inv = 1.f / (den + p.eps), w = x1[h] * inv;
                const f32x2 inv2 = sm100::pair(inv, inv), w2 = sm100::pair(w, w);
                uint32_t o[NT];
#pragma unroll
                for (int n = 0; n < NT; ++n)
                    o[n] = sm100::pack_bf16x2(sm100::fma2(sm100::pair(acc[n][2 * h], acc[n][2 * h + 1]), inv2, sm100::mul2(w2, of(nuH, n))));
                const int row = n0 + g + 8 * h;
                if (row < r.end) {
                    put_row<W>(p.out0, base + row, o);
                    if (p.den && t == 0) p.den[base + row] = den;
                }
            }
        } else {
            const Rows<W> y = in.rows(1);
            float u[4];
            vector_product<W>(u, y, vectors);
            product<W>(acc, y, smem + L::ROWWISE);              // h'' = G S''^T  /  V R''^T
            float scale[2], c1[2], cz[2];                       // out_d = scale * (acc_d + c1 + cz * a'_d)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                ynu[h] = (from_column(u, h, 6) + from_column(u, h, 5)) + from_column(u, h, 4);
                scale[h] = cz[h] = 1.f;
                c1[h] = ynu[h] + w0;
            }
            if constexpr (MODE == kApplyBackwardQ) {
                float qh[2];                        // (1 + x') . h''
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    f32x2 d = row_part(x.x[h], [&](int n) { return sm100::pair(acc[n][2 * h], acc[n][2 * h + 1]); });
#pragma unroll
                    for (int n = 0; n < NT; ++n) d = sm100::add2(d, sm100::pair(acc[n][2 * h], acc[n][2 * h + 1]));
                    qh[h] = across(d);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // h = (G.nu) 1 + h'',  Z = N 1 + Z',  gq = (h - (q.h / dn) Z) / dn
                    const float dn = fN * x1[h] + a_sum + xa[h] + p.eps;
                    scale[h] = 1.f / dn;
                    const float q_h = ynu[h] * x1[h] + qh[h];         // q . h
                    cz[h] = -q_h * scale[h];                                                  // dl_i = -(G_i . O_i)
                    c1[h] = fmaf(cz[h], fN, ynu[h]);                                          // (G.nu) + dl N
                }
                // operands of the reverse sums: the weighted queries x' / dn, and the planes of dl_i and 1 / dn_i
                Rows<W> xs;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool real = n0 + g + 8 * h < r.end;
                    const float wq = real ? scale[h] : 0.f, dl = real ? cz[h] : 0.f;
#pragma unroll
                    for (int n = 0; n < NT; ++n) xs.x[h][n] = sm100::pack_bf16x2(sm100::mul2(sm100::pair_bf16(x.x[h][n]), sm100::pair(wq, wq)));
                    if (t == 0) {
                        uint32_t pl[3];
                        split2<3>(dl, wq, pl);
                        uint16_t* w = reinterpret_cast<uint16_t*>(smem + L::PLANES + (odd ? WARPS * 256 : 0)) + warp * 64 + 8 * h + g;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            w[k * 16] = (uint16_t)pl[k];
                            w[WARPS * 64 + k * 16] = (uint16_t)(pl[k] >> 16);
                        }
                        w_sum = fmaf(dl, wq, w_sum);
                    }
                }
                in.put_rows(0, xs);
                __syncthreads();
                in.request(n0 + in.AHEAD * CHUNK);          // into the slot that every warp has left by now
                const uint16_t* planes = reinterpret_cast<const uint16_t*>(smem + L::PLANES + (odd ? WARPS * 256 : 0));
                const uint32_t slot = smem_u32(smem + L::RING + in.read);
                st.template add<true>(slot, slot + in.TILE, in.BYTES, min(WARPS, (r.end - c0 + ROWS - 1) / ROWS), planes, planes + WARPS * 64);
                odd = !odd;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const f32x2 s2 = sm100::pair(scale[h], scale[h]), z2 = sm100::pair(cz[h], cz[h]), c2 = sm100::pair(c1[h], c1[h]), one2 = sm100::pair(1.f, 1.f);
                uint32_t o[NT];
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    f32x2 v = sm100::mul2(s2, sm100::add2(sm100::fma2(z2, of(aH, n), sm100::pair(acc[n][2 * h], acc[n][2 * h + 1])), c2));
                    // phi'(x) from x' = elu(x): 1 where x' > 0, else 1 + x', i.e. 1 + min(x', 0)
                    if constexpr (ELU) v = sm100::mul2(v, sm100::add2(sm100::pair_bf16(sm100::min_bf16x2(x.x[h][n], 0u)), one2));
                    o[n] = sm100::pack_bf16x2(v);
                }
                if (n0 + g + 8 * h < r.end) put_row<W>(p.out0, base + n0 + g + 8 * h, o);
            }
            if constexpr (MODE == kApplyBackwardKV) {           // gV = (1 + k').1 nu_R + k' R''
                product<W>(acc, x, smem + L::COLWISE);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const f32x2 x2 = sm100::pair(x1[h], x1[h]);
                    uint32_t o[NT];
#pragma unroll
                    for (int n = 0; n < NT; ++n)
                        o[n] = sm100::pack_bf16x2(sm100::fma2(x2, of(nuH, n), sm100::pair(acc[n][2 * h], acc[n][2 * h + 1])));
                    if (n0 + g + 8 * h < r.end) put_row<W>(p.out1, base + n0 + g + 8 * h, o);
                }
            }
        }
        in.next();
    }
    if constexpr (kSums) {
        float* rec_out = p.rec_out + (int64_t)blockIdx.x * kRecFloats;
        if (lane % 4 == 0) {            // the lanes of t == 0, then the warps in their order
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) w_sum += __shfl_xor_sync(0x11111111u, w_sum, o);
        }
        if (lane == 0) sScal[4 + warp] = w_sum;
        __syncthreads();
        w_sum = 0.f;
        for (int k = 0; k < WARPS; ++k) w_sum += sScal[4 + k];
        st.put_record(reinterpret_cast<float*>(smem + L::RING), rec_out, w_sum);
    }
    zero_rows<W, THREADS>(p.out0, base + r.zero_lo, base + r.zero_hi);
    if (MODE == kApplyBackwardKV) zero_rows<W, THREADS>(p.out1, base + r.zero_lo, base + r.zero_hi);
    if (MODE == kApplyForward && p.den)
        for (int64_t i = base + r.zero_lo + tid; i < base + r.zero_hi; i += THREADS) p.den[i] = 0.f;
}

}  // namespace lin
}  // namespace tc
}  // namespace la
