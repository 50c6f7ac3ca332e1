// Causal form (Eq. 8-15) at fp32 accuracy on mma.sync (la_mma.cuh): fp32 problems, and bf16 ones of shapes or feature
// maps that the tcgen05 kernels do not take; M <= 64, any D.  Also bf16 problems with D = M = 32, on kernels of
// their own (la_causal_warp.cuh).
//
// A sequence is cut into pieces, one CTA each; a CTA walks its piece in chunks of T = 64 positions.  Per chunk a strip of
// sixteen rows (queries in the forward sweeps, keys in the reverse one) belongs to a pair of warps, and so do sixteen
// rows of the running state, kept in fp32 registers.  The operands that all warps read (K | V, or Q / dn | G) and the
// state before the chunk lie in shared memory as bf16 planes; scores never leave the registers of their warp.
//
//   forward   O  = [(q k^T o L) [V | 1] + q [S | Z]],            S += k^T V,  Z += k^T 1
//   dQ sweep  h  = (G V^T o L) k + G S^T,  Zc = L k + Z,  dn = q . Zc + eps,
//             gq = (h - (q . h / dn) Zc) / dn                     (the same S, Z; dn and -(q . h) / dn are parked)
//   dK, dV    with q^ = q / dn, dl = -G . O:  gV = (q^ k^T o L)^T G + k R,
//             gk = ((G V^T + dl) o L)^T q^ + V R^T + r,           R += q^^T G,  r += q^^T dl  (chunks last to first)
//
// The two warps of a strip share the products: forward, one the state's part and one the scores' part; dQ, one G S^T and
// L k, one the scores' part; reverse, one dV and one dK.  The partial sums of the first two are added through shared
// memory (the state planes, once nobody reads them any more).  Two warps per strip at 128 registers keep four warps on
// a scheduler; one warp per strip at 168 to 255 registers kept two, and the tensor pipe 45 % busy.
//
// Pieces other than the first (last, for the reverse sweep) start from the sum of the records [S | Z] of the pieces
// before (after) them, which a pre-pass writes to the workspace.
#include <math.h>
#include <stdlib.h>

#include <type_traits>

#include "la_causal_warp.cuh"
#include "la_mma_sweep.cuh"

namespace la {
namespace {

using namespace mma;
using namespace sweep;

template <typename C, int DP, int MP> using ForwardLayout = Layout<C::WPS, DP, MP, C::NQ, C::NV, C::NQ, DP, C::NS, MP>;
template <typename C, int DP, int MP> using DqLayout = Layout<C::WPS, DP, MP, C::NQ, C::NV, C::NV, MP, C::NS, DP>;
// (kScaled: after the vectors G / dn in three planes, and 1 / dn)
template <typename C, int DP, int MP> struct DkvLayout : Layout<C::WPS, DP, MP, kScaled<C> ? 1 : C::NR, C::NV, 0, 0, C::NS, 0> {
    using Base = Layout<C::WPS, DP, MP, kScaled<C> ? 1 : C::NR, C::NV, 0, 0, C::NS, 0>;
    static constexpr int GH = Base::BYTES, INV = GH + 3 * T * MP * 2, BYTES = kScaled<C> ? INV + T * 4 : Base::BYTES;
};

// named barriers: 1 = the state planes are no longer read; 2 + strip, 6 + strip = hand-overs within a pair of warps
__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int threads) {
    __threadfence_block();
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// a strip's partial results between its two warps, whose lanes hold the same positions
template <int NT8>
__device__ __forceinline__ void put_part(uint8_t* area, int strip, const float (&x)[NT8][4]) {
    float4* d = reinterpret_cast<float4*>(area) + strip * NT8 * 32 + (threadIdx.x & 31);
#pragma unroll
    for (int n = 0; n < NT8; ++n) d[n * 32] = make_float4(x[n][0], x[n][1], x[n][2], x[n][3]);
}
template <int NT8>
__device__ __forceinline__ void add_part(const uint8_t* area, int strip, float (&x)[NT8][4]) {
    const float4* d = reinterpret_cast<const float4*>(area) + strip * NT8 * 32 + (threadIdx.x & 31);
#pragma unroll
    for (int n = 0; n < NT8; ++n) {
        const float4 v = d[n * 32];
        x[n][0] += v.x; x[n][1] += v.y; x[n][2] += v.z; x[n][3] += v.w;
    }
}
// The A operand of a strip: planes in registers (one warp per strip), or read from a tile block by block (two warps).
template <int WPS, int NP, int C> struct StripOperand;
template <int NP, int C> struct StripOperand<1, NP, C> {
    uint32_t a[C / 16][NP][4];
    __device__ __forceinline__ const uint32_t (&block(int kk, uint32_t (&)[NP][4]) const)[NP][4] { return a[kk]; }
};
template <int NP, int C> struct StripOperand<2, NP, C> {
    uint32_t tile;
    int row0, lane;
    __device__ __forceinline__ const uint32_t (&block(int kk, uint32_t (&f)[NP][4]) const)[NP][4] {
        load_cols<NP, C>(f, tile, T * C * 2, row0, kk * 2, lane);
        return f;
    }
};

// The strip of a warp.  It alternates with the chunk, so that the strips with the most blocks go round the schedulers, and
// the second four warps have them the other way round, so that the two warps of a scheduler together have a middling load.
__device__ __forceinline__ int strip_of(int warp, bool odd) {
    const int s = warp % STRIPS_T;
    return odd != (warp >= STRIPS_T) ? STRIPS_T - 1 - s : s;
}

// zero the scores of a diagonal block: columns right of the row (UPPER: left of it)
template <bool UPPER>
__device__ __forceinline__ void mask_diagonal(float (&s0)[4], float (&s1)[4], int g, int t) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int row = g + (j >> 1) * 8, col = 2 * t + (j & 1);
        if (UPPER ? col < row : col > row) s0[j] = 0.f;
        if (UPPER ? col + 8 < row : col + 8 > row) s1[j] = 0.f;
    }
}

// ---- forward ---------------------------------------------------------------------------------------------------
template <typename C, int DP, int MP, bool EXACT>
__global__ void __launch_bounds__(kThreads<C>, (C::ALONE ? 1 : resident<ForwardLayout<C, DP, MP>>()))
causal_mma_forward_kernel(const Params p) {
    using IO = typename C::IO;
    using Sh = ForwardLayout<C, DP, MP>;
    constexpr int NQ = C::NQ, NV = C::NV, NP = C::NP, NS = C::NS, WPS = C::WPS, THREADS = kThreads<C>;
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const bool state_part = WPS == 1 || warp < STRIPS_T, score_part = WPS == 1 || warp >= STRIPS_T;
    const int D = EXACT ? DP : p.D, M = EXACT ? MP : p.M, phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    wait_for_stream();
    release_next();
    const Range r = range_of(p, blockIdx.y);
    const IO* Q = (const IO*)p.Q + r.bh * p.N * D;
    const IO* K = (const IO*)p.K + r.bh * p.N * D;
    const IO* V = (const IO*)p.V + r.bh * p.N * M;
    IO* O = (IO*)p.O + r.bh * p.N * M;
    float* den = p.den ? p.den + r.bh * p.N : nullptr;

    State<DP, MP, 4 * WPS> st;
    st.init(p, p.S0 ? p.S0 + r.bh * D * M : nullptr, p.Z0 ? p.Z0 + r.bh * D : nullptr,
            p.rec + r.bh * p.records * (int64_t)(D * M + D), r.piece * parts_of<C, EXACT>(p));
    for (int64_t n0 = r.lo; n0 < r.end; n0 += T) {
        const uint32_t sK = smem_u32(smem + Sh::X), sV = smem_u32(smem + Sh::Y), sS = smem_u32(smem + Sh::S);
        float* sZ = reinterpret_cast<float*>(smem + Sh::Z);
        uint16_t* sZp = reinterpret_cast<uint16_t*>(smem + Sh::ZP);
        float* sden = reinterpret_cast<float*>(smem + Sh::W);
        const int cn = (int)(r.end - n0 < T ? r.end - n0 : T);
        const int strip = strip_of(warp, (n0 / T) & 1), row0 = strip * 16;
        StripOperand<WPS, NQ, DP> q;
        {
            RawTile<IO, T, DP, THREADS> rk;
            RawTile<IO, T, MP, THREADS> rv;
            std::conditional_t<WPS == 1, RawStrip<IO, DP>, RawTile<IO, T, DP, THREADS>> rq;
            rk.load(K + n0 * D, cn, D, pad);
            rv.load(V + n0 * M, cn, M, 0.f);
            if constexpr (WPS == 1) rq.load(Q + n0 * D, row0, cn, D, pad);
            else rq.load(Q + n0 * D, cn, D, pad);
            __syncthreads();         // the planes of the chunk before are no longer read
            st.template publish<NS>(smem + Sh::S, sZ, sZp);
            rk.template features<NQ>(smem + Sh::X, phi);
            rv.template values<NV>(smem + Sh::Y);
            if constexpr (WPS == 1) {
                RawStrip<typename FeatureType<NQ>::type, DP> fq;
                rq.template map<NQ>(phi, fq);
                fq.template planes<NQ>(q.a);
            } else {
                rq.template features<NQ>(smem + Sh::R, phi);
                q.tile = smem_u32(smem + Sh::R); q.row0 = row0; q.lane = lane;
            }
        }
        prefetch_rows<C>(Q, n0 + T, r.end, D);
        prefetch_rows<C>(K, n0 + T, r.end, D);
        prefetch_rows<C>(V, n0 + T, r.end, M);
        __syncthreads();
        const bool real = row0 < cn;
        float o[MP / 8][4], d0 = 0.f, d1 = 0.f;         // rows g, g + 8 of [num | den]; d0, d1 spread over the four lanes
        auto scores = [&](int from, int to) {           // o += ((q k^T) o L) V, d0, d1 += its row sums, key blocks from .. to
#pragma unroll 1
            for (int jb = from; jb <= to; ++jb) {
                float s0[4], s1[4];
                {
                    Chain c;
#pragma unroll
                    for (int kk = 0; kk < DP / 16; ++kk) {
                        uint32_t b[NQ][4], f[NQ][4];
                        load_rows<NQ, DP>(b, sK, T * DP * 2, jb * 16, kk * 2, lane);
                        c.step<NQ, NQ>(q.block(kk, f), b);
                    }
                    c.put(s0, s1);
                }
                if (jb == strip) mask_diagonal<false>(s0, s1, g, t);
                uint32_t pa[NP][4];
                operand_of<NP>(pa, s0, s1);
                d0 += (s0[0] + s0[1]) + (s1[0] + s1[1]);
                d1 += (s0[2] + s0[3]) + (s1[2] + s1[3]);
#pragma unroll
                for (int n = 0; n < MP / 16; ++n) {
                    uint32_t b[NV][4];
                    load_cols_t<NV, MP>(b, sV, T * MP * 2, jb * 16, n * 2, lane);
                    block_mma<NP, NV>(o[2 * n], o[2 * n + 1], pa, b);
                }
            }
        };
        // (long strips: the warp of the state's part takes the first block of scores as well)
        const bool shared_block = WPS == 2 && strip >= 2;
        if (state_part) {
            if (real) {
#pragma unroll
                for (int n = 0; n < MP / 16; ++n) {
                    Chain c;
#pragma unroll
                    for (int kk = 0; kk < DP / 16; ++kk) {
                        uint32_t b[NS][4], f[NQ][4];
                        load_cols_t<NS, MP>(b, sS, DP * MP * 2, kk * 16, n * 2, lane);
                        c.step<NQ, NS>(q.block(kk, f), b);
                    }
                    c.put(o[2 * n], o[2 * n + 1]);
                }
#pragma unroll
                for (int kk = 0; kk < DP / 16; ++kk) {
                    float u[4] = {0.f, 0.f, 0.f, 0.f};
                    uint32_t f[NQ][4];
                    vector_mma<NQ, DP>(u, q.block(kk, f), sZp, kk * 16, t);
                    d0 += t == 0 ? u[0] : 0.f;
                    d1 += t == 0 ? u[2] : 0.f;
                }
                if (shared_block) scores(0, 0);
            }
            if constexpr (WPS == 2) {
                bar_sync(1, 128);
                if (real) {
                    put_part(smem + Sh::S, strip, o);
                    d0 = quad_sum(d0);
                    d1 = quad_sum(d1);
                    if (t == 0) {
                        sden[row0 + g] = d0;
                        sden[row0 + g + 8] = d1;
                    }
                    bar_arrive(2 + strip, 64);
                }
            }
        }
        if (score_part && real) {
            if constexpr (WPS == 2) clear(o);
            scores(shared_block ? 1 : 0, strip);
            d0 = quad_sum(d0);
            d1 = quad_sum(d1);
            if constexpr (WPS == 2) {
                bar_sync(2 + strip, 64);
                add_part(smem + Sh::S, strip, o);
                d0 += sden[row0 + g];
                d1 += sden[row0 + g + 8];
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = row0 + g + 8 * h;
                const float inv = 1.f / ((h ? d1 : d0) + p.eps);
                if (row < cn) {
#pragma unroll
                    for (int n = 0; n < MP / 8; ++n)
                        if (n * 8 < M) store_pair<IO>(O + (n0 + row) * M + n * 8 + 2 * t, o[n][2 * h] * inv, o[n][2 * h + 1] * inv);
                    if (den && t == 0) den[n0 + row] = h ? d1 : d0;
                }
            }
        }
        st.template update<NQ, NV, true>(sK, sV, nullptr);
    }
    zero_rows<THREADS>(O, r.end, r.hi, M);
    if (den) zero_rows<THREADS>(den, r.end, r.hi, 1);
    if (r.piece == p.pieces - 1) st.write(p, p.S1 ? p.S1 + r.bh * D * M : nullptr, p.Z1 ? p.Z1 + r.bh * D : nullptr);
}

// ---- dQ sweep --------------------------------------------------------------------------------------------------
template <typename C, int DP, int MP, bool EXACT>
__global__ void __launch_bounds__(kThreads<C>, (C::ALONE ? 1 : resident<DqLayout<C, DP, MP>>()))
causal_mma_dq_kernel(const Params p) {
    using IO = typename C::IO;
    using Sh = DqLayout<C, DP, MP>;
    constexpr int NQ = C::NQ, NV = C::NV, NP = C::NP, NS = C::NS, WPS = C::WPS, THREADS = kThreads<C>;
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const bool state_part = WPS == 1 || warp < STRIPS_T, score_part = WPS == 1 || warp >= STRIPS_T;
    const int D = EXACT ? DP : p.D, M = EXACT ? MP : p.M, phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    wait_for_stream();
    release_next();
    const Range r = range_of(p, blockIdx.y);
    const IO* Q = (const IO*)p.Q + r.bh * p.N * D;
    const IO* K = (const IO*)p.K + r.bh * p.N * D;
    const IO* V = (const IO*)p.V + r.bh * p.N * M;
    const IO* G = (const IO*)p.G + r.bh * p.N * M;
    IO* dQ = (IO*)p.dQ + r.bh * p.N * D;
    float* dn_all = p.aux + r.bh * 2 * p.N;
    float* dl_all = dn_all + p.N;

    State<DP, MP, 4 * WPS> st;
    st.init(p, p.S0 ? p.S0 + r.bh * D * M : nullptr, p.Z0 ? p.Z0 + r.bh * D : nullptr,
            p.rec + r.bh * p.records * (int64_t)(D * M + D), r.piece * parts_of<C, EXACT>(p));
    for (int64_t n0 = r.lo; n0 < r.end; n0 += T) {
        const uint32_t sK = smem_u32(smem + Sh::X), sV = smem_u32(smem + Sh::Y), sS = smem_u32(smem + Sh::S);
        float* sZ = reinterpret_cast<float*>(smem + Sh::Z);
        float* sgo = reinterpret_cast<float*>(smem + Sh::W);
        const int cn = (int)(r.end - n0 < T ? r.end - n0 : T);
        const int strip = strip_of(warp, (n0 / T) & 1), row0 = strip * 16;
        StripOperand<WPS, NV, MP> ga;
        {
            RawTile<IO, T, DP, THREADS> rk;
            RawTile<IO, T, MP, THREADS> rv;
            std::conditional_t<WPS == 1, RawStrip<IO, MP>, RawTile<IO, T, MP, THREADS>> rg;
            rk.load(K + n0 * D, cn, D, pad);
            rv.load(V + n0 * M, cn, M, 0.f);
            if constexpr (WPS == 1) rg.load(G + n0 * M, row0, cn, M, 0.f);
            else rg.load(G + n0 * M, cn, M, 0.f);
            __syncthreads();
            st.template publish<NS>(smem + Sh::S, sZ, reinterpret_cast<uint16_t*>(smem + Sh::ZP));
            rk.template features<NQ>(smem + Sh::X, phi);
            rv.template values<NV>(smem + Sh::Y);
            if constexpr (WPS == 1) {
                rg.template planes<NV>(ga.a);
            } else {
                rg.template values<NV>(smem + Sh::R);
                ga.tile = smem_u32(smem + Sh::R); ga.row0 = row0; ga.lane = lane;
            }
        }
        prefetch_rows<C>(Q, n0 + T, r.end, D);
        prefetch_rows<C>(K, n0 + T, r.end, D);
        prefetch_rows<C>(V, n0 + T, r.end, M);
        prefetch_rows<C>(G, n0 + T, r.end, M);
        __syncthreads();
        const bool real = row0 < cn;
        // The first chunk of a sequence goes through twice, the second time with the G_i . O_i it found taken off the
        // scores: where few terms make up a row, h and (q . h / dn) Zc cancel almost entirely (in row 0 completely).
        // (A state it continues from may be zero as well and is treated alike, its part of h included, by single warps;
        // pairs have overwritten its planes by then and go through twice only where it has no part.)
        const int first_pass = n0 == 0 && (WPS == 1 || !p.S0) ? 0 : 1;
        float c0 = 0.f, c1 = 0.f;               // G_i . O_i of rows g, g + 8, as far as it is known
        float h[DP / 8][4], zc[DP / 8][4];
        auto ones_block = [&](uint32_t (&ones)[1][4], int jb) {         // the part of L in key block jb
            ones[0][0] = ones[0][1] = ones[0][2] = ones[0][3] = 0x3f803f80u;
            if (jb == strip) {
                ones[0][0] = ones[0][3] = (2 * t <= g ? 0x3f80u : 0u) | (2 * t + 1 <= g ? 0x3f800000u : 0u);
                ones[0][2] = 0u;
            }
        };
        auto start_zc = [&]() {
#pragma unroll
            for (int n = 0; n < DP / 8; ++n) {
                const float2 z = *reinterpret_cast<const float2*>(sZ + n * 8 + 2 * t);
                zc[n][0] = zc[n][2] = z.x;
                zc[n][1] = zc[n][3] = z.y;
            }
        };
        auto scores = [&]() {                   // h += ((G V^T - c) o L) k; one warp per strip: zc = L k + Z as well
            if constexpr (WPS == 1) start_zc();
#pragma unroll 1
            for (int jb = 0; jb <= strip; ++jb) {
                float s0[4], s1[4];
                {
                    Chain c;
#pragma unroll
                    for (int ee = 0; ee < MP / 16; ++ee) {
                        uint32_t b[NV][4], f[NV][4];
                        load_rows<NV, MP>(b, sV, T * MP * 2, jb * 16, ee * 2, lane);
                        c.step<NV, NV>(ga.block(ee, f), b);
                    }
                    c.put(s0, s1);
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    s0[j] -= c0; s1[j] -= c0;
                    s0[2 + j] -= c1; s1[2 + j] -= c1;
                }
                if (jb == strip) mask_diagonal<false>(s0, s1, g, t);
                uint32_t pa[NP][4], ones[1][4];
                operand_of<NP>(pa, s0, s1);
                if constexpr (WPS == 1) ones_block(ones, jb);
#pragma unroll
                for (int n = 0; n < DP / 16; ++n) {
                    uint32_t b[NQ][4];
                    load_cols_t<NQ, DP>(b, sK, T * DP * 2, jb * 16, n * 2, lane);
                    block_mma<NP, NQ>(h[2 * n], h[2 * n + 1], pa, b);
                    if constexpr (WPS == 1) block_mma<1, NQ>(zc[2 * n], zc[2 * n + 1], ones, b);
                }
            }
        };
        if (WPS == 2 && score_part) {
            for (int pass = first_pass; pass < 2; ++pass) {
                if (real) {
                    clear(h);
                    scores();
                }
                if (pass == first_pass) bar_sync(1, THREADS);
                if (real) {
                    put_part(smem + Sh::S, strip, h);
                    bar_arrive(2 + strip, 64);
                    if (pass == 0) {
                        bar_sync(6 + strip, 64);
                        c0 = sgo[row0 + g];
                        c1 = sgo[row0 + g + 8];
                    }
                }
            }
        }
        auto state_product = [&]() {            // h = G S^T
#pragma unroll
            for (int n = 0; n < DP / 16; ++n) {
                Chain c;
#pragma unroll
                for (int ee = 0; ee < MP / 16; ++ee) {
                    uint32_t b[NS][4], f[NV][4];
                    load_rows<NS, MP>(b, sS, DP * MP * 2, n * 16, ee * 2, lane);
                    c.step<NV, NS>(ga.block(ee, f), b);
                }
                c.put(h[2 * n], h[2 * n + 1]);
            }
        };
        if (state_part) {
            if (WPS == 2 && real) state_product();
            if constexpr (WPS == 2) bar_arrive(1, THREADS);
            if (real) {
                if constexpr (WPS == 2) {
                    start_zc();
#pragma unroll 1
                    for (int jb = 0; jb <= strip; ++jb) {
                        uint32_t ones[1][4];
                        ones_block(ones, jb);
#pragma unroll
                        for (int n = 0; n < DP / 16; ++n) {
                            uint32_t b[NQ][4];
                            load_cols_t<NQ, DP>(b, sK, T * DP * 2, jb * 16, n * 2, lane);
                            block_mma<1, NQ>(zc[2 * n], zc[2 * n + 1], ones, b);
                        }
                    }
                }
                for (int pass = first_pass; pass < 2; ++pass) {
                    if constexpr (WPS == 1) {
                        state_product();
                        if (pass > first_pass) {            // the second time: take G_i . O_i off the state's part too
#pragma unroll
                            for (int n = 0; n < DP / 8; ++n) {
                                const float2 z = *reinterpret_cast<const float2*>(sZ + n * 8 + 2 * t);
                                h[n][0] = fmaf(-c0, z.x, h[n][0]); h[n][1] = fmaf(-c0, z.y, h[n][1]);
                                h[n][2] = fmaf(-c1, z.x, h[n][2]); h[n][3] = fmaf(-c1, z.y, h[n][3]);
                            }
                        }
                    } else if (pass > first_pass) {
                        clear(h);
                    }
                    RawStrip<IO, DP> rq;        // element j of block kk: result column tile 2 kk + j / 2, row g + 8 (j & 1)
                    if constexpr (WPS == 2) {
                        rq.load(Q + n0 * D, row0, cn, D, pad);
                        bar_sync(2 + strip, 64);
                        add_part(smem + Sh::S, strip, h);
                    } else {
                        scores();
                        rq.load(Q + n0 * D, row0, cn, D, pad);
                    }
                    RawStrip<typename FeatureType<NQ>::type, DP> fq;
                    rq.template map<NQ>(phi, fq);
                    float qz[2] = {0.f, 0.f}, qh[2] = {0.f, 0.f};
#pragma unroll
                    for (int kk = 0; kk < DP / 16; ++kk)
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int n = 2 * kk + (j >> 1), b = j & 1;
                            qz[b] = fmaf(fq.r[kk][j].lo(), zc[n][2 * b], fmaf(fq.r[kk][j].hi(), zc[n][2 * b + 1], qz[b]));
                            qh[b] = fmaf(fq.r[kk][j].lo(), h[n][2 * b], fmaf(fq.r[kk][j].hi(), h[n][2 * b + 1], qh[b]));
                        }
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                        const int row = row0 + g + 8 * b;
                        const float dn = quad_sum(qz[b]) + p.eps;
                        const float inv = 1.f / dn;
                        const float go = (quad_sum(qh[b]) - (b ? c1 : c0) * p.eps) * inv;    // what is left of G_i . O_i
                        (b ? c1 : c0) += go;
                        if (pass == 1 && row < cn) {
#pragma unroll
                            for (int n = 0; n < DP / 8; ++n)
                                if (n * 8 < D) {
                                    const auto q = fq.r[n >> 1][(n & 1) * 2 + b];
                                    store_pair<IO>(dQ + (n0 + row) * D + n * 8 + 2 * t,
                                                   fmaf(-go, zc[n][2 * b], h[n][2 * b]) * inv * phi_slope_from_value(q.lo(), phi),
                                                   fmaf(-go, zc[n][2 * b + 1], h[n][2 * b + 1]) * inv * phi_slope_from_value(q.hi(), phi));
                                }
                            if (t == 0) {
                                dn_all[n0 + row] = dn;
                                dl_all[n0 + row] = b ? -c1 : -c0;
                            }
                        }
                    }
                    if (WPS == 2 && pass == 0) {
                        if (t == 0) {
                            sgo[row0 + g] = c0;
                            sgo[row0 + g + 8] = c1;
                        }
                        bar_arrive(6 + strip, 64);
                    }
                }
            }
        }
        st.template update<NQ, NV, true>(sK, sV, nullptr);
    }
    zero_rows<THREADS>(dQ, r.end, r.hi, D);
}

// ---- dK, dV sweep ----------------------------------------------------------------------------------------------
template <typename C, int DP, int MP, bool EXACT>
__global__ void __launch_bounds__(kThreads<C>, (C::ALONE ? 1 : resident<DkvLayout<C, DP, MP>>(C::WPS == 1 ? 3 : 2)))
causal_mma_dkv_kernel(const Params p) {
    using IO = typename C::IO;
    using Sh = DkvLayout<C, DP, MP>;
    constexpr int NQ = C::NQ, NV = C::NV, NP = C::NP, NS = C::NS, WPS = C::WPS, THREADS = kThreads<C>;
    constexpr bool SCALED = kScaled<C>;
    constexpr int NX = SCALED ? 1 : C::NR;          // planes of the queries' tile
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const bool v_part = WPS == 1 || warp < STRIPS_T, k_part = WPS == 1 || warp >= STRIPS_T;
    const int D = EXACT ? DP : p.D, M = EXACT ? MP : p.M, phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    wait_for_stream();
    release_next();
    const Range r = range_of(p, (int)(gridDim.y - 1 - blockIdx.y));
    const IO* Q = (const IO*)p.Q + r.bh * p.N * D;
    const IO* K = (const IO*)p.K + r.bh * p.N * D;
    const IO* V = (const IO*)p.V + r.bh * p.N * M;
    const IO* G = (const IO*)p.G + r.bh * p.N * M;
    IO* dK = (IO*)p.dK + r.bh * p.N * D;
    IO* dV = (IO*)p.dV + r.bh * p.N * M;
    const float* dn = p.aux + r.bh * 2 * p.N;
    const float* delta = dn + p.N;

    State<DP, MP, 4 * WPS> st;           // record i is the sum of piece i + 1
    st.init(p, p.S0 ? p.S0 + r.bh * D * M : nullptr, p.Z0 ? p.Z0 + r.bh * D : nullptr,
            p.rec + (r.bh * p.records + r.piece * parts_of<C, EXACT>(p)) * (int64_t)(D * M + D), (p.pieces - 1 - r.piece) * parts_of<C, EXACT>(p));
    const int64_t chunks = (r.end - r.lo + T - 1) / T;
    for (int64_t c = chunks - 1; c >= 0; --c) {
        const uint32_t sQ = smem_u32(smem + Sh::X), sG = smem_u32(smem + Sh::Y), sR = smem_u32(smem + Sh::S);
        float* sr = reinterpret_cast<float*>(smem + Sh::Z);
        float* sdl = reinterpret_cast<float*>(smem + Sh::W);
        uint16_t* wpl = reinterpret_cast<uint16_t*>(smem + Sh::WP);
        const int64_t n0 = r.lo + c * T;
        const int cn = (int)(r.end - n0 < T ? r.end - n0 : T), blocks = (cn + 15) / 16;
        const int strip = strip_of(warp, c & 1), row0 = strip * 16;
        {
            std::conditional_t<SCALED, ScaledRows<IO, DP, MP, THREADS>, ReverseRows<IO, DP, MP, THREADS>> rr;
            rr.load(Q, G, dn, delta, n0, cn, D, M, pad);
            __syncthreads();
            st.template publish<NS>(smem + Sh::S, sr, reinterpret_cast<uint16_t*>(smem + Sh::ZP));
            if constexpr (SCALED) rr.store(smem + Sh::X, smem + Sh::Y, smem + Sh::GH, sdl, reinterpret_cast<float*>(smem + Sh::INV), wpl);
            else rr.template store<C::NR, NV>(smem + Sh::X, smem + Sh::Y, sdl, wpl, phi);
        }
        if (c > 0) {
            prefetch_rows<C>(Q, n0 - T, r.end, D);
            prefetch_rows<C>(K, n0 - T, r.end, D);
            prefetch_rows<C>(V, n0 - T, r.end, M);
            prefetch_rows<C>(G, n0 - T, r.end, M);
        }
        __syncthreads();
        auto scale_columns = [&](int ib, float (&s0)[4], float (&s1)[4]) {       // the scores of queries 16 ib .. by their 1 / dn
            const float* v = reinterpret_cast<const float*>(smem + Sh::INV) + ib * 16 + 2 * t;
            const float2 i0 = load_pair(v), i1 = load_pair(v + 8);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                s0[2 * h] *= i0.x; s0[2 * h + 1] *= i0.y;
                s1[2 * h] *= i1.x; s1[2 * h + 1] *= i1.y;
            }
        };
        if (v_part && row0 < cn) {
            uint32_t ka[DP / 16][NQ][4];
            {
                RawStrip<IO, DP> rk;
                rk.load(K + n0 * D, row0, cn, D, pad);
                RawStrip<typename FeatureType<NQ>::type, DP> fk;
                rk.template map<NQ>(phi, fk);
                fk.template planes<NQ>(ka);
            }
            float gv[MP / 8][4];
#pragma unroll
            for (int n = 0; n < MP / 16; ++n) {
                Chain c;
#pragma unroll
                for (int kk = 0; kk < DP / 16; ++kk) {
                    uint32_t b[NS][4];
                    load_cols_t<NS, MP>(b, sR, DP * MP * 2, kk * 16, n * 2, lane);
                    c.step<NQ, NS>(ka[kk], b);
                }
                c.put(gv[2 * n], gv[2 * n + 1]);
            }
#pragma unroll 1
            for (int ib = strip; ib < blocks; ++ib) {
                float s0[4], s1[4];
                {
                    Chain c;
#pragma unroll
                    for (int kk = 0; kk < DP / 16; ++kk) {
                        uint32_t b[NX][4];
                        load_rows<NX, DP>(b, sQ, T * DP * 2, ib * 16, kk * 2, lane);
                        c.step<NQ, NX>(ka[kk], b);
                    }
                    c.put(s0, s1);
                }
                if constexpr (SCALED) scale_columns(ib, s0, s1);
                if (ib == strip) mask_diagonal<true>(s0, s1, g, t);
                uint32_t pa[NP][4];
                operand_of<NP>(pa, s0, s1);
#pragma unroll
                for (int n = 0; n < MP / 16; ++n) {
                    uint32_t b[NV][4];
                    load_cols_t<NV, MP>(b, sG, T * MP * 2, ib * 16, n * 2, lane);
                    block_mma<NP, NV>(gv[2 * n], gv[2 * n + 1], pa, b);
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = row0 + g + 8 * h;
                if (row < cn) {
#pragma unroll
                    for (int n = 0; n < MP / 8; ++n)
                        if (n * 8 < M) store_pair<IO>(dV + (n0 + row) * M + n * 8 + 2 * t, gv[n][2 * h], gv[n][2 * h + 1]);
                }
            }
        }
        if (k_part && row0 < cn) {
            uint32_t va[MP / 16][NV][4];
            {
                RawStrip<IO, MP> rv;
                rv.load(V + n0 * M, row0, cn, M, 0.f);
                rv.template planes<NV>(va);
            }
            float gk[DP / 8][4];
#pragma unroll
            for (int n = 0; n < DP / 8; ++n) {
                const float2 z = *reinterpret_cast<const float2*>(sr + n * 8 + 2 * t);
                gk[n][0] = gk[n][2] = z.x;
                gk[n][1] = gk[n][3] = z.y;
            }
#pragma unroll
            for (int n = 0; n < DP / 16; ++n) {
                Chain c;
#pragma unroll
                for (int ee = 0; ee < MP / 16; ++ee) {
                    uint32_t b[NS][4];
                    load_rows<NS, MP>(b, sR, DP * MP * 2, n * 16, ee * 2, lane);
                    c.step<NV, NS>(va[ee], b);
                }
                c.add_to(gk[2 * n], gk[2 * n + 1]);
            }
#pragma unroll 1
            for (int ib = strip; ib < blocks; ++ib) {
                const float2 w0 = *reinterpret_cast<const float2*>(sdl + ib * 16 + 2 * t);
                const float2 w1 = *reinterpret_cast<const float2*>(sdl + ib * 16 + 8 + 2 * t);
                float s0[4] = {w0.x, w0.y, w0.x, w0.y}, s1[4] = {w1.x, w1.y, w1.x, w1.y};
                {
                    Chain c;
#pragma unroll
                    for (int ee = 0; ee < MP / 16; ++ee) {
                        uint32_t b[NV][4];
                        load_rows<NV, MP>(b, sG, T * MP * 2, ib * 16, ee * 2, lane);
                        c.step<NV, NV>(va[ee], b);
                    }
                    c.add_to(s0, s1);
                }
                if constexpr (SCALED) scale_columns(ib, s0, s1);
                if (ib == strip) mask_diagonal<true>(s0, s1, g, t);
                uint32_t pa[NP][4];
                operand_of<NP>(pa, s0, s1);
#pragma unroll
                for (int n = 0; n < DP / 16; ++n) {
                    uint32_t b[NX][4];
                    load_cols_t<NX, DP>(b, sQ, T * DP * 2, ib * 16, n * 2, lane);
                    block_mma<NP, NX>(gk[2 * n], gk[2 * n + 1], pa, b);
                }
            }
            RawStrip<IO, DP> rk;
            rk.load(K + n0 * D, row0, cn, D, pad);
            RawStrip<typename FeatureType<NQ>::type, DP> fk;
            rk.template map<NQ>(phi, fk);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = row0 + g + 8 * h;
                if (row < cn) {
#pragma unroll
                    for (int n = 0; n < DP / 8; ++n)
                        if (n * 8 < D) {
                            const auto k = fk.r[n >> 1][(n & 1) * 2 + h];
                            store_pair<IO>(dK + (n0 + row) * D + n * 8 + 2 * t, gk[n][2 * h] * phi_slope_from_value(k.lo(), phi),
                                           gk[n][2 * h + 1] * phi_slope_from_value(k.hi(), phi));
                        }
                }
            }
        }
        if constexpr (SCALED) st.template update<1, 3, false>(sQ, smem_u32(smem + Sh::GH), wpl);
        else st.template update<C::NR, NV, false>(sQ, sG, wpl);
    }
    zero_rows<THREADS>(dK, r.end, r.hi, D);
    zero_rows<THREADS>(dV, r.end, r.hi, M);
    if (r.piece == 0) st.write(p, p.S1 ? p.S1 + r.bh * D * M : nullptr, p.Z1 ? p.Z1 + r.bh * D : nullptr);
}

// ---- bf16, D = M = 32: a warp per piece (la_causal_warp.cuh) -----------------------------------------------------
enum WarpPass { kWarpForward, kWarpSums, kWarpDq, kWarpDqReverse, kWarpReverseSums, kWarpDkv, kWarpDkvFew };
constexpr int warp_ring(int pass) {
    return pass == kWarpForward ? warp32::Ring<3, false>::BYTES : pass == kWarpSums ? warp32::Ring<2, false>::BYTES :
           pass == kWarpReverseSums ? warp32::Ring<2, true>::BYTES : pass >= kWarpDkv ? warp32::Ring<4, true>::BYTES : warp32::Ring<4, false>::BYTES;
}
// Registers for twelve warps on an SM; for eight in the dQ sweep that keeps two kinds of sums, and in the dK, dV sweep where all warps find
// room that way too (128x8x784 157.5 -> 155.7 us a step, 111x8x300 73.1 -> 71.7, but 200x8x640 190 -> 200).
constexpr int warp_resident(int pass) {
    return pass == kWarpDqReverse || pass == kWarpDkvFew ? 8 : pass == kWarpSums || pass == kWarpReverseSums ? 16 : 12;
}
template <int PASS> constexpr int kWarpRing = warp_ring(PASS);
template <int PASS, bool ELU>
__global__ void __launch_bounds__(32, warp_resident(PASS)) causal_warp_kernel(const Params p) {
    __shared__ __align__(128) uint8_t smem[kWarpRing<PASS>];
    wait_for_stream();
    release_next();
    if constexpr (PASS == kWarpForward) warp32::forward<ELU>(p, smem);
    if constexpr (PASS == kWarpSums) warp32::sums<ELU>(p, smem);
    if constexpr (PASS == kWarpDq) warp32::dq<ELU, false>(p, smem);
    if constexpr (PASS == kWarpDqReverse) warp32::dq<ELU, true>(p, smem);
    if constexpr (PASS == kWarpReverseSums) warp32::reverse_sums<ELU>(p, smem);
    if constexpr (PASS >= kWarpDkv) warp32::dkv<ELU>(p, smem);
}

// ---- host ------------------------------------------------------------------------------------------------------
// Which bf16 problems with D = M = 32 a warp per piece takes: all that the cluster kernels leave (la_cluster.cu: short sequences of
// few heads; more than 296 tiles of 128 positions, 512 from eight tiles on, or more than sixteen tiles), whatever the context.
// Forward + backward, us, tcgen05 kernels (128x8x784, 60x8x300, 56x8x64: former ones of this file) / a warp per piece, in bursts of the same
// step: 128x8x784 282 / 156, 60x8x300 65 / 57, 16x8x3072 136 / 112, 32x8x3072 263 / 195, 8x8x16384 378 / 254, 64x8x2048 365 / 254, 1x8x4096
// 73 / 51, 1x1x16384 153 / 78, 2x1x65536 355 / 159, 1x8x65536 273 / 218, 16x8x700 48.5 / 46.3, 16x8x300 33.0 / 31.3, 20x8x256 40.6 / 32.8,
// 56x8x64 22.5 / 21.5; of 401 sizes, in captured graphs, four are slower by more than 1 % (B*H 444 N 64 16.1 / 17.2, N 128 24.9 / 25.4; five whole
// chunks of one wave of tcgen05 CTAs, B*H 128 N 640 37.3 / 39.9, 148 38.3 / 39.8).  Forward passes alone: causal_mma_leaves_forward().
bool of_warps(const la_problem& p) {
    if (p.dtype != LA_BF16 || p.D != 32 || p.M != 32 || p.N > (1 << 30)) return false;
    const int64_t tiles = (p.N + 127) / 128, ctas = tiles * p.B * p.H;
    return tiles > 16 || (ctas > 296 && (tiles < 8 || ctas > 512));
}

struct Plan { int pieces; int64_t len; };

// The estimates of choose_plan() for kernels that leave an SM little to gain from a second CTA, in units of one chunk of the main
// kernels (forward and backward together, 21.8 us in fp32 and 19.4 with Fourier features) of a CTA that has an SM to itself: their time
// with 1 to 5 CTAs per SM (uneven: with two on some, 149 to 221), for each of more, and for an odd one among those; a CTA's start
// and what each record costs it; the pre-pass's time per chunk, its start, and its time for each CTA per SM.  A CTA left over has its SM
// to itself, so that 3 and 5 are hardly less than 4 and 6.  Chosen over forced pieces of 8 to 352 sequences of 2 to 64 chunks: 0.5 % above
// the best number of pieces in the mean where the other rule is 5.3 % (fp32) and 10.6 % (Fourier) above it, and slower than that one in
// 7 of 460 and 9 of 350 cases, by 6 and 4 % at most.  us, forward + backward, at the pieces of the other rule / of this one (B x H x N:
// pieces): fp32 4x8x1416 8: 207 / 4: 198, 15x8x2354 2: 953 / 1: 824; Fourier 3x8x1999 11: 241 / 6: 188, 13x8x1271 5: 441 / 1: 402, 23x8x405
// 1: 316 / 2: 271.
struct WideCosts { double sms[5], uneven, more_sms, odd, start, record, sum, sum_start, sum_sms; };
constexpr WideCosts kFp32Costs = {{1.0, 1.86, 3.44, 3.8, 5.5}, 1.92, 0.94, 1.7, 0.34, 0.12, 0.18, 1.03, 0.58};
constexpr WideCosts kFourierCosts = {{1.0, 1.9, 3.33, 3.64, 5.0}, 2.39, 0.92, 0.92, 0.85, 0.2, 0.17, 1.22, 0.45};

double wide_cost(const WideCosts& w, int64_t bh, int64_t chunks, int64_t n) {
    const int64_t per = (chunks + n - 1) / n, cut = (chunks + per - 1) / per;        // cut: the pieces that this makes
    auto sms = [&](int64_t pieces) { return (bh * pieces + 147) / 148; };
    const int64_t m = sms(cut);
    double t = (double)per + w.start + w.record * (double)(cut - 1);
    t *= m == 2 && bh * cut < 222 ? w.uneven : m <= 5 ? w.sms[m - 1] : w.more_sms * (double)(m - m % 2) + w.odd * (double)(m % 2);
    if (cut > 1) t += w.sum * (double)per * (sms(cut - 1) == 1 ? 1.0 : w.sum_sms * (double)sms(cut - 1)) + w.sum_start;
    return t;
}

// What n pieces of a sequence cost a warp per piece, in us: warps in waves of as many as an SM holds, each a little slower the more of
// them share it; the records that a piece adds up; the kernels' starts.  (The first 64 positions go through the dQ sweep twice.)  Fitted to
// 2500 measured numbers of pieces for 450 sizes, B*H 150 to 900, N 192 to 4096: 7 % off in the mean.
double warp_wave(int64_t warps, double sixteens, int64_t most, double alone, double each) {
    const int64_t wave = 148 * most, rest = (warps % wave + 147) / 148;
    return sixteens * ((double)(warps / wave) * (alone + each * (double)most) + (rest ? alone + each * (double)rest : 0.0));
}
double warp_cost(int64_t bh, int64_t N, int64_t n, bool forward_alone) {
    const int64_t chunks = (N + T - 1) / T, per = (chunks + n - 1) / n;
    n = (chunks + per - 1) / per;
    const int64_t warps = bh * n;
    const double r = (double)(((per * T < N ? per * T : N) + 15) / 16), records = (double)(n - 1) * (double)warps / 148.0;
    double t = warp_wave(warps, r, 12, 0.44, 0.06) + 0.025 * records + 2.5;
    if (n > 1) t += warp_wave(bh * (n - 1), r, 16, 0.2, 0.035) + 1.2;
    if (forward_alone) return t;
    return t + warp_wave(warps, r + 0.5 * (r < 4.0 ? r : 4.0), 8, 0.74, 0.03) + warp_wave(warps, r, warps <= 8 * 148 ? 8 : 12, 0.25, 0.15) + 0.05 * records + 6.9;
}

// Pieces for a warp each, of a training step or of a forward pass that keeps no sums: eight warps on an SM, the most that the dQ sweep with
// both sums has registers for, and no more than a piece's start makes good (forward + backward, us, B x H x N: number of pieces: 16x8x3072
// 4: 131, 8: 106, 12: 115; 8x8x16384 8: 322, 16: 251, 24: 280; 1x8x16384 32: 106, 64: 88, 128: 113; 1x8x4096 16: 61, 32: 51, 64: 59; 2x1x65536
// 64: 190, 128: 154).  Beyond 148 sequences another number where the estimate above finds it faster by its own error (just past a full wave
// above all: 400x1x2048 3: 235, 8: 201; 444x1x512 3: 73, 4: 58; 592x1x784 3: 114, 2: 104; forward alone 400x1x2048 3: 71, 4: 59): 2 % off the
// best of the measured numbers in the mean, where the first rule alone is 4 % off (forward alone 2 and 6).  One piece: two chunks (500x1x100
// 1: 25.1, 2: 28.2), three of as many sequences as run one on a scheduler (530x1x192 1: 36.1, 3: 38.4; but 640x1x192 1: 46.1, 2: 44.2, and
// 180x1x192 1: 35.7, 3: 22.6), and more than 888 sequences (900x1x784 1: 155, 2: 181, 3: 164).
int64_t warp_pieces(int64_t bh, int64_t N, bool forward_alone) {
    const int64_t chunks = (N + T - 1) / T, most = (int64_t)(4.0 * sqrt((double)chunks));
    if (bh > 888 || chunks <= 2 || (chunks == 3 && bh >= 444 && bh <= 592)) return 1;
    int64_t best = bh > 592 ? 2 : bh > 394 ? 3 : 1184 / bh;
    if (best > most) best = most;
    if (best > chunks) best = chunks;
    if (bh <= 148) return best;
    double least = 0.93 * warp_cost(bh, N, best, forward_alone);
    for (int64_t n = 1; n <= 16 && n <= chunks && n * bh <= 4000; ++n) {        // (as far as it was measured)
        const double t = warp_cost(bh, N, n, forward_alone);
        if (t < least) { least = t; best = n; }
    }
    return best;
}

// Pieces per sequence, by the estimated time: fp32 D = M = 64 and Fourier features as above; the others in units of one chunk of a main
// kernel (about 10 us alone on an SM):
// an SM runs two CTAs in 1.25 times the time of one; a CTA's start costs about a chunk, and 0.2 for each record it sums, of
// which it has half of them on average; the pre-pass does 0.35 of a main kernel's work per chunk (fp32 D = M = 32, B4 H8 N2000,
// pieces 1 / 4 / 8 / 12 / 16: 353 / 141 / 113 / 131 / 119; B22 H8 N3316 903 / 732 / 749 / 733 / 757).  At most sixteen: the estimates
// are checked up to N = 4096 only (for few sequences much longer than that they would want more).
enum PlanFor { kStep, kForwardAlone, kNoRecords };        // a training step; a forward pass that keeps no sums; no room for records
Plan choose_plan(const la_problem& p, PlanFor what) {
    const int64_t chunks = (p.N + T - 1) / T, bh = p.B * p.H;
    int64_t best = 1;
    const int forced = tc::causal_pieces_override();
    const bool wide = p.dtype == LA_F32 ? p.D == 64 && p.M == 64 : p.phi == LA_PHI_IDENTITY && p.D == 128 && p.M == 64;
    if (what == kNoRecords) {
        best = 1;
    } else if (forced > 0) {
        best = forced < chunks ? forced : chunks;
        if (best > 1024) best = 1024;
    } else if (of_warps(p)) {
        best = warp_pieces(bh, p.N, what == kForwardAlone);
    } else if (!(wide && bh >= 222 && bh <= 296)) {          // (two CTAs on an SM as they are: one piece was the best of 112 measured sizes of 2 to 64 chunks)
        auto waves = [](int64_t ctas) {
            const int64_t sm = (ctas + 147) / 148;
            return 1.25 * (double)(sm / 2) + (double)(sm % 2);
        };
        auto cost = [&](int64_t n) {
            if (wide) return wide_cost(p.dtype == LA_F32 ? kFp32Costs : kFourierCosts, bh, chunks, n);
            const double per = (double)((chunks + n - 1) / n);
            return (per + 1.0 + 0.1 * (n - 1)) * waves(bh * n) + (n > 1 ? 0.35 * (per + 1.0) * waves(bh * (n - 1)) : 0.0);
        };
        for (int64_t n = 2; n <= 16 && n <= chunks; ++n)
            if (cost(n) < cost(best)) best = n;
    }
    const int64_t len = (chunks + best - 1) / best * T;
    return Plan{(int)((p.N + len - 1) / len), len};
}

// Records of a piece: where sequences are two pieces of 128 bf16 features, their sums are shared out over the SMs that would have none
// (Fourier B8 H8 N1000, pieces of eight chunks, three passes over the sums: 14, 14 and 27 us with 64 CTAs that load a chunk when they
// need it, 10, 10 and 15 with 128 that load it ahead; pieces of three chunks B8 H8 N300 fwd 19.5 / 18.7, of two N256 20.6 / 22.3).  Not where
// there are more pieces: each adds up all records before its own, and four for one took B1 H1 N4000 (16 pieces) from 179 to 382 us.
int record_parts(const la_problem& p, const Plan& pl) {
    if (p.dtype != LA_BF16 || p.phi != LA_PHI_IDENTITY || p.D != 128 || p.M != 64 || pl.pieces != 2 || pl.len < 3 * T) return 1;     // (see parts_of())
    const int64_t idle = 148 / (p.B * p.H);
    return (int)(idle < 1 ? 1 : idle < 4 ? idle : 4);
}
size_t record_bytes(const la_problem& p, const Plan& pl) {
    return (size_t)(p.B * p.H) * (size_t)(pl.pieces - 1) * (size_t)record_parts(p, pl) * (size_t)(p.D * p.M + p.D) * sizeof(float);
}
size_t aux_bytes(const la_problem& p) { return ((size_t)(p.B * p.H) * (size_t)p.N * 2 * sizeof(float) + 15) & ~(size_t)15; }

Params make_params(const la_problem& p, const Plan& pl, const int* lengths) {
    Params a = {};
    a.lengths = lengths;
    a.N = p.N; a.piece_len = pl.len; a.pieces = pl.pieces;
    // Small grids only, whose CTAs find SMs of their own beside those of the kernel before (fp32 B1 H2 N256 D32: 39 -> 25
    // us a step); otherwise CTAs that wait on the SMs with room leave the kernel unevenly spread (B32 H8 N4096 D64
    // backward 2007 -> 2862 us, released at the kernel's end B37 H8 N512 267 -> 328 us).
    a.chained = 2 * p.B * p.H * pl.pieces <= 148;
    a.parts = record_parts(p, pl);
    a.records = (pl.pieces - 1) * a.parts;
    a.heads = (int)p.H; a.D = (int)p.D; a.M = (int)p.M; a.phi = p.phi; a.eps = p.eps;
    return a;
}

template <typename C, int DP, int MP, bool EXACT> struct Kernels {
    static constexpr int THREADS = kThreads<C>;
    static int sums(const la_problem& p, const Params& a, bool reverse, cudaStream_t st) {
        if (a.pieces == 1) return LA_OK;
        const unsigned bh = (unsigned)(p.B * p.H), y = (unsigned)a.records;
        if (reverse)
            return launch<causal_mma_sum_kernel<C, DP, MP, EXACT, true>>(kProfMmaSum, THREADS, bh, y, SumLayout<C, DP, MP, true>::BYTES, a, st);
        return launch<causal_mma_sum_kernel<C, DP, MP, EXACT, false>>(kProfMmaSum, THREADS, bh, y, SumLayout<C, DP, MP, false>::BYTES, a, st);
    }
    static int forward(const la_problem& p, const Params& a, cudaStream_t st) {
        if (int rc = sums(p, a, false, st)) return rc;
        return launch<causal_mma_forward_kernel<C, DP, MP, EXACT>>(kProfMmaForward, THREADS, (unsigned)(p.B * p.H), (unsigned)a.pieces,
                      ForwardLayout<C, DP, MP>::BYTES, a, st);
    }
    static int backward(const la_problem& p, const Params& fwd, const Params& rev, cudaStream_t st) {
        const unsigned bh = (unsigned)(p.B * p.H), y = (unsigned)fwd.pieces;
        if (int rc = sums(p, fwd, false, st)) return rc;
        if (int rc = launch<causal_mma_dq_kernel<C, DP, MP, EXACT>>(kProfMmaDq, THREADS, bh, y, DqLayout<C, DP, MP>::BYTES, fwd, st)) return rc;
        if (int rc = sums(p, rev, true, st)) return rc;
        return launch<causal_mma_dkv_kernel<C, DP, MP, EXACT>>(kProfMmaDkv, THREADS, bh, y, DkvLayout<C, DP, MP>::BYTES, rev, st);
    }
};

struct WarpKernels {
    template <int PASS> static int run(const la_problem& p, ProfKernel prof, int pieces, const Params& a, cudaStream_t st) {
        if (p.phi == LA_PHI_IDENTITY) return launch<causal_warp_kernel<PASS, false>>(prof, 32, (unsigned)(p.B * p.H), (unsigned)pieces, 0, a, st);
        return launch<causal_warp_kernel<PASS, true>>(prof, 32, (unsigned)(p.B * p.H), (unsigned)pieces, 0, a, st);
    }
    static int forward(const la_problem& p, const Params& a, cudaStream_t st) {
        if (a.pieces > 1)
            if (int rc = run<kWarpSums>(p, kProfMmaSum, a.pieces - 1, a, st)) return rc;
        return run<kWarpForward>(p, kProfMmaForward, a.pieces, a, st);
    }
    // (with a stamp: the forward pass has left the sums)
    static int backward(const la_problem& p, const Params& fwd, const Params& rev, cudaStream_t st) {
        if (fwd.pieces > 1 && !fwd.stamp)
            if (int rc = run<kWarpSums>(p, kProfMmaSum, fwd.pieces - 1, fwd, st)) return rc;
        // The dQ sweep that can form both kinds of sums, eight warps on an SM with all registers they want, also where one kind is enough
        // (128x8x784 155.7 us a step, with the other 158; 256x8x500 210 / 213), unless twelve make one wave of what eight would make two
        // (160x8x512 159.8 / 151.6, 200x8x640 193.5 / 184.9).  Two pieces of one chunk, which only a forced plan makes, have a kernel for the
        // reverse sums (100x8x128 34.9 / 37.1 us a step; 50x8x128 28.1 / 25.0).
        const int64_t warps = p.B * p.H * fwd.pieces;
        if (fwd.pieces > 2 || (fwd.pieces == 2 && p.N > 128) || (fwd.pieces == 1 && (warps <= 8 * 148 || warps > 12 * 148))) {
            if (int rc = run<kWarpDqReverse>(p, kProfMmaDq, fwd.pieces, fwd, st)) return rc;
        } else {
            if (int rc = run<kWarpDq>(p, kProfMmaDq, fwd.pieces, fwd, st)) return rc;
            if (fwd.pieces > 1)
                if (int rc = run<kWarpReverseSums>(p, kProfMmaSum, fwd.pieces - 1, rev, st)) return rc;
        }
        return warps <= 8 * 148 ? run<kWarpDkvFew>(p, kProfMmaDkv, fwd.pieces, rev, st) : run<kWarpDkv>(p, kProfMmaDkv, fwd.pieces, rev, st);
    }
};

// Tiles are padded to 32, 64 or (D) 128 columns; EXACT: D and M are those sizes.  One warp per strip was measured, and is
// instantiated, at the exact sizes only; padded ones take two whatever the grid.
template <typename F> int dispatch(const la_problem& p, int pieces, F f) {
    const bool full = p.B * p.H * pieces >= 222;            // one and a half CTAs per SM and more
    const bool few = p.B * p.H * pieces <= 148;
    const bool exact = (p.D == 32 || p.D == 64 || p.D == 128) && p.M == (p.D == 32 ? 32 : 64);
    if (p.dtype == LA_F32) {
        if (p.D <= 32 && p.M <= 32) return exact ? f(Kernels<Fp32, 32, 32, true>()) : f(Kernels<Fp32, 32, 32, false>());
        if (exact && p.D == 64 && full) return f(Kernels<Fp32One, 64, 64, true>());
        if (exact && p.D == 64 && few) return f(Kernels<Fp32Alone, 64, 64, true>());
        if (p.D <= 64) return exact ? f(Kernels<Fp32, 64, 64, true>()) : f(Kernels<Fp32, 64, 64, false>());
        return f(Kernels<Fp32, 128, 64, false>());
    }
    if (of_warps(p)) return f(WarpKernels());
    if (p.phi == LA_PHI_IDENTITY) {
        if (p.D <= 64) return f(Kernels<Bf16Features, 64, 64, false>());
        if (exact && full) return f(Kernels<Bf16FeaturesOne, 128, 64, true>());
        if (exact && few) return f(Kernels<Bf16FeaturesAlone, 128, 64, true>());
        return exact ? f(Kernels<Bf16Features, 128, 64, true>()) : f(Kernels<Bf16Features, 128, 64, false>());
    }
    return p.D <= 64 ? f(Kernels<Bf16Wide, 64, 64, false>()) : f(Kernels<Bf16Wide, 128, 64, false>());
}

}  // namespace

bool causal_mma_supported(const la_problem& p) {
    static const bool disabled = getenv("LA_DISABLE_TC") != nullptr;
    return !disabled && p.M <= 64;
}

bool causal_mma_preferred(const la_problem& p) { return of_warps(p); }

// Of a warp per piece, which forward passes that keep no sums run on the tcgen05 kernels all the same: where one CTA of those per
// sequence is a wave of its own, well filled, the more of them the longer the sequences (their plan makes two pieces up to 74 sequences, and 149
// are two waves).  us, tcgen05 / a warp per piece, from a state in brackets, B*H x N: 90x512 8.2 / 9.8, 100x512 8.2 / 10.0 (9.5 / 10.8), 128x512 8.2 /
// 10.5 (9.5 / 11.3), 112x1024 12.9 / 14.9, 128x1024 13.1 / 15.2, 140x1280 15.4 / 18.7, 128x4096 42.0 / 45.3; at the edges 112x1500 0.98 of the
// time, 128x1500 1.00, 148x900 0.93, 100x1000 0.98, 90x784 0.96, 74x640 0.67, 150x512 0.74.  A training step is faster on warps.
bool causal_mma_leaves_forward(const la_problem& p) {
    if (!of_warps(p) || tc::causal_pieces_override() >= 0 || p.B * p.H * p.N >= (1LL << 31)) return false;        // (32-bit TMA coordinates)
    const int64_t bh = p.B * p.H, tiles = (p.N + 127) / 128, from = 56 + 6 * tiles;
    return bh <= 148 && bh > (from < 112 ? from : 112);
}

// The forward's workspace is optional for all problems of this file but those that a warp per piece took over from the tcgen05 kernels.
bool causal_mma_needs_workspace(const la_problem& p) { return of_warps(p) && (p.B * p.H < 3 * 148 || p.N > 1024); }

size_t causal_mma_workspace(const la_problem& p, bool backward) {
    const size_t rec = record_bytes(p, choose_plan(p, backward ? kStep : kForwardAlone));
    if (!backward && causal_mma_leaves_forward(p)) return tc::causal_forward_workspace(p);
    return backward ? aux_bytes(p) + (of_warps(p) ? 2 * rec : rec) : rec;
}
// the records of a forward pass, and the plan they were written under
size_t causal_mma_saved_bytes(const la_problem& p) {
    const size_t rec = of_warps(p) ? record_bytes(p, choose_plan(p, kStep)) : 0;
    return rec ? kStampBytes + rec : 0;
}

int causal_mma_forward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const float* S_in,
                       const float* Z_in, void* O, float* den, float* S_out, float* Z_out, void* saved, void* ws, size_t ws_bytes, cudaStream_t st) {
    if (saved && !causal_mma_saved_bytes(p)) saved = nullptr;
    Plan pl = choose_plan(p, saved ? kStep : kForwardAlone);
    if (saved) ws = (char*)saved + kStampBytes;
    else if (!ws || !aligned16(ws) || ws_bytes < record_bytes(p, pl)) pl = choose_plan(p, kNoRecords);        // one piece per sequence
    Params a = make_params(p, pl, lengths);
    a.Q = Q; a.K = K; a.V = V; a.O = O; a.den = den;
    a.S0 = S_in; a.Z0 = Z_in; a.S1 = S_out; a.Z1 = Z_out;
    a.rec = (float*)ws;
    a.stamp = (int*)saved;
    return dispatch(p, pl.pieces, [&](auto k) { return decltype(k)::forward(p, a, st); });
}

int causal_mma_backward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const void* G,
                        const StateArgs& sa, const void* saved, void* dQ, void* dK, void* dV, void* ws, cudaStream_t st) {
    const Plan pl = choose_plan(p, kStep);
    Params f = make_params(p, pl, lengths);
    f.Q = Q; f.K = K; f.V = V; f.G = G; f.dQ = dQ; f.dK = dK; f.dV = dV;
    f.aux = (float*)ws;
    f.rec = (float*)((char*)ws + aux_bytes(p));
    if (saved && causal_mma_saved_bytes(p)) {
        f.stamp = (int*)saved;
        f.status = device_status_ptr();
        if (!f.status) return fail(LA_ERR_CUDA, "device status word unavailable");
    }
    Params r = f;
    if (of_warps(p)) r.rec = f.rec_out = (float*)((char*)f.rec + record_bytes(p, pl));
    if (f.stamp) f.rec = (float*)((char*)saved + kStampBytes);
    f.S0 = sa.S_in; f.Z0 = sa.Z_in;
    r.first_record = 1;
    r.S0 = sa.dS_out; r.Z0 = sa.dZ_out; r.S1 = sa.dS_in; r.Z1 = sa.dZ_in;
    return dispatch(p, pl.pieces, [&](auto k) { return decltype(k)::backward(p, f, r, st); });
}

}  // namespace la
