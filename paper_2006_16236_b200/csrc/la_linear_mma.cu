// Non-causal form (Eq. 5-6) at fp32 accuracy on mma.sync (la_mma.cuh): fp32 problems and bf16 ones of shapes or feature maps
// that the tcgen05 kernels do not take; M <= 64, any D.
//
// Sums of k [V | 1]^T per split of a sequence (one record each, causal_mma_sum_kernel), then kernels that add a sequence's
// records up, hold the result [S | Z] as bf16 planes in shared memory and take it to every position:
//   forward  O = q S / (q . Z + eps)
//   dQ       h = G S^T, dn = q . Z + eps, dQ = (h - (q . h / dn) Z) / dn o phi'(Q); dn and -(q . h) / dn are parked
//   dK, dV   with R = sum of q / dn [G | dl]^T over the records of the same sums kernel: gk = V R^T + r, dV = k R
// A warp takes sixteen positions at a time from global memory into registers and their results back: no barrier after the
// state is there, so the warps of an SM overlap freely.  Bound: the products and conversions, then HBM.
#include <stdlib.h>

#include "la_mma_sweep.cuh"

namespace la {
namespace {

using namespace mma;
using namespace sweep;

constexpr int THREADS = 256;

template <typename C, int DP, int MP> struct ApplyLayout {      // state planes, vector, vector planes
    static constexpr int S = 0, Z = C::NS * DP * MP * 2, ZP = Z + DP * 4, BYTES = ZP + 3 * DP * 2;
};

// the sum of the sequence's records in registers and in shared memory
template <typename C, int DP, int MP>
__device__ __forceinline__ void load_state(State<DP, MP, THREADS / 32>& st, const Params& p, int64_t bh, uint8_t* smem) {
    using Sh = ApplyLayout<C, DP, MP>;
    st.init(p, nullptr, nullptr, p.rec + bh * p.records * (int64_t)(p.D * p.M + p.D), p.records);
    st.template publish<C::NS>(smem + Sh::S, reinterpret_cast<float*>(smem + Sh::Z), reinterpret_cast<uint16_t*>(smem + Sh::ZP));
    __syncthreads();
}

template <typename C, int DP, int MP, bool EXACT>
__global__ void __launch_bounds__(THREADS, 2)
linear_mma_forward_kernel(const Params p) {
    using IO = typename C::IO;
    using Sh = ApplyLayout<C, DP, MP>;
    constexpr int NQ = C::NQ, NS = C::NS;
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int D = EXACT ? DP : p.D, M = EXACT ? MP : p.M, phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    const uint32_t sS = smem_u32(smem + Sh::S);
    const uint16_t* sZp = reinterpret_cast<const uint16_t*>(smem + Sh::ZP);
    wait_for_stream();
    release_next();
    const Range r = range_of(p, blockIdx.y);
    const IO* Q = (const IO*)p.Q + r.bh * p.N * D;
    IO* O = (IO*)p.O + r.bh * p.N * M;
    float* den = p.den ? p.den + r.bh * p.N : nullptr;
    auto rows_at = [&](int64_t n0) { return (int)(r.end - n0 < 16 ? (r.end > n0 ? r.end - n0 : 0) : 16); };

    int64_t n0 = r.lo + 16 * warp;
    RawStrip<IO, DP> next;              // requested ahead of the records and of the strip before
    next.load(Q + n0 * D, 0, rows_at(n0), D, pad);
    {
        State<DP, MP, THREADS / 32> st;
        load_state<C>(st, p, r.bh, smem);
        if (r.piece == 0) st.write(p, p.S1 ? p.S1 + r.bh * D * M : nullptr, p.Z1 ? p.Z1 + r.bh * D : nullptr);
    }
    for (; n0 < r.end; n0 += 16 * (THREADS / 32)) {
        const int cn = rows_at(n0);
        uint32_t qa[DP / 16][NQ][4];
        {
            RawStrip<typename FeatureType<NQ>::type, DP> fq;
            next.template map<NQ>(phi, fq);
            fq.template planes<NQ>(qa);
        }
        const int64_t n1 = n0 + 16 * (THREADS / 32);
        next.load(Q + n1 * D, 0, rows_at(n1), D, pad);
        float d[2] = {0.f, 0.f};
#pragma unroll
        for (int kk = 0; kk < DP / 16; ++kk) {
            float u[4] = {0.f, 0.f, 0.f, 0.f};
            vector_mma<NQ, DP>(u, qa[kk], sZp, kk * 16, t);
            d[0] += u[0];
            d[1] += u[2];
        }
        const float inv[2] = {1.f / (d[0] + p.eps), 1.f / (d[1] + p.eps)};
#pragma unroll
        for (int n = 0; n < MP / 16; ++n) {
            Chain c;
#pragma unroll
            for (int kk = 0; kk < DP / 16; ++kk) {
                uint32_t b[NS][4];
                load_cols_t<NS, MP>(b, sS, DP * MP * 2, kk * 16, n * 2, lane);
                c.step<NQ, NS>(qa[kk], b);
            }
            float o[2][4];
            c.put(o[0], o[1]);
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (g + 8 * h < cn) {
                    IO* row = O + (n0 + g + 8 * h) * M + n * 16 + 2 * t;
                    if (n * 16 < M) store_pair<IO>(row, o[0][2 * h] * inv[h], o[0][2 * h + 1] * inv[h]);
                    if (n * 16 + 8 < M) store_pair<IO>(row + 8, o[1][2 * h] * inv[h], o[1][2 * h + 1] * inv[h]);
                }
        }
        if (den && t == 0) {
            if (g < cn) den[n0 + g] = d[0];
            if (g + 8 < cn) den[n0 + g + 8] = d[1];
        }
    }
    zero_rows<THREADS>(O, r.end, r.hi, M);
    if (den) zero_rows<THREADS>(den, r.end, r.hi, 1);
}

template <typename C, int DP, int MP, bool EXACT>
__global__ void __launch_bounds__(THREADS, 2)
linear_mma_dq_kernel(const Params p) {
    using IO = typename C::IO;
    using Sh = ApplyLayout<C, DP, MP>;
    constexpr int NQ = C::NQ, NV = C::NV, NS = C::NS;
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int D = EXACT ? DP : p.D, M = EXACT ? MP : p.M, phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    const uint32_t sS = smem_u32(smem + Sh::S);
    const float* sZ = reinterpret_cast<const float*>(smem + Sh::Z);
    wait_for_stream();
    release_next();
    const Range r = range_of(p, blockIdx.y);
    const IO* Q = (const IO*)p.Q + r.bh * p.N * D;
    const IO* G = (const IO*)p.G + r.bh * p.N * M;
    IO* dQ = (IO*)p.dQ + r.bh * p.N * D;
    float* dn_all = p.aux + r.bh * 2 * p.N;
    float* dl_all = dn_all + p.N;
    const int4 stamp = p.stamp ? *reinterpret_cast<const int4*>(p.stamp) : plan_stamp(p);        // (on its way beside the records)
    {
        State<DP, MP, THREADS / 32> st;
        load_state<C>(st, p, r.bh, smem);
    }
    if (other_plan(p, stamp)) return;
    for (int64_t n0 = r.lo + 16 * warp; n0 < r.end; n0 += 16 * (THREADS / 32)) {
        const int cn = (int)(r.end - n0 < 16 ? r.end - n0 : 16);
        RawStrip<IO, DP> rq;            // element j of block kk: result column tile 2 kk + j / 2, row g + 8 (j & 1)
        uint32_t ga[MP / 16][NV][4];
        {
            RawStrip<IO, MP> rg;
            rg.load(G + n0 * M, 0, cn, M, 0.f);
            rq.load(Q + n0 * D, 0, cn, D, pad);
            rg.template planes<NV>(ga);
        }
        float h[DP / 8][4];
#pragma unroll
        for (int n = 0; n < DP / 16; ++n) {
            Chain c;
#pragma unroll
            for (int ee = 0; ee < MP / 16; ++ee) {
                uint32_t b[NS][4];
                load_rows<NS, MP>(b, sS, DP * MP * 2, n * 16, ee * 2, lane);
                c.step<NV, NS>(ga[ee], b);
            }
            c.put(h[2 * n], h[2 * n + 1]);
        }
        RawStrip<typename FeatureType<NQ>::type, DP> fq;
        rq.template map<NQ>(phi, fq);
        float qz[2] = {0.f, 0.f}, qh[2] = {0.f, 0.f};
#pragma unroll
        for (int kk = 0; kk < DP / 16; ++kk)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int n = 2 * kk + (j >> 1), b = j & 1;
                const float2 z = *reinterpret_cast<const float2*>(sZ + n * 8 + 2 * t);
                qz[b] = fmaf(fq.r[kk][j].lo(), z.x, fmaf(fq.r[kk][j].hi(), z.y, qz[b]));
                qh[b] = fmaf(fq.r[kk][j].lo(), h[n][2 * b], fmaf(fq.r[kk][j].hi(), h[n][2 * b + 1], qh[b]));
            }
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int row = g + 8 * b;
            const float dn = quad_sum(qz[b]) + p.eps, inv = 1.f / dn;
            const float go = quad_sum(qh[b]) * inv;             // G_i . O_i
            if (row < cn) {
#pragma unroll
                for (int n = 0; n < DP / 8; ++n)
                    if (n * 8 < D) {
                        const float2 z = *reinterpret_cast<const float2*>(sZ + n * 8 + 2 * t);
                        const auto q = fq.r[n >> 1][(n & 1) * 2 + b];
                        store_pair<IO>(dQ + (n0 + row) * D + n * 8 + 2 * t,
                                       fmaf(-go, z.x, h[n][2 * b]) * inv * phi_slope_from_value(q.lo(), phi),
                                       fmaf(-go, z.y, h[n][2 * b + 1]) * inv * phi_slope_from_value(q.hi(), phi));
                    }
                if (t == 0) {
                    dn_all[n0 + row] = dn;
                    dl_all[n0 + row] = -go;
                }
            }
        }
    }
    zero_rows<THREADS>(dQ, r.end, r.hi, D);
}

template <typename C, int DP, int MP, bool EXACT>
__global__ void __launch_bounds__(THREADS, 2)
linear_mma_dkv_kernel(const Params p) {
    using IO = typename C::IO;
    using Sh = ApplyLayout<C, DP, MP>;
    constexpr int NQ = C::NQ, NV = C::NV, NS = C::NS;
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int D = EXACT ? DP : p.D, M = EXACT ? MP : p.M, phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    const uint32_t sR = smem_u32(smem + Sh::S);
    const float* sr = reinterpret_cast<const float*>(smem + Sh::Z);
    wait_for_stream();
    release_next();
    const Range r = range_of(p, blockIdx.y);
    const IO* K = (const IO*)p.K + r.bh * p.N * D;
    const IO* V = (const IO*)p.V + r.bh * p.N * M;
    IO* dK = (IO*)p.dK + r.bh * p.N * D;
    IO* dV = (IO*)p.dV + r.bh * p.N * M;
    const int4 stamp = p.stamp ? *reinterpret_cast<const int4*>(p.stamp) : plan_stamp(p);
    {
        State<DP, MP, THREADS / 32> st;
        load_state<C>(st, p, r.bh, smem);
    }
    if (other_plan(p, stamp)) return;
    for (int64_t n0 = r.lo + 16 * warp; n0 < r.end; n0 += 16 * (THREADS / 32)) {
        const int cn = (int)(r.end - n0 < 16 ? r.end - n0 : 16);
        RawStrip<typename FeatureType<NQ>::type, DP> fk;
        RawStrip<IO, MP> rv;
        {
            RawStrip<IO, DP> rk;
            rk.load(K + n0 * D, 0, cn, D, pad);
            rv.load(V + n0 * M, 0, cn, M, 0.f);
            rk.template map<NQ>(phi, fk);
        }
        {
            uint32_t ka[DP / 16][NQ][4];
            fk.template planes<NQ>(ka);
#pragma unroll
            for (int n = 0; n < MP / 16; ++n) {
                Chain c;
#pragma unroll
                for (int kk = 0; kk < DP / 16; ++kk) {
                    uint32_t b[NS][4];
                    load_cols_t<NS, MP>(b, sR, DP * MP * 2, kk * 16, n * 2, lane);
                    c.step<NQ, NS>(ka[kk], b);
                }
                float o[2][4];
                c.put(o[0], o[1]);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (g + 8 * h < cn) {
                        IO* row = dV + (n0 + g + 8 * h) * M + n * 16 + 2 * t;
                        if (n * 16 < M) store_pair<IO>(row, o[0][2 * h], o[0][2 * h + 1]);
                        if (n * 16 + 8 < M) store_pair<IO>(row + 8, o[1][2 * h], o[1][2 * h + 1]);
                    }
            }
        }
        uint32_t va[MP / 16][NV][4];
        rv.template planes<NV>(va);
#pragma unroll
        for (int n = 0; n < DP / 16; ++n) {
            Chain c;
#pragma unroll
            for (int ee = 0; ee < MP / 16; ++ee) {
                uint32_t b[NS][4];
                load_rows<NS, MP>(b, sR, DP * MP * 2, n * 16, ee * 2, lane);
                c.step<NV, NS>(va[ee], b);
            }
            float o[2][4];
            c.put(o[0], o[1]);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float2 z = *reinterpret_cast<const float2*>(sr + n * 16 + i * 8 + 2 * t);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (g + 8 * h < cn && n * 16 + i * 8 < D) {
                        const auto k = fk.r[n][i * 2 + h];
                        store_pair<IO>(dK + (n0 + g + 8 * h) * D + n * 16 + i * 8 + 2 * t,
                                       (o[i][2 * h] + z.x) * phi_slope_from_value(k.lo(), phi),
                                       (o[i][2 * h + 1] + z.y) * phi_slope_from_value(k.hi(), phi));
                    }
            }
        }
    }
    zero_rows<THREADS>(dK, r.end, r.hi, D);
    zero_rows<THREADS>(dV, r.end, r.hi, M);
}

// ---- host ------------------------------------------------------------------------------------------------------
struct Plan { int splits; int64_t len; };

// fp32, D = M = 64, forward + backward in us, splits 2 / 4 / 5 / 8 / 16: B8 H8 N4096 487 / 376 / 513 / 401 / 474;
// B1 H8 N1000 119 / 70 / - / 48 / 48 (the shared-memory kernels before: 993 and 116).
Plan choose_plan(const la_problem& p) {
    const int64_t chunks = (p.N + T - 1) / T, bh = p.B * p.H;
    int64_t want = bh < 2 * 148 ? 2 * 148 / bh : 1;     // two CTAs per SM at most
    const int forced = tc::linear_splits_override();
    if (forced > 0) want = forced;
    const int64_t most = (chunks + 1) / 2;              // at least two chunks (a strip per warp of the apply kernels)
    if (want > most) want = most;
    if (want > 64) want = 64;
    const int64_t len = (chunks + want - 1) / want * T;
    return Plan{(int)((p.N + len - 1) / len), len};
}

size_t record_bytes(const la_problem& p) {
    return (size_t)(p.B * p.H) * (size_t)choose_plan(p).splits * (size_t)(p.D * p.M + p.D) * sizeof(float);
}

template <typename C, int DP, int MP, bool EXACT> struct Kernels {
    template <bool REVERSE> static int sums(const la_problem& p, const Params& a, cudaStream_t st) {
        return launch<causal_mma_sum_kernel<C, DP, MP, EXACT, REVERSE>>(kProfMmaSum, kThreads<C>, (unsigned)(p.B * p.H), (unsigned)a.pieces,
                                                                        SumLayout<C, DP, MP, REVERSE>::BYTES, a, st);
    }
    template <auto KERNEL> static int apply(const la_problem& p, const Params& a, cudaStream_t st) {
        return launch<KERNEL>(kProfMmaApply, THREADS, (unsigned)(p.B * p.H), (unsigned)a.pieces, ApplyLayout<C, DP, MP>::BYTES, a, st);
    }
    static int forward(const la_problem& p, const Params& a, cudaStream_t st) {
        if (int rc = sums<false>(p, a, st)) return rc;
        return apply<linear_mma_forward_kernel<C, DP, MP, EXACT>>(p, a, st);
    }
    static int backward(const la_problem& p, const Params& fwd, const Params& rev, bool have_sums, cudaStream_t st) {
        if (!have_sums)
            if (int rc = sums<false>(p, fwd, st)) return rc;
        if (int rc = apply<linear_mma_dq_kernel<C, DP, MP, EXACT>>(p, fwd, st)) return rc;
        if (int rc = sums<true>(p, rev, st)) return rc;
        return apply<linear_mma_dkv_kernel<C, DP, MP, EXACT>>(p, rev, st);
    }
};

// Tiles are padded to 32, 64 or (D) 128 columns; EXACT: D and M are those sizes.
template <typename F> int dispatch(const la_problem& p, F f) {
    const bool exact = (p.D == 32 || p.D == 64) && p.M == p.D;
    if (p.dtype == LA_F32) {
        if (p.D <= 32 && p.M <= 32) return exact ? f(Kernels<Fp32, 32, 32, true>()) : f(Kernels<Fp32, 32, 32, false>());
        if (p.D <= 64) return exact ? f(Kernels<Fp32, 64, 64, true>()) : f(Kernels<Fp32, 64, 64, false>());
        return f(Kernels<Fp32, 128, 64, false>());
    }
    if (p.phi == LA_PHI_IDENTITY) return p.D <= 64 ? f(Kernels<Bf16Features, 64, 64, false>()) : f(Kernels<Bf16Features, 128, 64, false>());
    return p.D <= 64 ? f(Kernels<Bf16Wide, 64, 64, false>()) : f(Kernels<Bf16Wide, 128, 64, false>());
}

Params make_params(const la_problem& p, const int* lengths) {
    const Plan pl = choose_plan(p);
    Params a = {};
    a.lengths = lengths;
    a.N = p.N; a.piece_len = pl.len; a.pieces = pl.splits; a.records = pl.splits; a.parts = 1;
    a.chained = 2 * p.B * p.H * pl.splits <= 148;       // (small grids only, as in la_causal_mma.cu)
    a.heads = (int)p.H; a.D = (int)p.D; a.M = (int)p.M; a.phi = p.phi; a.eps = p.eps;
    return a;
}

}  // namespace

bool linear_mma_supported(const la_problem& p) {
    static const bool disabled = getenv("LA_DISABLE_TC") != nullptr;
    return !disabled && p.M <= 64;
}

size_t linear_mma_workspace(const la_problem& p, bool backward) {
    if (!backward) return kStampBytes + record_bytes(p);
    return 2 * record_bytes(p) + (((size_t)(p.B * p.H) * (size_t)p.N * 2 * sizeof(float) + 15) & ~(size_t)15);
}

int linear_mma_forward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, void* O, float* den,
                       float* KV, float* Zs, void* saved, void* ws, cudaStream_t st) {
    Params a = make_params(p, lengths);
    a.Q = Q; a.K = K; a.V = V; a.O = O; a.den = den; a.S1 = KV; a.Z1 = Zs;
    a.stamp = saved ? (int*)saved : (int*)ws;            // kept for the backward pass if asked
    a.rec = (float*)((char*)a.stamp + kStampBytes);
    return dispatch(p, [&](auto k) { return decltype(k)::forward(p, a, st); });
}

int linear_mma_backward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const void* saved,
                        const void* G, void* dQ, void* dK, void* dV, void* ws, cudaStream_t st) {
    Params f = make_params(p, lengths);
    f.Q = Q; f.K = K; f.V = V; f.G = G; f.dQ = dQ; f.dK = dK; f.dV = dV;
    if (saved) {
        f.stamp = (int*)saved;
        f.status = device_status_ptr();
        if (!f.status) return fail(LA_ERR_CUDA, "device status word unavailable");
    }
    Params r = f;
    f.rec = saved ? (float*)((char*)saved + kStampBytes) : (float*)ws;
    r.rec = (float*)((char*)ws + record_bytes(p));
    f.aux = r.aux = (float*)((char*)ws + 2 * record_bytes(p));
    return dispatch(p, [&](auto k) { return decltype(k)::backward(p, f, r, saved != nullptr, st); });
}

}  // namespace la
