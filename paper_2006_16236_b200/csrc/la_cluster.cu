// Short sequences in one launch: a thread-block cluster per (batch, head), a CTA per 64 or 128 positions, for problems whose
// time is latency (a prompt, one utterance, a model being tried out).
//
// The other kernels cut a sequence into pieces too, but hand the state from piece to piece through memory: one kernel sums
// the pieces, the next one starts from the sums, and either costs a launch, a first load and a drain of its own.  Here the
// CTAs of a cluster keep their tiles in shared memory, form their own sums, and give each other the sums of the CTAs before
// them (after them, of all of them) through distributed shared memory:
//   CTA c of R owns a part of the state's rows.  Every CTA sends its sums of those rows to CTA c, which adds them up in order
//   and sends each running sum, as the operand planes that the products take, to the CTA that starts from it.
// Every number crosses the cluster twice, whatever R is, between two cluster barriers; what does not need the other CTAs
// (the products inside the diagonal block) runs between the barrier's arrival and its completion.  The backward pass keeps its
// tiles for both sweeps: one launch that reads every input once, in place of four.
//
// The products are those of la_causal_mma.cu (planes and accuracy by configuration) and, for bf16 encoders, those of
// la_tc_linear.cu with the summed state in two planes in place of a centred one.
//
// What bounds them: the chain load, sums, exchange, products, each one to three thousand cycles of dependent work that runs
// once (causal forward bf16 D = 64, 16 CTAs: 1900 sums, 3900 send and diagonal block, 4200 exchange, 1500 barrier, 2500 result);
// not bandwidth, and the tensor pipe is nearly idle.  16 rows and a
// warp per strip (two warps where planes are three) and one tile per CTA keep that chain short; which problems: at the end.
#include <stdlib.h>

#include "la_mma_sweep.cuh"

namespace la {
namespace {

using namespace mma;
using namespace sweep;

constexpr int kMaxCluster = 16;

#ifdef LA_TC_TRACE
__device__ long long g_trace_cluster[32 * 16];
#define LA_TRACE_CLUSTER(slot) do { if (threadIdx.x == 0 && blockIdx.y == 0) g_trace_cluster[blockIdx.x * 32 + (slot)] = clock64(); } while (0)
#else
#define LA_TRACE_CLUSTER(slot) do { } while (0)
#endif

// ---- cluster barrier and distributed shared memory ---------------------------------------------------------------
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ int cluster_rank() { uint32_t r; asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return (int)r; }
__device__ __forceinline__ int cluster_size() { uint32_t r; asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return (int)r; }
__device__ __forceinline__ uint32_t address_in(uint32_t addr, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void peer_store(uint32_t a, float x, float y) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t a, float x) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(x) : "memory"); }
__device__ __forceinline__ void peer_store(uint32_t a, uint32_t x, uint32_t y) {
    asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t a, uint32_t x) { asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(a), "r"(x) : "memory"); }

// ---- sums over the cluster -------------------------------------------------------------------------------------
// CTA c owns rows c * rows .. of the state's matrix [DP][MP] and of its vector, and has an inbox with a slot [rows][MP | 1] for
// each CTA.  The CTAs send their sums straight from registers into the owners' inboxes; the owner reads its own shared memory
// and sends what it adds up to the CTAs that need it.  Nobody waits for a load from another SM: reading the other CTAs'
// records instead took 2700 to 5400 cycles an exchange, this way 2100 to 4200 (sixteen CTAs, D = 64).
template <int DP, int MP> struct Inbox {
    static constexpr int FLOATS = (DP + kMaxCluster) * (MP + 1) + 4 * kMaxCluster;      // at most R * slot()
    uint32_t at;
    int R, me, rows;
    __device__ __forceinline__ explicit Inbox(uint32_t at) : at(at), R(cluster_size()), me(cluster_rank()), rows((DP + R - 1) / R) {}
    __device__ __forceinline__ int slot() const { return (rows * (MP + 1) + 3) & ~3; }
    // this CTA's sums to their owners
    template <int WARPS> __device__ __forceinline__ void send(const State<DP, MP, WARPS>& st) const {
        using St = State<DP, MP, WARPS>;
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
        if (!St::owner()) return;
#pragma unroll
        for (int i = 0; i < St::SD; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int d = St::strip(i) * 16 + g + 8 * h, owner = d / rows, row = d - owner * rows;
                const uint32_t slot_at = address_in(at + me * slot() * 4, owner), to = slot_at + (row * MP + St::n0() * 8 + 2 * t) * 4;
#pragma unroll
                for (int n = 0; n < St::NC; ++n) peer_store(to + n * 32, st.s[i][n][2 * h], st.s[i][n][2 * h + 1]);
                if (t == 0 && St::n0() == 0) peer_store(slot_at + (rows * MP + row) * 4, st.z[i][h]);
            }
    }
    // f(d, e, x): numbers (d, e) .. (d, e + 3) of CTA c's matrix are at x + c * slot(), for the rows that this CTA owns;
    // v(d, c, x): number d of the vectors likewise, a thread for every c
    template <int THREADS, typename F, typename G> __device__ __forceinline__ void for_own_rows(const float* inbox, F f, G v) const {
        const int d0 = me * rows, own = min(rows, DP - d0);
#pragma unroll 1
        for (int i = threadIdx.x; i < own * (MP / 4); i += THREADS) f(d0 + i / (MP / 4), i % (MP / 4) * 4, inbox + i * 4);
        for (int i = THREADS - 1 - (int)threadIdx.x; i < own * R; i += THREADS) v(d0 + i / R, i % R, inbox + rows * MP + i / R);
    }
};

// Four numbers, in packed pairs (an addition of two is one instruction)
struct Four {
    sm100::f32x2 a, b;
    __device__ __forceinline__ Four() : a(0), b(0) {}
    __device__ __forceinline__ Four(const float* p) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        a = sm100::pair(v.x, v.y);
        b = sm100::pair(v.z, v.w);
    }
    __device__ __forceinline__ Four operator+(const Four& y) const {
        Four r;
        r.a = sm100::add2(a, y.a);
        r.b = sm100::add2(b, y.b);
        return r;
    }
    __device__ __forceinline__ float4 get() const {
        float4 v;
        sm100::unpair(a, v.x, v.y);
        sm100::unpair(b, v.z, v.w);
        return v;
    }
};

// Four numbers of a state's matrix as operand planes, for CTA c.
template <int NS, int DP, int MP>
__device__ __forceinline__ void give_planes(uint32_t tile, const float4& v, int c) {
    uint32_t o0[NS], o1[NS];
    split2<NS>(v.x, v.y, o0);
    split2<NS>(v.z, v.w, o1);
    const uint32_t to = address_in(tile, c);
#pragma unroll
    for (int k = 0; k < NS; ++k) peer_store(to + k * (DP * MP * 2), o0[k], o1[k]);
}

// Where a CTA has its inbox and receives the sum that it starts from: planes of the matrix, the vector in fp32 and in three
// planes.
struct Exchange { uint8_t* inbox; uint32_t tile, vec, vpl; };
enum Order { kBefore, kAfter };

// To every CTA the sum of what the CTAs before it (after it) have sent.  S0, Z0: what the first CTA in the order starts from
// (each or null); S1, Z1: where the sum over all of them goes (each or null).  Between two cluster barriers.
template <Order ORDER, int NS, int DP, int MP, int THREADS>
__device__ __forceinline__ void running_sums(const Exchange& x, const float* S0, const float* Z0, float* S1, float* Z1) {
    const Inbox<DP, MP> in(smem_u32(x.inbox));
    const int R = in.R, slot = in.slot();
    in.template for_own_rows<THREADS>(reinterpret_cast<const float*>(x.inbox), [&](int d, int e, const float* from) {
        // (the given state, often much larger than the sums, is added to each of them and not a term that they start with: one
        // rounding of its size instead of sixteen)
        Four run, s0;
        if (S0) s0 = Four(S0 + d * MP + e);
        const uint32_t tile = x.tile + tile_at<MP>(d, e / 8) + e % 8 * 2;
#pragma unroll 4
        for (int i = 0; i < R; ++i) {
            const int c = ORDER == kBefore ? i : R - 1 - i;
            const Four v(from + c * slot);
            give_planes<NS, DP, MP>(tile, (run + s0).get(), c);
            run = run + v;
        }
        if (S1) *reinterpret_cast<float4*>(S1 + d * MP + e) = (run + s0).get();
    }, [&](int d, int c, const float* from) {
        const int before = ORDER == kBefore ? c : R - 1 - c;           // CTAs ahead of c
        const float z0 = Z0 ? Z0[d] : 0.f;
        float run = 0.f;
#pragma unroll 4
        for (int i = 0; i < before; ++i) run += from[(ORDER == kBefore ? i : R - 1 - i) * slot];
        uint32_t o[3];
        split2<3>(run + z0, 0.f, o);
        peer_store(address_in(x.vec + d * 4, c), run + z0);
#pragma unroll
        for (int k = 0; k < 3; ++k) asm volatile("st.shared::cluster.b16 [%0], %1;" ::"r"(address_in(x.vpl + (k * DP + d) * 2, c)), "h"((uint16_t)o[k]) : "memory");
        if (Z1 && before == R - 1) Z1[d] = (run + from[c * slot]) + z0;
    });
}

// ---- tiles -----------------------------------------------------------------------------------------------------
// T rows of COLS columns on their way to shared memory: bf16 straight into the operand tile, fp32 row by row into `raw`, which
// convert() turns into planes.  Rows cn .. T - 1 become zeros.
__device__ __forceinline__ void copy16(uint32_t dst, const void* src, bool there) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(there ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copies_done() {
    asm volatile("cp.async.wait_all;" ::: "memory");
}
// (thread id of THREADS)
template <int T, int COLS, int THREADS, typename IO>
__device__ __forceinline__ void request_rows(int id, uint8_t* tile, uint8_t* raw, const IO* src, int cn) {
    constexpr int GROUPS = COLS / 8;            // of eight numbers
#pragma unroll
    for (int u = 0; u < T * GROUPS / THREADS; ++u) {
        const int i = id + u * THREADS, row = i / GROUPS;
        const IO* from = src + (row < cn ? i * 8 : 0);
        if constexpr (sizeof(IO) == 2) {
            copy16(smem_u32(tile) + tile_at<COLS>(row, i % GROUPS), from, row < cn);
        } else {
            copy16(smem_u32(raw) + i * 32, from, row < cn);
            copy16(smem_u32(raw) + i * 32 + 16, from + 4, row < cn);
        }
    }
}
// what the same thread has requested, once copies_done() -> NP planes of f(x); rows cn .. T - 1 stay zeros
template <int NP, int T, int COLS, int THREADS, typename F>
__device__ __forceinline__ void convert_rows(int id, uint8_t* tile, const uint8_t* raw, int cn, F f) {
    constexpr int GROUPS = COLS / 8;
#pragma unroll 1
    for (int i = id; i < T * GROUPS; i += THREADS) {
        const int row = i / GROUPS;
        Group8<float> r;
        float x[8];
        r.load(reinterpret_cast<const float*>(raw) + i * 8);
        r.get(x);
        uint32_t o[NP][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t p[NP];
            split2<NP>(f(x[2 * j]), f(x[2 * j + 1]), p);
#pragma unroll
            for (int k = 0; k < NP; ++k) o[k][j] = row < cn ? p[k] : 0u;
        }
#pragma unroll
        for (int k = 0; k < NP; ++k)
            *reinterpret_cast<uint4*>(tile + k * (T * COLS * 2) + tile_at<COLS>(row, i % GROUPS)) = make_uint4(o[k][0], o[k][1], o[k][2], o[k][3]);
    }
}
// the same in place for bf16, f taking a pair to a pair
template <int T, int COLS, int THREADS, typename F>
__device__ __forceinline__ void map_rows(int id, uint8_t* tile, int cn, F f) {
    constexpr int GROUPS = COLS / 8;
#pragma unroll
    for (int i = id; i < T * GROUPS; i += THREADS) {
        uint4* x = reinterpret_cast<uint4*>(tile + tile_at<COLS>(i / GROUPS, i % GROUPS));
        uint4 v = *x;
        v.x = f(v.x); v.y = f(v.y); v.z = f(v.z); v.w = f(v.w);
        *x = i / GROUPS < cn ? v : make_uint4(0u, 0u, 0u, 0u);
    }
}
// the planes of a feature-mapped tile, and of a tile of values
template <typename C, int T, int COLS, int THREADS>
__device__ __forceinline__ void feature_planes(int id, uint8_t* tile, const uint8_t* raw, int cn, int phi) {
    if constexpr (sizeof(typename C::IO) == 4) {
        with_phi<C::NQ>(phi, [&](auto f) { convert_rows<C::NQ, T, COLS, THREADS>(id, tile, raw, cn, f); });
    } else {
        static_assert(C::NQ == 1, "from bf16 to bf16");
        if (C::MAPPED && phi != LA_PHI_IDENTITY) map_rows<T, COLS, THREADS>(id, tile, cn, [](uint32_t w) { return tc::phi_pair(w); });
    }
}
template <typename C, int T, int COLS, int THREADS>
__device__ __forceinline__ void value_planes(int id, uint8_t* tile, const uint8_t* raw, int cn) {
    if constexpr (sizeof(typename C::IO) == 4) convert_rows<C::NV, T, COLS, THREADS>(id, tile, raw, cn, [](float x) { return x; });
}

struct ClusterParams : Params {
    // What a forward pass leaves in the saved buffer of the tcgen05 kernels (or null): the features, and the stamp.
    void *keep_q, *keep_k;
    int stamp_value[tc::kPlanStampInts];
    // Behind a kernel of the same call that has waited for everything before it and whose results this one does not read: it
    // starts beside that kernel and waits for its end at its own.
    int late;
};
__device__ __forceinline__ void wait_first(const ClusterParams& p) { if (!p.late) wait_for_stream(); }
__device__ __forceinline__ void wait_last(const ClusterParams& p) { if (p.late) wait_for_stream(); }

// positions [n0, n0 + cn) real, [n0 + cn, n0 + hi) padding, of this CTA
struct Rows { int64_t bh, n0; int cn, hi; };
template <int T>
__device__ __forceinline__ Rows rows_of(const Params& p) {
    Rows r;
    r.bh = blockIdx.y;
    r.n0 = (int64_t)blockIdx.x * T;
    int64_t len = p.N;
    if (p.lengths) len = min((int64_t)max(p.lengths[r.bh / p.heads], 0), p.N);
    r.cn = (int)min(max(len - r.n0, (int64_t)0), (int64_t)T);
    r.hi = (int)min(p.N - r.n0, (int64_t)T);
    return r;
}

// Warps: a strip of sixteen rows each, or (WPS = 2) two to a strip with half of the result's columns each.  The strips are
// dealt out so that the warps of a scheduler (four apart) have blocks that add up to about the same number.
template <int STRIPS> __device__ __forceinline__ int strip_of_warp(int warp) {
    const int s = warp % STRIPS;
    if (STRIPS > 4) return s < 4 ? s : STRIPS + 3 - s;
    return warp >= 4 ? STRIPS - 1 - s : s;
}

// zero the scores of a diagonal block: columns right of the row (UPPER: left of it)
template <bool UPPER>
__device__ __forceinline__ void mask_diagonal_block(float (&s0)[4], float (&s1)[4], int g, int t) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int row = g + (j >> 1) * 8, col = 2 * t + (j & 1);
        if (UPPER ? col < row : col > row) s0[j] = 0.f;
        if (UPPER ? col + 8 < row : col + 8 > row) s1[j] = 0.f;
    }
}

// The strip's own rows as A operand: in registers where they have one plane, else read block by block.
template <int NP, int T, int C> struct StripOperand {
    uint32_t tile;
    int row0, lane;
    __device__ __forceinline__ StripOperand(uint32_t tile, int row0, int lane) : tile(tile), row0(row0), lane(lane) {}
    __device__ __forceinline__ const uint32_t (&block(int kk, uint32_t (&f)[NP][4]) const)[NP][4] {
        load_cols<NP, C>(f, tile, T * C * 2, row0, kk * 2, lane);
        return f;
    }
};
template <int T, int C> struct StripOperand<1, T, C> {
    uint32_t a[C / 16][1][4];
    __device__ __forceinline__ StripOperand(uint32_t tile, int row0, int lane) {
#pragma unroll
        for (int kk = 0; kk < C / 16; ++kk) load_cols<1, C>(a[kk], tile, 0, row0, kk * 2, lane);
    }
    __device__ __forceinline__ const uint32_t (&block(int kk, uint32_t (&)[1][4]) const)[1][4] { return a[kk]; }
};

// ---- causal forward --------------------------------------------------------------------------------------------
// B1 H8 N2048 D64 bf16 continued from a state 22.1 -> 11.9 us, N1000 19.7 -> 9 (the call's host work is 7.7).
template <typename C, int DP, int MP, int STRIPS> struct ForwardShared {
    static constexpr int T = 16 * STRIPS, K = 0, Q = K + C::NQ * T * DP * 2, V = Q + C::NQ * T * DP * 2, S = V + C::NV * T * MP * 2,
                         VEC = S + C::NS * DP * MP * 2, VPL = VEC + DP * 4, IN = VPL + 3 * DP * 2, END = IN + Inbox<DP, MP>::FLOATS * 4;
    // fp32 inputs lie where the states will be until they are planes
    static constexpr int RAW = S, RAW_K = RAW, RAW_Q = RAW_K + T * DP * 4, RAW_V = RAW_Q + T * DP * 4, RAW_END = sizeof(typename C::IO) == 4 ? RAW_V + T * MP * 4 : 0,
                         BYTES = END > RAW_END ? END : RAW_END;
};

template <typename C, int DP, int MP, int STRIPS, int WPS>
__global__ void __launch_bounds__(32 * STRIPS * WPS, STRIPS * WPS <= 8 ? 2 : 1)
causal_cluster_forward_kernel(const ClusterParams p) {
    using IO = typename C::IO;
    using Sh = ForwardShared<C, DP, MP, STRIPS>;
    constexpr int NQ = C::NQ, NV = C::NV, NP = C::NP, NS = C::NS, T = 16 * STRIPS, WARPS = STRIPS * WPS, THREADS = 32 * WARPS;
    constexpr int NT = MP / 16 / WPS;       // sixteen-column blocks of the result that a warp has
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const uint32_t sK = smem_u32(smem + Sh::K), sV = smem_u32(smem + Sh::V), sS = smem_u32(smem + Sh::S);
    const uint16_t* sZp = reinterpret_cast<const uint16_t*>(smem + Sh::VPL);
    const Exchange ex = {smem + Sh::IN, sS, smem_u32(smem + Sh::VEC), smem_u32(smem + Sh::VPL)};
    LA_TRACE_CLUSTER(0);
    wait_first(p);
    release_next();
    const Rows r = rows_of<T>(p);
    const int64_t base = r.bh * p.N + r.n0;
    const int strip = strip_of_warp<STRIPS>(warp), row0 = strip * 16, nb0 = warp / STRIPS * NT;
    const int id = threadIdx.x;
    request_rows<T, DP, THREADS>(id, smem + Sh::K, smem + Sh::RAW_K, (const IO*)p.K + base * DP, r.cn);
    request_rows<T, MP, THREADS>(id, smem + Sh::V, smem + Sh::RAW_V, (const IO*)p.V + base * MP, r.cn);
    request_rows<T, DP, THREADS>(id, smem + Sh::Q, smem + Sh::RAW_Q, (const IO*)p.Q + base * DP, r.cn);
    copies_done();
    feature_planes<C, T, DP, THREADS>(id, smem + Sh::K, smem + Sh::RAW_K, r.cn, phi);
    value_planes<C, T, MP, THREADS>(id, smem + Sh::V, smem + Sh::RAW_V, r.cn);
    feature_planes<C, T, DP, THREADS>(id, smem + Sh::Q, smem + Sh::RAW_Q, r.cn, phi);
    __syncwarp();
    cluster_arrive();
    __syncthreads();
    if constexpr (NQ == 1 && C::MAPPED) {
        if (p.stamp && blockIdx.x == 0 && blockIdx.y == 0 && id < tc::kPlanStampInts) p.stamp[id] = p.stamp_value[id];
        if (p.keep_q)
            for (int i = id; i < r.hi * (DP / 8); i += THREADS) {
                const uint32_t at = tile_at<DP>(i / (DP / 8), i % (DP / 8));
                reinterpret_cast<uint4*>((IO*)p.keep_q + base * DP)[i] = *reinterpret_cast<const uint4*>(smem + Sh::Q + at);
                reinterpret_cast<uint4*>((IO*)p.keep_k + base * DP)[i] = *reinterpret_cast<const uint4*>(smem + Sh::K + at);
            }
    }
    const StripOperand<NQ, T, DP> q(smem_u32(smem + Sh::Q), row0, lane);
    LA_TRACE_CLUSTER(1);
    {
        State<DP, MP, WARPS> st;
        st.init(p, nullptr, nullptr, nullptr, 0);
        st.template update<NQ, NV, true, T>(sK, sV, nullptr);
        __syncwarp();
        cluster_wait();         // every CTA is there, and has no more inputs where its inbox is
        Inbox<DP, MP>(smem_u32(ex.inbox)).send(st);
    }
    __syncwarp();
    LA_TRACE_CLUSTER(2);
    cluster_arrive();
    float o[2 * NT][4], d0 = 0.f, d1 = 0.f;         // rows g, g + 8 of [num | den]; d0, d1 spread over the four lanes
    clear(o);
    if (row0 < r.cn) {
#pragma unroll 1
        for (int jb = 0; jb <= strip; ++jb) {
            float s0[4], s1[4];
            {
                Chain c;
#pragma unroll
                for (int kk = 0; kk < DP / 16; ++kk) {
                    uint32_t b[NQ][4];
                    load_rows<NQ, DP>(b, sK, T * DP * 2, jb * 16, kk * 2, lane);
                    uint32_t a[NQ][4];
                    c.template step<NQ, NQ>(q.block(kk, a), b);
                }
                c.put(s0, s1);
            }
            if (jb == strip) mask_diagonal_block<false>(s0, s1, g, t);
            uint32_t pa[NP][4];
            operand_of<NP>(pa, s0, s1);
            if constexpr (NP == 1) {            // numerator and normaliser see the same rounded scores
                float u[4] = {0.f, 0.f, 0.f, 0.f};
                mma16816(u, pa[0], 0x3f803f80u, 0x3f803f80u);
                d0 += t == 0 ? u[0] : 0.f;
                d1 += t == 0 ? u[2] : 0.f;
            } else {
                d0 += (s0[0] + s0[1]) + (s1[0] + s1[1]);
                d1 += (s0[2] + s0[3]) + (s1[2] + s1[3]);
            }
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                uint32_t b[NV][4];
                load_cols_t<NV, MP>(b, sV, T * MP * 2, jb * 16, (nb0 + n) * 2, lane);
                block_mma<NP, NV>(o[2 * n], o[2 * n + 1], pa, b);
            }
        }
    }
    __syncwarp();
    LA_TRACE_CLUSTER(3);
    cluster_wait();
    LA_TRACE_CLUSTER(4);
    running_sums<kBefore, NS, DP, MP, THREADS>(ex, p.S0 ? p.S0 + r.bh * DP * MP : nullptr, p.Z0 ? p.Z0 + r.bh * DP : nullptr,
                                               p.S1 ? p.S1 + r.bh * DP * MP : nullptr, p.Z1 ? p.Z1 + r.bh * DP : nullptr);
    __syncwarp();
    LA_TRACE_CLUSTER(5);
    cluster_arrive();
    cluster_wait();
    LA_TRACE_CLUSTER(6);
    if (row0 < r.cn) {
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            Chain c;
#pragma unroll
            for (int kk = 0; kk < DP / 16; ++kk) {
                uint32_t b[NS][4];
                load_cols_t<NS, MP>(b, sS, DP * MP * 2, kk * 16, (nb0 + n) * 2, lane);
                uint32_t a[NQ][4];
                c.template step<NQ, NS>(q.block(kk, a), b);
            }
            c.add_to(o[2 * n], o[2 * n + 1]);
        }
#pragma unroll
        for (int kk = 0; kk < DP / 16; ++kk) {
            float u[4] = {0.f, 0.f, 0.f, 0.f};
            uint32_t a[NQ][4];
            vector_mma<NQ, DP>(u, q.block(kk, a), sZp, kk * 16, t);
            d0 += t == 0 ? u[0] : 0.f;
            d1 += t == 0 ? u[2] : 0.f;
        }
        d0 = quad_sum(d0);
        d1 = quad_sum(d1);
        IO* O = (IO*)p.O + base * MP;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = row0 + g + 8 * h;
            const float inv = 1.f / ((h ? d1 : d0) + p.eps);
            if (row < r.cn) {
#pragma unroll
                for (int n = 0; n < 2 * NT; ++n) store_pair<IO>(O + row * MP + nb0 * 16 + n * 8 + 2 * t, o[n][2 * h] * inv, o[n][2 * h + 1] * inv);
                if (p.den && t == 0 && nb0 == 0) p.den[base + row] = h ? d1 : d0;
            }
        }
    }
    LA_TRACE_CLUSTER(7);
    if (r.cn < r.hi) {
        zero_rows<THREADS>((IO*)p.O + base * MP, r.cn, r.hi, MP);
        if (p.den) zero_rows<THREADS>(p.den + base, r.cn, r.hi, 1);
    }
    wait_last(p);
}

// ---- causal backward -------------------------------------------------------------------------------------------
// Both sweeps of la_causal_mma.cu over the tiles that the CTA keeps: dQ from the state S before it, then dK and dV from the
// state R after it, with q^ = q / dn and dl = -G . O in between.  Two warps per strip: dQ, one [G S^T | L k] and one the
// scores' part; dK and dV, one each.
struct BackwardParams : ClusterParams {
    const float *R0, *r0;       // gradient of the final state, each or null
    float *R1, *r1;             // gradient of the initial state, each or null
};

template <typename C, int DP, int MP, int STRIPS> struct BackwardShared {
    static constexpr int T = 16 * STRIPS, K = 0, V = K + C::NQ * T * DP * 2, G = V + C::NV * T * MP * 2, Q = G + C::NV * T * MP * 2,
                         S = Q + C::NR * T * DP * 2, VEC = S + C::NS * DP * MP * 2, VPL = VEC + DP * 4, DL = VPL + 3 * DP * 2, DLP = DL + T * 4,
                         GO = DLP + 3 * T * 2, PART = GO + T * 4, IN = PART + T * DP * 4, END = IN + Inbox<DP, MP>::FLOATS * 4;
    static constexpr int RAW_K = S, RAW_V = RAW_K + T * DP * 4, RAW_G = RAW_V + T * MP * 4, RAW_END = sizeof(typename C::IO) == 4 ? RAW_G + T * MP * 4 : 0,
                         BYTES = END > RAW_END ? END : RAW_END;
};

// (a barrier for each direction: a warp that arrives at one and goes on to wait at the same one would complete it by itself)
__device__ __forceinline__ void pair_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pair_arrive(int id) {
    __threadfence_block();
    asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory");
}

template <typename C, int DP, int MP, int STRIPS>
__global__ void __launch_bounds__(64 * STRIPS, (227 * 1024 / (BackwardShared<C, DP, MP, STRIPS>::BYTES + 1024) >= 2 ? 2 : 1))
causal_cluster_backward_kernel(const BackwardParams p) {
    using IO = typename C::IO;
    using Sh = BackwardShared<C, DP, MP, STRIPS>;
    constexpr int NQ = C::NQ, NV = C::NV, NP = C::NP, NS = C::NS, NR = C::NR, T = 16 * STRIPS, WARPS = 2 * STRIPS, THREADS = 32 * WARPS;
    static_assert(2 * STRIPS < 16, "named barriers");
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    const uint32_t sK = smem_u32(smem + Sh::K), sV = smem_u32(smem + Sh::V), sG = smem_u32(smem + Sh::G), sQ = smem_u32(smem + Sh::Q),
                   sS = smem_u32(smem + Sh::S);
    const float* sZ = reinterpret_cast<const float*>(smem + Sh::VEC);
    float *sdl = reinterpret_cast<float*>(smem + Sh::DL), *sgo = reinterpret_cast<float*>(smem + Sh::GO);
    uint16_t* sdlp = reinterpret_cast<uint16_t*>(smem + Sh::DLP);
    const Exchange ex = {smem + Sh::IN, sS, smem_u32(smem + Sh::VEC), smem_u32(smem + Sh::VPL)};
    LA_TRACE_CLUSTER(0);
    wait_for_stream();
    release_next();
    const Rows r = rows_of<T>(p);
    const int64_t base = r.bh * p.N + r.n0;
    const bool first = warp < STRIPS;           // of the strip's two warps
    const int strip = strip_of_warp<STRIPS>(warp), row0 = strip * 16, to_first = 1 + strip, to_second = 1 + STRIPS + strip;
    const bool real = row0 < r.cn;
    const IO *Q = (const IO*)p.Q + base * DP, *K = (const IO*)p.K + base * DP;
    RawStrip<IO, DP> rq;                        // element j of block kk: result column tile 2 kk + j / 2, row g + 8 (j & 1)
    const int id = threadIdx.x;
    request_rows<T, DP, THREADS>(id, smem + Sh::K, smem + Sh::RAW_K, K, r.cn);
    request_rows<T, MP, THREADS>(id, smem + Sh::V, smem + Sh::RAW_V, (const IO*)p.V + base * MP, r.cn);
    request_rows<T, MP, THREADS>(id, smem + Sh::G, smem + Sh::RAW_G, (const IO*)p.G + base * MP, r.cn);
    if (first) rq.load(Q, row0, r.cn, DP, pad);
    copies_done();
    feature_planes<C, T, DP, THREADS>(id, smem + Sh::K, smem + Sh::RAW_K, r.cn, phi);
    value_planes<C, T, MP, THREADS>(id, smem + Sh::V, smem + Sh::RAW_V, r.cn);
    value_planes<C, T, MP, THREADS>(id, smem + Sh::G, smem + Sh::RAW_G, r.cn);
    __syncwarp();
    cluster_arrive();
    __syncthreads();
    LA_TRACE_CLUSTER(1);
    State<DP, MP, WARPS> st;
    st.init(p, nullptr, nullptr, nullptr, 0);
    st.template update<NQ, NV, true, T>(sK, sV, nullptr);
    __syncwarp();
    cluster_wait();             // every CTA is there, and has no more inputs where its inbox is
    Inbox<DP, MP>(smem_u32(ex.inbox)).send(st);
    __syncwarp();
    LA_TRACE_CLUSTER(2);
    cluster_arrive();

    // ---- dQ
    // The first chunk of a sequence goes through twice, the second time with the G_i . O_i it found taken off the scores and
    // off the given state's part: where few terms make up a row, h and (q . h / dn) Zc cancel almost entirely.
    const bool twice = r.n0 == 0, state_before = r.n0 > 0 || p.S0 || p.Z0;
    float c0 = 0.f, c1 = 0.f;                   // G_i . O_i of rows g, g + 8, as far as it is known
    float h[DP / 8][4], zc[DP / 8][4];
    auto scores = [&] {                         // h = ((G V^T - c) o L) k
        clear(h);
#pragma unroll 1
        for (int jb = 0; jb <= strip; ++jb) {
            float s0[4], s1[4];
            {
                Chain c;
#pragma unroll
                for (int ee = 0; ee < MP / 16; ++ee) {
                    uint32_t a[NV][4], b[NV][4];
                    load_cols<NV, MP>(a, sG, T * MP * 2, row0, ee * 2, lane);
                    load_rows<NV, MP>(b, sV, T * MP * 2, jb * 16, ee * 2, lane);
                    c.template step<NV, NV>(a, b);
                }
                c.put(s0, s1);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                s0[j] -= c0; s1[j] -= c0;
                s0[2 + j] -= c1; s1[2 + j] -= c1;
            }
            if (jb == strip) mask_diagonal_block<false>(s0, s1, g, t);
            uint32_t pa[NP][4];
            operand_of<NP>(pa, s0, s1);
#pragma unroll
            for (int n = 0; n < DP / 16; ++n) {
                uint32_t b[NQ][4];
                load_cols_t<NQ, DP>(b, sK, T * DP * 2, jb * 16, n * 2, lane);
                block_mma<NP, NQ>(h[2 * n], h[2 * n + 1], pa, b);
            }
        }
    };
    auto state_product = [&] {                  // h = G S^T
#pragma unroll
        for (int n = 0; n < DP / 16; ++n) {
            Chain c;
#pragma unroll
            for (int ee = 0; ee < MP / 16; ++ee) {
                uint32_t a[NV][4], b[NS][4];
                load_cols<NV, MP>(a, sG, T * MP * 2, row0, ee * 2, lane);
                load_rows<NS, MP>(b, sS, DP * MP * 2, n * 16, ee * 2, lane);
                c.template step<NV, NS>(a, b);
            }
            c.put(h[2 * n], h[2 * n + 1]);
        }
    };
    float4* part = reinterpret_cast<float4*>(smem + Sh::PART) + strip * (DP / 8) * 32 + lane;
    auto give_scores = [&] {
#pragma unroll
        for (int n = 0; n < DP / 8; ++n) part[n * 32] = make_float4(h[n][0], h[n][1], h[n][2], h[n][3]);
        pair_arrive(to_first);
    };
    auto take_scores = [&] {
        pair_sync(to_first);
#pragma unroll
        for (int n = 0; n < DP / 8; ++n) {
            const float4 v = part[n * 32];
            h[n][0] += v.x; h[n][1] += v.y; h[n][2] += v.z; h[n][3] += v.w;
        }
    };
    RawStrip<typename FeatureType<NQ>::type, DP> fq;
    float inv[2];
    auto row_sums = [&] {                       // dn and what is left of G_i . O_i
        float qz[2] = {0.f, 0.f}, qh[2] = {0.f, 0.f}, go[2];
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
            inv[b] = 1.f / (quad_sum(qz[b]) + p.eps);
            go[b] = (quad_sum(qh[b]) - (b ? c1 : c0) * p.eps) * inv[b];
        }
        c0 += go[0];
        c1 += go[1];
        return make_float2(go[0], go[1]);
    };
    clear(zc);
    if (real && first) {
        rq.template map<NQ, false>(phi, fq);
#pragma unroll 1
        for (int jb = 0; jb <= strip; ++jb) {                   // zc = L k
            uint32_t ones[1][4] = {{0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u}};
            if (jb == strip) {
                ones[0][0] = ones[0][3] = (2 * t <= g ? 0x3f80u : 0u) | (2 * t + 1 <= g ? 0x3f800000u : 0u);
                ones[0][2] = 0u;
            }
#pragma unroll
            for (int n = 0; n < DP / 16; ++n) {
                uint32_t b[NQ][4];
                load_cols_t<NQ, DP>(b, sK, T * DP * 2, jb * 16, n * 2, lane);
                block_mma<1, NQ>(zc[2 * n], zc[2 * n + 1], ones, b);
            }
        }
    }
    // (one loop around everything, and the exchange inside it: each product is in the code once, and what does not need the
    // state before this CTA is done ahead of it)
    float2 go = make_float2(0.f, 0.f);
    bool exchanged = false;
#pragma unroll 1
    for (int pass = twice ? 0 : 1; pass < 2; ++pass) {
        if (real && !first) scores();
        if (!exchanged && (pass == 1 || state_before)) {
            exchanged = true;
            __syncwarp();
            LA_TRACE_CLUSTER(3);
            cluster_wait();
            LA_TRACE_CLUSTER(4);
            running_sums<kBefore, NS, DP, MP, THREADS>(ex, p.S0 ? p.S0 + r.bh * DP * MP : nullptr, p.Z0 ? p.Z0 + r.bh * DP : nullptr, nullptr, nullptr);
            __syncwarp();
            LA_TRACE_CLUSTER(5);
            cluster_arrive();
            cluster_wait();
            LA_TRACE_CLUSTER(6);
            if (first && state_before)
#pragma unroll
                for (int n = 0; n < DP / 8; ++n) {
                    const float2 z = load_pair(sZ + n * 8 + 2 * t);
                    zc[n][0] += z.x; zc[n][2] += z.x;
                    zc[n][1] += z.y; zc[n][3] += z.y;
                }
        }
        if (!real) continue;
        if (first) {
            clear(h);
            if (state_before) {
                state_product();
#pragma unroll
                for (int n = 0; n < DP / 8; ++n) {              // (c0 and c1 are zero but for the second time)
                    const float2 z = load_pair(sZ + n * 8 + 2 * t);
                    h[n][0] = fmaf(-c0, z.x, h[n][0]); h[n][1] = fmaf(-c0, z.y, h[n][1]);
                    h[n][2] = fmaf(-c1, z.x, h[n][2]); h[n][3] = fmaf(-c1, z.y, h[n][3]);
                }
            }
            take_scores();
            go = row_sums();
            if (pass == 0) {
                if (t == 0) {
                    sgo[row0 + g] = c0;
                    sgo[row0 + g + 8] = c1;
                }
                __syncwarp();
                pair_arrive(to_second);
            }
        } else {
            give_scores();
            if (pass == 0) {
                pair_sync(to_second);
                c0 = sgo[row0 + g];
                c1 = sgo[row0 + g + 8];
            }
        }
    }
    if (real && first) {
        IO* dQ = (IO*)p.dQ + base * DP;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int row = row0 + g + 8 * b;
            if (row < r.cn) {
#pragma unroll
                for (int n = 0; n < DP / 8; ++n) {
                    const auto q = fq.r[n >> 1][(n & 1) * 2 + b];
                    const float gb = b ? go.y : go.x;
                    store_pair<IO>(dQ + row * DP + n * 8 + 2 * t, fmaf(-gb, zc[n][2 * b], h[n][2 * b]) * inv[b] * phi_slope_from_value(q.lo(), phi),
                                   fmaf(-gb, zc[n][2 * b + 1], h[n][2 * b + 1]) * inv[b] * phi_slope_from_value(q.hi(), phi));
                }
            }
        }
    }
    if (first) {                                // q^ and dl; zeros where there is no position
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int row = row0 + g + 8 * b;
            const bool there = row < r.cn;
#pragma unroll
            for (int n = 0; n < DP / 8; ++n) {
                uint32_t o[NR];
                float x = 0.f, y = 0.f;
                if (there) {
                    const auto q = fq.r[n >> 1][(n & 1) * 2 + b];
                    x = q.lo() * inv[b];
                    y = q.hi() * inv[b];
                }
                split2<NR>(x, y, o);
#pragma unroll
                for (int k = 0; k < NR; ++k) *reinterpret_cast<uint32_t*>(smem + Sh::Q + k * (T * DP * 2) + tile_at<DP>(row, n) + t * 4) = o[k];
            }
            if (t == 0) {
                const float dl = there ? -(b ? c1 : c0) : 0.f;
                sdl[row] = dl;
                uint32_t o[3];
                split2<3>(dl, 0.f, o);
#pragma unroll
                for (int k = 0; k < 3; ++k) sdlp[k * T + row] = (uint16_t)o[k];
            }
        }
    }
    __syncthreads();
    LA_TRACE_CLUSTER(7);

    // ---- dK, dV
    st.init(p, nullptr, nullptr, nullptr, 0);
    st.template update<NR, NV, false, T>(sQ, sG, sdlp);
    Inbox<DP, MP>(smem_u32(ex.inbox)).send(st);
    __syncwarp();
    LA_TRACE_CLUSTER(8);
    cluster_arrive();
    const int blocks = (r.cn + 15) / 16;
    constexpr int NT = (DP > MP ? DP : MP) / 8;
    float acc[NT][4];                           // dV of the strip's first warp, dK of its second
    clear(acc);
    if (real && first) {
#pragma unroll 1
        for (int ib = strip; ib < blocks; ++ib) {               // (q^ k^T o L)^T G
            float s0[4], s1[4];
            {
                Chain c;
#pragma unroll
                for (int kk = 0; kk < DP / 16; ++kk) {
                    uint32_t a[NQ][4], b[NR][4];
                    load_cols<NQ, DP>(a, sK, T * DP * 2, row0, kk * 2, lane);
                    load_rows<NR, DP>(b, sQ, T * DP * 2, ib * 16, kk * 2, lane);
                    c.template step<NQ, NR>(a, b);
                }
                c.put(s0, s1);
            }
            if (ib == strip) mask_diagonal_block<true>(s0, s1, g, t);
            uint32_t pa[NP][4];
            operand_of<NP>(pa, s0, s1);
#pragma unroll
            for (int n = 0; n < MP / 16; ++n) {
                uint32_t b[NV][4];
                load_cols_t<NV, MP>(b, sG, T * MP * 2, ib * 16, n * 2, lane);
                block_mma<NP, NV>(acc[2 * n], acc[2 * n + 1], pa, b);
            }
        }
    }
    RawStrip<IO, DP> rk;
    if (real && !first) {
        rk.load(K, row0, r.cn, DP, pad);        // (for the slope, at the end)
#pragma unroll 1
        for (int ib = strip; ib < blocks; ++ib) {               // ((G V^T + dl) o L)^T q^
            const float2 w0 = *reinterpret_cast<const float2*>(sdl + ib * 16 + 2 * t);
            const float2 w1 = *reinterpret_cast<const float2*>(sdl + ib * 16 + 8 + 2 * t);
            float s0[4] = {w0.x, w0.y, w0.x, w0.y}, s1[4] = {w1.x, w1.y, w1.x, w1.y};
            {
                Chain c;
#pragma unroll
                for (int ee = 0; ee < MP / 16; ++ee) {
                    uint32_t a[NV][4], b[NV][4];
                    load_cols<NV, MP>(a, sV, T * MP * 2, row0, ee * 2, lane);
                    load_rows<NV, MP>(b, sG, T * MP * 2, ib * 16, ee * 2, lane);
                    c.template step<NV, NV>(a, b);
                }
                c.add_to(s0, s1);
            }
            if (ib == strip) mask_diagonal_block<true>(s0, s1, g, t);
            uint32_t pa[NP][4];
            operand_of<NP>(pa, s0, s1);
#pragma unroll
            for (int n = 0; n < DP / 16; ++n) {
                uint32_t b[NR][4];
                load_cols_t<NR, DP>(b, sQ, T * DP * 2, ib * 16, n * 2, lane);
                block_mma<NP, NR>(acc[2 * n], acc[2 * n + 1], pa, b);
            }
        }
    }
    __syncwarp();
    LA_TRACE_CLUSTER(9);
    cluster_wait();
    running_sums<kAfter, NS, DP, MP, THREADS>(ex, p.R0 ? p.R0 + r.bh * DP * MP : nullptr, p.r0 ? p.r0 + r.bh * DP : nullptr,
                                              p.R1 ? p.R1 + r.bh * DP * MP : nullptr, p.r1 ? p.r1 + r.bh * DP : nullptr);
    __syncwarp();
    LA_TRACE_CLUSTER(10);
    cluster_arrive();
    cluster_wait();
    LA_TRACE_CLUSTER(11);
    if (real && first) {
#pragma unroll
        for (int n = 0; n < MP / 16; ++n) {                     // k R
            Chain c;
#pragma unroll
            for (int kk = 0; kk < DP / 16; ++kk) {
                uint32_t a[NQ][4], b[NS][4];
                load_cols<NQ, DP>(a, sK, T * DP * 2, row0, kk * 2, lane);
                load_cols_t<NS, MP>(b, sS, DP * MP * 2, kk * 16, n * 2, lane);
                c.template step<NQ, NS>(a, b);
            }
            c.add_to(acc[2 * n], acc[2 * n + 1]);
        }
        IO* dV = (IO*)p.dV + base * MP;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int row = row0 + g + 8 * b;
            if (row < r.cn)
#pragma unroll
                for (int n = 0; n < MP / 8; ++n) store_pair<IO>(dV + row * MP + n * 8 + 2 * t, acc[n][2 * b], acc[n][2 * b + 1]);
        }
    }
    if (real && !first) {
#pragma unroll
        for (int n = 0; n < DP / 16; ++n) {                     // V R^T + r (which often cancel), then the scores' part
            const float2 z0 = load_pair(sZ + n * 16 + 2 * t), z1 = load_pair(sZ + n * 16 + 8 + 2 * t);
            float s0[4] = {z0.x, z0.y, z0.x, z0.y}, s1[4] = {z1.x, z1.y, z1.x, z1.y};
            Chain c;
#pragma unroll
            for (int ee = 0; ee < MP / 16; ++ee) {
                uint32_t a[NV][4], b[NS][4];
                load_cols<NV, MP>(a, sV, T * MP * 2, row0, ee * 2, lane);
                load_rows<NS, MP>(b, sS, DP * MP * 2, n * 16, ee * 2, lane);
                c.template step<NV, NS>(a, b);
            }
            c.add_to(s0, s1);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                acc[2 * n][j] += s0[j];
                acc[2 * n + 1][j] += s1[j];
            }
        }
        RawStrip<typename FeatureType<NQ>::type, DP> fk;
        rk.template map<NQ, false>(phi, fk);        // (as the tile has them)
        IO* dK = (IO*)p.dK + base * DP;
#pragma unroll
        for (int n = 0; n < DP / 8; ++n) {
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int row = row0 + g + 8 * b;
                const auto k = fk.r[n >> 1][(n & 1) * 2 + b];
                if (row < r.cn)
                    store_pair<IO>(dK + row * DP + n * 8 + 2 * t, acc[n][2 * b] * phi_slope_from_value(k.lo(), phi),
                                   acc[n][2 * b + 1] * phi_slope_from_value(k.hi(), phi));
            }
        }
    }
    LA_TRACE_CLUSTER(12);
    if (r.cn < r.hi) {
        zero_rows<THREADS>((IO*)p.dQ + base * DP, r.cn, r.hi, DP);
        zero_rows<THREADS>((IO*)p.dK + base * DP, r.cn, r.hi, DP);
        zero_rows<THREADS>((IO*)p.dV + base * MP, r.cn, r.hi, MP);
    }
}

// ---- non-causal forward, bf16 ----------------------------------------------------------------------------------
// As in la_tc_linear.cu the operands are x' = phi(x) - 1 and the parts of rank one stay in fp32:
//   S = 1 ysum^T + A', A' = sum k' V^T, Z = N 1 + a';  num = (q . 1) ysum + 1 A' + q' A',  den = N (q . 1) + 1 . a' + q' . a'
// The operand A' of the last product has two planes (16 bits; la_tc_linear.cu rounds a centred one to 8), all else 32 bits.
// A CTA takes `piece_len` positions, T at a time.
template <int DP, int STRIPS> struct LinearShared {          // (the second stage of K | V at the end: not there where one tile is all)
    static constexpr int T = 16 * STRIPS, NS = 3, K = 0, V = K + T * DP * 2, Q = V + T * DP * 2, S = Q + T * DP * 2,
                         A = S + NS * DP * DP * 2, Y = A + DP * 4, M = Y + DP * 4, IN = M + DP * 4, IN2 = IN + Inbox<DP, DP>::FLOATS * 4,
                         STAGE = (IN2 + (DP + kMaxCluster) * 4 + 127) / 128 * 128, BYTES = STAGE + 2 * T * DP * 2;
};

struct Centred {        // x' of a pair
    bool elu;
    __device__ __forceinline__ explicit Centred(int phi) : elu(phi != LA_PHI_IDENTITY) {}
    __device__ __forceinline__ uint32_t operator()(uint32_t w) const {
        const float x = __uint_as_float(w << 16), y = __uint_as_float(w & 0xffff0000u);
        if (!elu) return pack_rn(x - 1.f, y - 1.f);
        float e, f;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x * 1.4426950408889634f));
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(y * 1.4426950408889634f));
        return pack_rn(x > 0.f ? x : e - 1.f, y > 0.f ? y : f - 1.f);
    }
};

template <int DP, int STRIPS>
__global__ void __launch_bounds__(32 * STRIPS, 2)
linear_cluster_forward_kernel(const ClusterParams p) {
    using IO = __nv_bfloat16;
    using Sh = LinearShared<DP, STRIPS>;
    constexpr int NS = Sh::NS, T = 16 * STRIPS, WARPS = STRIPS, THREADS = 32 * WARPS;
    using St = State<DP, DP, WARPS>;
    extern __shared__ __align__(128) uint8_t smem[];
    const int id = threadIdx.x, lane = id & 31, warp = id >> 5, g = lane >> 2, t = lane & 3;
    const uint32_t sS = smem_u32(smem + Sh::S);
    const Centred f(p.phi);
    LA_TRACE_CLUSTER(0);
    wait_first(p);
    release_next();
    const int64_t bh = blockIdx.y, lo = (int64_t)blockIdx.x * p.piece_len, hi = min(lo + p.piece_len, p.N);
    int64_t len = p.N;
    if (p.lengths) len = min((int64_t)max(p.lengths[bh / p.heads], 0), p.N);
    const int64_t end = max(min(hi, len), lo);
    const IO *Q = (const IO*)p.Q + bh * p.N * DP, *K = (const IO*)p.K + bh * p.N * DP, *V = (const IO*)p.V + bh * p.N * DP;
    auto real_rows = [&](int64_t n0, int most) { return (int)min(max(end - n0, (int64_t)0), (int64_t)most); };

    int64_t s0 = lo + 16 * warp;            // the warp's rows of Q: sixteen at a time, the first with the first tiles
    uint8_t* strip = smem + Sh::Q + warp * 16 * DP * 2;
    auto request = [&](int64_t n0, int stage) {
        request_rows<T, DP, THREADS>(id, smem + stage * Sh::STAGE + Sh::K, nullptr, K + n0 * DP, real_rows(n0, T));
        request_rows<T, DP, THREADS>(id, smem + stage * Sh::STAGE + Sh::V, nullptr, V + n0 * DP, real_rows(n0, T));
    };
    request(lo, 0);
    request_rows<16, DP, 32>(lane, strip, nullptr, Q + s0 * DP, real_rows(s0, 16));
    __syncwarp();
    cluster_arrive();
    const Inbox<DP, DP> in(smem_u32(smem + Sh::IN));
    const uint32_t in2 = smem_u32(smem + Sh::IN2);
    {
        St st;
        st.init(p, nullptr, nullptr, nullptr, 0);
        float y[St::NC][4];                 // column sums of V in the warps of the first strip
        clear(y);
        int stage = 0;
#pragma unroll 1
        for (int64_t n0 = lo; n0 < end; n0 += T, stage ^= 1) {
            const uint32_t sK = smem_u32(smem + stage * Sh::STAGE + Sh::K), sV = smem_u32(smem + stage * Sh::STAGE + Sh::V);
            copies_done();
            map_rows<T, DP, THREADS>(id, smem + stage * Sh::STAGE + Sh::K, real_rows(n0, T), f);
            __syncthreads();
            if (n0 + T < end) request(n0 + T, stage ^ 1);
            LA_TRACE_CLUSTER(1);
            st.template update<1, 1, true, T>(sK, sV, nullptr);
            if (St::owner() && St::strip(0) == 0) {
                const uint32_t ones[4] = {0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u};
#pragma unroll 1
                for (int b = 0; b < T / 16; b += 4) {
                    float u[St::NC][4];
                    clear(u);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int n = 0; n < St::NC / 2; ++n) {
                            uint32_t v[1][4];
                            load_cols_t<1, DP>(v, sV, 0, (b + i) * 16, St::n0() + n * 2, lane);
                            mma16816(u[2 * n], ones, v[0][0], v[0][1]);
                            mma16816(u[2 * n + 1], ones, v[0][2], v[0][3]);
                        }
#pragma unroll
                    for (int n = 0; n < St::NC; ++n) { y[n][0] += u[n][0]; y[n][1] += u[n][1]; }
                }
            }
        }
        __syncwarp();
        cluster_wait();                     // every CTA is there
        in.send(st);
        if (St::owner() && St::strip(0) == 0 && g == 0)         // ysum
#pragma unroll
            for (int n = 0; n < St::NC; ++n)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int col = (St::n0() + n) * 8 + 2 * t + j, owner = col / in.rows;
                    peer_store(address_in(in2 + (in.me * in.rows + col - owner * in.rows) * 4, owner), y[n][j]);
                }
    }
    __syncwarp();
    LA_TRACE_CLUSTER(2);
    cluster_arrive();
    // x' of the strip as A operand, and q . 1
    uint32_t qa[DP / 16][1][4];
    float x1[2];
    auto take_rows = [&] {
        copies_done();
        map_rows<16, DP, 32>(lane, strip, 16, f);
        __syncwarp();
        x1[0] = x1[1] = 0.f;
#pragma unroll
        for (int kk = 0; kk < DP / 16; ++kk) {
            load_cols<1, DP>(qa[kk], smem_u32(strip), 0, 0, kk * 2, lane);
#pragma unroll
            for (int j = 0; j < 4; ++j) x1[j & 1] += __uint_as_float(qa[kk][0][j] << 16) + __uint_as_float(qa[kk][0][j] & 0xffff0000u);
        }
        __syncwarp();
        if (s0 + T < end) request_rows<16, DP, 32>(lane, strip, nullptr, Q + (s0 + T) * DP, real_rows(s0 + T, 16));
        x1[0] = (float)DP + quad_sum(x1[0]);
        x1[1] = (float)DP + quad_sum(x1[1]);
    };
    take_rows();
    LA_TRACE_CLUSTER(3);
    cluster_wait();
    LA_TRACE_CLUSTER(4);
    {
        const int R = in.R, slot = in.slot();
        const uint32_t vectors = smem_u32(smem + Sh::A);
        const float* sums = reinterpret_cast<const float*>(smem + Sh::IN2);
        in.template for_own_rows<THREADS>(reinterpret_cast<const float*>(smem + Sh::IN), [&](int d, int e, const float* from) {
            float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
            for (int c = 0; c < R; ++c) {
                const float4 v = *reinterpret_cast<const float4*>(from + c * slot);
                s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
            }
            uint32_t o0[NS], o1[NS];
            split2<NS>(s.x, s.y, o0);
            split2<NS>(s.z, s.w, o1);
            const uint32_t to = sS + tile_at<DP>(d, e / 8) + e % 8 * 2;
#pragma unroll 4
            for (int c = 0; c < R; ++c) {
                const uint32_t there = address_in(to, c);
#pragma unroll
                for (int k = 0; k < NS; ++k) peer_store(there + k * (DP * DP * 2), o0[k], o1[k]);
            }
            if (p.S1) *reinterpret_cast<float4*>(p.S1 + bh * DP * DP + d * DP + e) = s;       // (ysum is added below)
        }, [&](int d, int c, const float* from) {
            float a = 0.f, y = 0.f;
#pragma unroll 4
            for (int i = 0; i < R; ++i) {
                a += from[i * slot];
                y += sums[i * in.rows + d - in.me * in.rows];
            }
            const uint32_t to = address_in(vectors + d * 4, c);
            peer_store(to, a);
            peer_store(to + DP * 4, y);
            if (c == 0 && p.Z1) p.Z1[bh * DP + d] = a + (float)len;
        });
    }
    __syncwarp();
    LA_TRACE_CLUSTER(5);
    cluster_arrive();
    cluster_wait();
    LA_TRACE_CLUSTER(6);
    const float* sA = reinterpret_cast<const float*>(smem + Sh::A);
    const float* sY = reinterpret_cast<const float*>(smem + Sh::Y);
    float* sM = reinterpret_cast<float*>(smem + Sh::M);         // 1 . A', eight columns per warp
    if (warp < DP / 8) {
        const uint32_t ones[4] = {0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u};
        float u[NS][4] = {};            // (all three planes: these sums stay in 32 bits)
#pragma unroll
        for (int kk = 0; kk < DP / 16; ++kk) {
            uint32_t b[NS][4];
            load_cols_t<NS, DP>(b, sS, DP * DP * 2, kk * 16, warp / 2 * 2, lane);
#pragma unroll
            for (int k = 0; k < NS; ++k) mma16816(u[k], ones, warp % 2 ? b[k][2] : b[k][0], warp % 2 ? b[k][3] : b[k][1]);
        }
        if (g == 0) store_pair<float>(sM + warp * 8 + 2 * t, u[0][0] + (u[1][0] + u[2][0]), u[0][1] + (u[1][1] + u[2][1]));
    }
    if (p.S1) {                             // this CTA's rows of S = 1 ysum^T + A'
        const int d0 = in.me * in.rows, rows = min(in.rows, DP - d0);
        for (int i = id; i < rows * DP; i += THREADS) p.S1[bh * DP * DP + d0 * DP + i] += sY[i % DP];
    }
    float suma = 0.f;                       // 1 . a'
    for (int i = lane; i < DP; i += 32) suma += sA[i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) suma += __shfl_xor_sync(0xffffffffu, suma, off);
    IO* O = (IO*)p.O + bh * p.N * DP;
    float* den = p.den ? p.den + bh * p.N : nullptr;
    const float n = (float)len;
    __syncthreads();
#pragma unroll 1
    for (bool first = true; s0 < end; s0 += T, first = false) {
        const int cn = real_rows(s0, 16);
        if (!first) take_rows();
        float xa[2] = {0.f, 0.f}, inv[2];       // q' . a'
#pragma unroll
        for (int kk = 0; kk < DP / 16; ++kk)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 a = *reinterpret_cast<const float2*>(sA + kk * 16 + 2 * t + (j >> 1) * 8);
                xa[j & 1] = fmaf(__uint_as_float(qa[kk][0][j] << 16), a.x, fmaf(__uint_as_float(qa[kk][0][j] & 0xffff0000u), a.y, xa[j & 1]));
            }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float d = fmaf(n, x1[h], suma + quad_sum(xa[h]));
            inv[h] = 1.f / (d + p.eps);
            if (den && t == 0 && g + 8 * h < cn) den[s0 + g + 8 * h] = d;
        }
#pragma unroll
        for (int nn = 0; nn < DP / 16; ++nn) {
            float u[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}}, l[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
            for (int kk = 0; kk < DP / 16; ++kk) {
                uint32_t b[2][4];
                load_cols_t<2, DP>(b, sS, DP * DP * 2, kk * 16, nn * 2, lane);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    mma16816(u[i], qa[kk][0], b[0][2 * i], b[0][2 * i + 1]);
                    mma16816(l[i], qa[kk][0], b[1][2 * i], b[1][2 * i + 1]);
                }
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int col = nn * 16 + i * 8 + 2 * t;
                const float2 y = load_pair(sY + col);
                const float2 m = load_pair(sM + col);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (g + 8 * h < cn)
                        store_pair<IO>(O + (s0 + g + 8 * h) * DP + col, fmaf(x1[h], y.x, m.x + u[i][2 * h] + l[i][2 * h]) * inv[h],
                                       fmaf(x1[h], y.y, m.y + u[i][2 * h + 1] + l[i][2 * h + 1]) * inv[h]);
            }
        }
    }
    LA_TRACE_CLUSTER(7);
    if (end < hi) {
        zero_rows<THREADS>(O, end, hi, DP);
        if (den) zero_rows<THREADS>(den, end, hi, 1);
    }
    wait_last(p);
}

// ---- host ------------------------------------------------------------------------------------------------------
struct ClusterShape { int threads; unsigned ctas, bh; int smem, most_smem; };

template <auto KERNEL>
int opt_in(int most_smem) {
    static std::atomic<uint64_t> opted_in{0};           // devices on which the kernel may use that much shared memory and 16 CTAs
    int dev = 0;
    LA_CUDA_TRY(cudaGetDevice(&dev));
    const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0;
    if (!bit || !(opted_in.load(std::memory_order_acquire) & bit)) {
        LA_CUDA_TRY(cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, most_smem));
        LA_CUDA_TRY(cudaFuncSetAttribute(KERNEL, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        opted_in.fetch_or(bit, std::memory_order_release);
    }
    return LA_OK;
}

cudaLaunchConfig_t cluster_launch(const ClusterShape& s, cudaStream_t st, cudaLaunchAttribute (&attr)[2]) {
    cudaLaunchConfig_t cfg = tc::chained_launch(1, (unsigned)s.threads, (size_t)s.smem, st, attr);
    cfg.gridDim = dim3(s.ctas, s.bh);
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = s.ctas;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
    return cfg;
}

// The number of the context that the stream's work runs in, never the same for two contexts; 0: not known.  A stream of a
// green context (some of the device's SMs) belongs to the context of the whole device otherwise: 0 as well.
uint64_t context_number(cudaStream_t st) {
    typedef CUresult (*green_fn)(CUstream, CUgreenCtx*);
    typedef CUresult (*number_fn)(CUcontext, unsigned long long*);
    auto entry = [](const char* name) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint(name, &fn, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess) return fn;
        cudaGetLastError();
        return (void*)nullptr;
    };
    static const green_fn green_of = reinterpret_cast<green_fn>(entry("cuStreamGetGreenCtx"));
    static const number_fn number_of = reinterpret_cast<number_fn>(entry("cuCtxGetId"));
    CUgreenCtx green = nullptr;
    unsigned long long number = 0;
    if (!green_of || !number_of || green_of((CUstream)st, &green) != CUDA_SUCCESS || green) return 0;
    return number_of(nullptr, &number) == CUDA_SUCCESS ? number : 0;
}

// How many clusters the context of the stream runs at once: 0 where none has room (a cluster of sixteen CTAs needs them all in one
// GPC; a context that is limited to some SMs of the device may not have that).  Asked once per context, kernel and size: the
// question takes 0.7 us, a tenth of the smallest calls.
template <auto KERNEL>
int64_t clusters_at_once(const ClusterShape& s, cudaStream_t st) {
    static std::atomic<uint64_t> answers[2][kMaxCluster + 1];          // number of the context << 16 | answer
    std::atomic<uint64_t>& known = answers[s.smem != s.most_smem][s.ctas];
    const uint64_t context = context_number(st), last = known.load(std::memory_order_relaxed);
    if (context && last >> 16 == context) return (int64_t)(last & 0xffff);
    if (opt_in<KERNEL>(s.most_smem) != LA_OK) return 0;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_launch(s, st, attr);
    cfg.attrs = attr + 1;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, KERNEL, &cfg) != cudaSuccess) {
        cudaGetLastError();         // not an error of the caller's: the other kernels take the problem
        return 0;
    }
    if (context && context >> 48 == 0) known.store(context << 16 | (uint64_t)n, std::memory_order_relaxed);
    return n;
}

template <auto KERNEL, typename P>
int launch_cluster(ProfKernel prof, const ClusterShape& s, const P& a, cudaStream_t st) {
    if (int rc = opt_in<KERNEL>(s.most_smem)) return rc;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_launch(s, st, attr);
    prof_begin(prof, st);
    LA_CUDA_TRY(cudaLaunchKernelEx(&cfg, KERNEL, a));
    note_launch();
    prof_end(prof, st);
    return LA_OK;
}

ClusterParams cluster_params(const la_problem& p, const int* lengths) {
    ClusterParams a = {};
    a.lengths = lengths;
    a.N = p.N;
    a.heads = (int)p.H; a.D = (int)p.D; a.M = (int)p.M; a.phi = p.phi; a.eps = p.eps;
    return a;
}

template <typename C, int DP, int MP, int STRIPS, int WPS> struct Forward {
    static constexpr int T = 16 * STRIPS, BYTES = ForwardShared<C, DP, MP, STRIPS>::BYTES;
    static ClusterShape shape(const la_problem& p) {
        return {32 * STRIPS * WPS, (unsigned)((p.N + T - 1) / T), (unsigned)(p.B * p.H), BYTES, BYTES};
    }
    static int64_t at_once(const la_problem& p, cudaStream_t st) {
        return clusters_at_once<causal_cluster_forward_kernel<C, DP, MP, STRIPS, WPS>>(shape(p), st);
    }
    static int launch(const la_problem& p, const ClusterParams& a, cudaStream_t st) {
        return launch_cluster<causal_cluster_forward_kernel<C, DP, MP, STRIPS, WPS>>(kProfClusterForward, shape(p), a, st);
    }
};
template <typename C, int DP, int MP> struct Backward {
    static constexpr int STRIPS = 4, T = 16 * STRIPS, BYTES = BackwardShared<C, DP, MP, STRIPS>::BYTES;
    static ClusterShape shape(const la_problem& p) {
        return {64 * STRIPS, (unsigned)((p.N + T - 1) / T), (unsigned)(p.B * p.H), BYTES, BYTES};
    }
    static int64_t at_once(const la_problem& p, cudaStream_t st) {
        return clusters_at_once<causal_cluster_backward_kernel<C, DP, MP, STRIPS>>(shape(p), st);
    }
    static int launch(const la_problem& p, const BackwardParams& a, cudaStream_t st) {
        return launch_cluster<causal_cluster_backward_kernel<C, DP, MP, STRIPS>>(kProfClusterBackward, shape(p), a, st);
    }
};
template <int DP> struct Linear {
    static constexpr int STRIPS = 8, T = 16 * STRIPS;
    static int64_t tiles_per_cta(const la_problem& p) { return ((p.N + T - 1) / T + kMaxCluster - 1) / kMaxCluster; }
    static ClusterShape shape(const la_problem& p) {
        const int64_t tiles = (p.N + T - 1) / T, per = tiles_per_cta(p);
        return {32 * STRIPS, (unsigned)((tiles + per - 1) / per), (unsigned)(p.B * p.H),
                per > 1 ? LinearShared<DP, STRIPS>::BYTES : LinearShared<DP, STRIPS>::STAGE, LinearShared<DP, STRIPS>::BYTES};
    }
    static int64_t at_once(const la_problem& p, cudaStream_t st) { return clusters_at_once<linear_cluster_forward_kernel<DP, STRIPS>>(shape(p), st); }
    static int launch(const la_problem& p, ClusterParams a, cudaStream_t st) {
        a.piece_len = tiles_per_cta(p) * T;
        return launch_cluster<linear_cluster_forward_kernel<DP, STRIPS>>(kProfClusterLinear, shape(p), a, st);
    }
};

// the kernel of a problem that has one
template <typename F> auto with_forward(const la_problem& p, F f) {
    if (p.D == 128) return f(Forward<Bf16Features, 128, 64, 4, 2>());
    if (p.dtype == LA_F32) return p.D == 32 ? f(Forward<Fp32, 32, 32, 4, 2>()) : f(Forward<Fp32, 64, 64, 4, 2>());
    return p.D == 32 ? f(Forward<Bf16, 32, 32, 8, 1>()) : f(Forward<Bf16, 64, 64, 8, 1>());
}
template <typename F> auto with_backward(const la_problem& p, F f) {
    if (p.D == 128) return f(Backward<Bf16Features, 128, 64>());
    if (p.dtype == LA_F32) return p.D == 32 ? f(Backward<Fp32, 32, 32>()) : f(Backward<Fp32, 64, 64>());
    return p.D == 32 ? f(Backward<Bf16, 32, 32>()) : f(Backward<Bf16, 64, 64>());
}
template <typename F> auto with_linear(const la_problem& p, F f) { return p.D == 32 ? f(Linear<32>()) : f(Linear<64>()); }

int64_t tiles_of(const la_problem& p, int rows) { return (p.N + rows - 1) / rows; }

bool enabled() {
    static const bool on = getenv("LA_DISABLE_TC") == nullptr;
    return on;
}
bool fourier(const la_problem& p) { return p.dtype == LA_BF16 && p.D == 128 && p.M == 64 && p.phi == LA_PHI_IDENTITY; }
bool square(const la_problem& p) { return p.D == p.M && (p.D == 32 || p.D == 64); }

}  // namespace

// Which problems: those that one wave of clusters holds (clusters_at_once(): on a whole B200 with two CTAs per SM 148 of 2 CTAs, 93 of
// 3, 71 of 4, 45 of 6, 33 of 8, 26 of 10, 21 of 12, 14 of 14 to 16; with one 74, 45, 33, 22, 15, 11, 7, 7), or little more.
// us of GPU time, the other kernels / these, B x H x N:
//   forward, bf16 (128 positions a CTA, two CTAs per SM): up to 256 positions the tcgen05 kernel is one launch too (D = 64 1x8x128
//     5.1 / 9.4).  D = 64: 1x8x600 16.4 / 7.7, 6x8x500 15.4 / 10.9, 1x8x2048 18.8 / 11.3; three tiles with CTAs that share an SM 5x8x384
//     8.8 / 8.0, but 6x8x300 10.0 / 10.4, 6x8x384 9.0 / 10.8 (from a state, which costs the other kernel 3, 12.1 / 11.1); a second wave
//     pays from eight tiles on (2x8x2048 22.7 / 18.1, 6x8x1024 21.4 / 20.8, 3x8x2048 23.2 / 21.8), a third does not (4x8x2048 27.4 / 29.0).
//     D = 32: 1x8x600 14.2 / 4.5, 10x8x300 8.3 / 5.9 but 12x8x300, a second wave, 8.2 / 8.9; 9x8x512 16.6 / 8.8, 8x8x1000 20.8 / 11.3
//   ... with a saved buffer whose records the tcgen05 backward kernels take, their pre-pass being on top: D = 64 6x8x500 15.9 / 13.2,
//     4x8x1000 20.6 / 20.2, but in two waves 6x8x1024 22.1 / 25.1, 8x8x1000 24.8 / 31.9, 4x8x2048 28.4 / 36.4 (forward + backward 73.0 /
//     85.0); D = 32 5x8x1024 19.5 / 14.8, 3x8x2048 21.1 / 19.0, 5x8x1536 22.2 / 22.4, 4x8x2048 24.4 / 24.8 (without the buffer 23.8 / 16.6)
//   backward (64 positions a CTA), bf16: D = 32 4x8x576 34.4 / 18.5, 6x8x384 18.2 / 18.0, but 9x8x256, two chunks of the other kernel,
//     14.9 / 15.9; D = 64 4x8x320 25.1 / 19.6, 1x8x1024 34.9 / 19.9, 2x8x704 35.7 / 20.3; 1x8x128 10.3 / 14.4
//   fp32 (64 a CTA): one CTA per sequence is no gain (1x2x64 D = 32 15.8 / 17.9).  D = 64, one CTA per SM, forward and backward: 9x8x128 14.4 / 10.8
//     and 36.7 / 23.4, 4x8x256 15.9 / 10.8 and 38.3 / 24.1, 1x6x1000 19.8 / 11.1 and 44.6 / 24.6; in two waves, the second well filled
//     4x8x384 23.3 / 21.2 and 55.8 / 46.1, 7x8x192 19.3 / 20.3 and 49.5 / 44.9, 12x8x128 16.3 / 19.8 and 44.7 / 44.1, or not 6x8x192
//     15.5 / 19.9 and 37.3 / 44.5, 3x8x384 16.3 / 20.7 and 38.0 / 45.2, 1x8x700 18.2 / 20.5 and 40.5 / 45.6.  D = 32, two CTAs: 5x8x384
//     11.1 / 8.0 and 25.8 / 18.2; in two waves 12x8x192 10.6 / 12.1 and 25.5 / 28.3, 3x8x768 12.6 / 14.2 and 30.7 / 30.0, but these
//     calls are bound by the host, two launches for one and six: 14.5 / 12.6 and 34.1 / 28.5, 16.7 / 14.4 and 39.2 / 31.1
//   and with the 128 Fourier features, forward + backward 1x8x1000 130 / 75, 8x8x142 79 / 68, 3x8x512 117 / 73; 8x8x500 188 / 201
int64_t waves(const la_problem& p, int64_t at_once) { return at_once > 0 ? (p.B * p.H + at_once - 1) / at_once : INT64_MAX; }
// fp32, D = M = 64: one wave, or two of which the second is at least a fifth full
bool well_filled(const la_problem& p, int64_t at_once) {
    const int64_t w = waves(p, at_once);
    return w == 1 || (w == 2 && 5 * p.B * p.H >= 6 * at_once);
}

// saved: with a buffer for the tcgen05 backward kernels; state: from a given state
bool causal_cluster_forward_preferred(const la_problem& p, bool saved, bool state, cudaStream_t st) {
    if (!enabled() || tc::causal_pieces_override() >= 0 || !(square(p) || fourier(p))) return false;
    const bool exact = p.dtype == LA_F32 || fourier(p);
    const int64_t tiles = tiles_of(p, exact ? 64 : 128), ctas = tiles * p.B * p.H;
    if (tiles <= (exact ? 1 : 2) || tiles > kMaxCluster || ctas > 512) return false;
    const int64_t at_once = with_forward(p, [&](auto k) { return decltype(k)::at_once(p, st); }), w = waves(p, at_once);
    if (at_once == 0) return false;
    if (exact && p.D == 64) return ctas <= 192 && well_filled(p, at_once) && (w == 1 || tiles > 2);
    if (exact) return ctas <= (p.D == 32 ? 296 : 192);
    if (p.D == 32) return (ctas <= 296 && (tiles > 3 || w == 1)) || tiles >= 8;
    const bool records = saved && !causal_cluster_backward_size(p);
    return ctas <= (tiles > 3 ? 200 : state ? 148 : 132) || (tiles >= 8 && w <= (records ? 1 : 2));
}
bool causal_cluster_backward_size(const la_problem& p) {
    if (!enabled() || tc::causal_pieces_override() >= 0 || !(square(p) || fourier(p))) return false;
    const bool bf16 = p.dtype == LA_BF16;
    const int64_t tiles = tiles_of(p, 64), ctas = tiles * p.B * p.H;
    return tiles > (bf16 && p.D == 64 ? 4 : 1) && tiles <= kMaxCluster && ctas <= (p.D == 32 ? (bf16 && tiles == 4 ? 256 : 296) : 192);
}
bool causal_cluster_backward_preferred(const la_problem& p, cudaStream_t st) {
    if (!causal_cluster_backward_size(p)) return false;
    const int64_t at_once = with_backward(p, [&](auto k) { return decltype(k)::at_once(p, st); });
    return at_once > 0 && (p.dtype == LA_BF16 || p.D == 32 || well_filled(p, at_once));
}
// GPU us without a buffer for the sums / encoder forward + backward with one, whose sums need a kernel of their own (results do not
// depend on the buffer, so neither does the rule: where the two disagree a training step loses less than an encoder gains): D = 64 1x8x64
// 11.5 / 8.1 and 27.2 / 27.0, 1x8x1000 14.2 / 9.3 and 37.1 / 34.6, 4x8x384 15.4 / 8.8 and 40.8 / 36.0, 1x12x1500 16.1 / 14.2 and 40.5 / 41.8,
// 18x8x100 13.2 / 8.6 and 32.1 / 36.5; D = 32 1x8x1000 13.9 / 5.9 and 36.5 / 30.3, 56x8x128 42.0 / 12.2 and 101 / 90, 4x8x1024 15.0 / 8.0 and
// 38.2 / 39.3, 8x8x777 18.9 / 13.5 and 48.8 / 51.7, 3x8x1800 18.5 / 14.4 and 46.6 / 51.6, but in three waves 4x8x1700 18.3 / 20.2 and 49.0 /
// 59.0.  More than a tile per CTA: 1x8x4096 18.6 / 10.4 and 47.8 / 48.1, 1x8x8192 22.1 / 15.7 and 58.9 / 62.8, 4x8x4096 26.1 / 28.9
bool linear_cluster_preferred(const la_problem& p, cudaStream_t st) {
    if (!enabled() || tc::linear_splits_override() >= 0 || p.dtype != LA_BF16 || !square(p) || p.N < 1) return false;
    const int64_t tiles = tiles_of(p, 128);
    if (p.D == 64 ? tiles > 12 || tiles * p.B * p.H > 148
                  : tiles <= kMaxCluster ? tiles * p.B * p.H > 448 : tiles > 4 * kMaxCluster || kMaxCluster * p.B * p.H > 148) return false;
    const int64_t at_once = with_linear(p, [&](auto k) { return decltype(k)::at_once(p, st); });
    return waves(p, at_once) <= 2;
}

int causal_cluster_forward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const float* S_in,
                           const float* Z_in, void* O, float* den, float* S_out, float* Z_out, void* saved, cudaStream_t st) {
    ClusterParams a = cluster_params(p, lengths);
    a.Q = Q; a.K = K; a.V = V; a.O = O; a.den = den;
    a.S0 = S_in; a.Z0 = Z_in; a.S1 = S_out; a.Z1 = Z_out;
    if (saved) {                // what the tcgen05 backward pass finds there, where that is the one to come
        const tc::CausalPlan pl = tc::choose_plan(p);
        const tc::SavedLayout l = tc::saved_layout(p, pl);
        char* sv = (char*)saved;
        a.stamp = (int*)(sv + l.stamp);
        if (p.phi == LA_PHI_ELU1) { a.keep_q = sv + l.phiq; a.keep_k = sv + l.phik; }
        if (!causal_cluster_backward_size(p)) {
            tc::plan_stamp(pl, (int)p.D, a.stamp_value);
            if (pl.npieces() > 1) {
                if (int rc = tc::causal_keep_records(p, K, V, lengths, saved, st)) return rc;
                a.late = 1;
            }
        }
    }
    return with_forward(p, [&](auto k) { return decltype(k)::launch(p, a, st); });
}

int causal_cluster_backward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const void* G,
                            const StateArgs& sa, void* dQ, void* dK, void* dV, cudaStream_t st) {
    BackwardParams a = {};
    static_cast<ClusterParams&>(a) = cluster_params(p, lengths);
    a.Q = Q; a.K = K; a.V = V; a.G = G; a.dQ = dQ; a.dK = dK; a.dV = dV;
    a.S0 = sa.S_in; a.Z0 = sa.Z_in; a.R0 = sa.dS_out; a.r0 = sa.dZ_out; a.R1 = sa.dS_in; a.r1 = sa.dZ_in;
    return with_backward(p, [&](auto k) { return decltype(k)::launch(p, a, st); });
}

int linear_cluster_forward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, void* O, float* den,
                           float* KV, float* Zs, void* saved, cudaStream_t st) {
    ClusterParams a = cluster_params(p, lengths);
    a.Q = Q; a.K = K; a.V = V; a.O = O; a.den = den; a.S1 = KV; a.Z1 = Zs;
    if (saved) {                // the sums that the backward pass takes
        if (int rc = tc::linear_keep_sums(p, K, V, lengths, saved, st)) return rc;
        a.late = 1;
    }
    return with_linear(p, [&](auto k) { return decltype(k)::launch(p, a, st); });
}

}  // namespace la

#ifdef LA_TC_TRACE
extern "C" int la_debug_read_trace_cluster(long long* out, int n) {
    return (int)cudaMemcpyFromSymbol(out, la::g_trace_cluster, n * sizeof(long long));
}
#endif
