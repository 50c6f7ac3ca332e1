// Causal form (Eq. 8-15) at fp32 accuracy on mma.sync (la_mma.cuh): fp32 problems, and bf16 ones of shapes or feature
// maps that the tcgen05 kernels do not take; M <= 64, any D.
//
// A sequence is cut into pieces, one CTA of four warps each; a CTA walks its piece in chunks of T = 64 positions.
// Per chunk a warp owns a strip of sixteen rows (queries in the forward sweeps, keys in the reverse one) whose
// operand it loads from global memory into registers, and sixteen rows of the running state per 64 of D, kept in
// fp32 registers.  The other operands (K | V, or Q / dn | G) and the state before the chunk lie in shared memory as
// bf16 planes.  Two barriers per chunk: planes free, planes written.
//
//   forward   O  = [(q k^T o L) [V | 1] + q [S | Z]],            S += k^T V,  Z += k^T 1
//   dQ sweep  h  = (G V^T o L) k + G S^T,  Zc = L k + Z,  dn = q . Zc + eps,
//             gq = (h - (q . h / dn) Zc) / dn                     (the same S, Z; dn and -(q . h) / dn are parked)
//   dK, dV    with q^ = q / dn, dl = -G . O:  gV = (q^ k^T o L)^T G + k R,
//             gk = ((G V^T + dl) o L)^T q^ + V R^T + r,           R += q^^T G,  r += q^^T dl  (chunks last to first)
//
// Pieces other than the first (last, for the reverse sweep) start from the sum of the records [S | Z] of the pieces
// before (after) them, which a pre-pass writes to the workspace.
#include "la_mma.cuh"
#include "la_tc.cuh"

namespace la {
namespace {

using namespace mma;

constexpr int T = 64;
constexpr int THREADS = 128;
constexpr int WARPS = THREADS / 32;
static_assert(T == 16 * WARPS, "one strip of sixteen rows per warp");

struct Params {
    const void *Q, *K, *V, *G;
    void *O, *dQ, *dK, *dV;
    float* den;
    const float *S0, *Z0;        // state the sweep starts from (forward: S_in, Z_in; reverse: dS_out, dZ_out), each or null
    float *S1, *Z1;              // where the state it ends with goes (S_out, Z_out / dS_in, dZ_in), each or null
    float* rec;                  // [bh][pieces - 1][D * M + D]: sums of pieces 0 .. pieces - 2 (reverse: 1 .. pieces - 1)
    float* aux;                  // [bh][2][N]: dn_i, -G_i . O_i
    const int* lengths;
    int64_t N, piece_len;
    int pieces, heads, D, M, phi;
    float eps;
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

template <typename IO>
__device__ void zero_rows(IO* x, int64_t from, int64_t to, int cols) {       // rows from .. to - 1
    for (int64_t i = from * cols + threadIdx.x; i < to * cols; i += THREADS) x[i] = from_f32<IO>(0.f);
}

// The running sums of a warp: rows d = 16 strip + g (+ 8), strip = warp (+ 4); with two strips (D <= 32) two warps
// share one and take half of its columns each.  Columns e = 8 (n0 + n) + 2 t (+ 1).
template <int DP, int MP>
struct State {
    static constexpr int STRIPS = DP / 16, SHARE = STRIPS < WARPS ? WARPS / STRIPS : 1, SD = STRIPS < WARPS ? 1 : STRIPS / WARPS;
    static constexpr int NC = MP / 8 / SHARE;
    static __device__ __forceinline__ int strip(int i) { return ((int)threadIdx.x >> 5) % STRIPS + WARPS * i; }
    static __device__ __forceinline__ int n0() { return SHARE == 1 ? 0 : ((int)threadIdx.x >> 5) / STRIPS * NC; }
    float s[SD][NC][4];
    float z[SD][2];             // in every warp that shares the strip

    __device__ __forceinline__ void init(const Params& p, const float* S0, const float* Z0, const float* rec, int nrec) {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, c0 = n0();
        const int size = p.D * p.M + p.D;
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
            for (int r = 0; r < nrec; ++r) {
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
    // the operand planes [DP][MP] of the matrix and the vector in fp32
    template <int NS>
    __device__ __forceinline__ void publish(uint8_t* tile, float* vec) const {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, c0 = n0();
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
                vec[d] = z[i][0];
                vec[d + 8] = z[i][1];
            }
        }
    }
    // s += X^T Y, z += X^T w over the rows of the tiles X [T][DP] (NX planes), Y [T][MP] (NY);
    // w: ones, or the vector whose three planes of T elements are at wpl
    // (a chunk that is not full has zeros in the tiles' other rows)
    template <int NX, int NY, bool ONES>
    __device__ __forceinline__ void update(uint32_t X, uint32_t Y, const uint16_t* wpl) {
        const int lane = threadIdx.x & 31, t = lane & 3, c0 = n0();
#pragma unroll
        for (int i = 0; i < SD; ++i) {
            uint32_t a[T / 16][NX][4];
            float zs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int b = 0; b < T / 16; ++b)
                {
                    load_rows_t<NX, DP>(a[b], X, T * DP * 2, b * 16, strip(i) * 2, lane);
                    float u[4] = {0.f, 0.f, 0.f, 0.f};
                    if constexpr (ONES) {
#pragma unroll
                        for (int k = NX - 1; k >= 0; --k) mma16816(u, a[b][k], 0x3f803f80u, 0x3f803f80u);
                    } else {
                        uint32_t w[3][2];
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            w[k][0] = *reinterpret_cast<const uint32_t*>(wpl + k * T + b * 16 + 2 * t);
                            w[k][1] = *reinterpret_cast<const uint32_t*>(wpl + k * T + b * 16 + 8 + 2 * t);
                        }
#pragma unroll
                        for (int sum = 2; sum >= 0; --sum)
#pragma unroll
                            for (int k = 0; k < NX; ++k)
                                if (sum - k >= 0) mma16816(u, a[b][k], w[sum - k][0], w[sum - k][1]);
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
                for (int b = 0; b < T / 16; ++b) {
                        uint32_t y[NY][4];
                        load_cols_t<NY, MP>(y, Y, T * MP * 2, b * 16, c0 + n * 2, lane);
                        c.step<NX, NY>(a[b], y);
                    }
                c.add_to(s[i][2 * n], s[i][2 * n + 1]);
            }
        }
    }
};

// I/O type and planes of each kind of operand: feature-mapped rows (NQ), value rows V, G (NV), scores (NP), state (NS),
// q / dn (NR).  Everything computed in fp32 has three planes; bf16 values, and features that are bf16 as given, one.
struct Fp32 { using IO = float; static constexpr int NQ = 3, NV = 3, NP = 3, NS = 3, NR = 3, BUF = 1; static constexpr bool MAPPED = true; };
struct Bf16Wide { using IO = __nv_bfloat16; static constexpr int NQ = 3, NV = 1, NP = 3, NS = 3, NR = 3, BUF = 1; static constexpr bool MAPPED = true; };
struct Bf16Features { using IO = __nv_bfloat16; static constexpr int NQ = 1, NV = 1, NP = 3, NS = 3, NR = 3, BUF = 1; static constexpr bool MAPPED = false; };
// bf16 operands throughout (with fp32 sums), as the tcgen05 kernels have them.  BUF = 2: the small tiles are there twice,
// one barrier per chunk (the other set was last read before the barrier of this chunk).
struct Bf16 { using IO = __nv_bfloat16; static constexpr int NQ = 1, NV = 1, NP = 1, NS = 1, NR = 1, BUF = 2; static constexpr bool MAPPED = true; };

template <int DP, int MP, int NX, int NY, int NS> struct Shared {       // tile X [T][DP], tile Y [T][MP], state planes, vectors
    static constexpr int X = 0, Y = X + NX * T * DP * 2, S = Y + NY * T * MP * 2, Z = S + NS * DP * MP * 2,
                         W = Z + DP * 4, WP = W + T * 4, BYTES = (WP + 3 * T * 2 + 127) / 128 * 128;
};
// CTAs of an SM that the registers are shared out for: as many as shared memory holds, at most `most`
template <typename Sh, typename C> constexpr int resident(int most) {
    const int fit = 227 * 1024 / (C::BUF * Sh::BYTES + 1024);
    return fit < most ? fit : most;
}

template <typename C, typename Sh>
__device__ __forceinline__ void flip(uint8_t*& buf, uint8_t* smem) {
    if constexpr (C::BUF == 2) buf = buf == smem ? smem + Sh::BYTES : smem;
}

template <typename IO>
__device__ __forceinline__ void prefetch_rows(const IO* x, int64_t n0, int64_t end, int cols) {
    if (n0 < 0 || n0 >= end) return;
    const int64_t rows = end - n0 < T ? end - n0 : T;
    const char* p = reinterpret_cast<const char*>(x + n0 * cols);
    for (int64_t o = threadIdx.x * 128; o < rows * cols * (int64_t)sizeof(IO); o += THREADS * 128) prefetch_l2(p + o);
}

// feature-mapped pairs in registers: bf16 where features have one plane
template <int NQ> struct FeatureType { using type = float; };
template <> struct FeatureType<1> { using type = __nv_bfloat16; };

// ---- forward ---------------------------------------------------------------------------------------------------
template <typename C, int DP, int MP, bool EXACT>
__global__ void __launch_bounds__(THREADS, (resident<Shared<DP, MP, C::NQ, C::NV, C::NS>, C>(C::NP == 1 ? 4 : sizeof(typename C::IO) == 4 && DP == 64 ? 2 : 3)))
causal_mma_forward_kernel(const Params p) {
    using IO = typename C::IO;
    constexpr int NQ = C::NQ, NV = C::NV, NP = C::NP, NS = C::NS;
    using Sh = Shared<DP, MP, NQ, NV, NS>;
    extern __shared__ __align__(128) uint8_t smem[];
    uint8_t* buf = smem;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int D = EXACT ? DP : p.D, M = EXACT ? MP : p.M, phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    const Range r = range_of(p, blockIdx.y);
    const IO* Q = (const IO*)p.Q + r.bh * p.N * D;
    const IO* K = (const IO*)p.K + r.bh * p.N * D;
    const IO* V = (const IO*)p.V + r.bh * p.N * M;
    IO* O = (IO*)p.O + r.bh * p.N * M;
    float* den = p.den ? p.den + r.bh * p.N : nullptr;

    State<DP, MP> st;
    st.init(p, p.S0 ? p.S0 + r.bh * D * M : nullptr, p.Z0 ? p.Z0 + r.bh * D : nullptr,
            p.rec + r.bh * (p.pieces - 1) * (int64_t)(D * M + D), r.piece);
    for (int64_t n0 = r.lo; n0 < r.end; n0 += T) {
        const uint32_t sK = smem_u32(buf + Sh::X), sV = smem_u32(buf + Sh::Y), sS = smem_u32(buf + Sh::S);
        float* sZ = reinterpret_cast<float*>(buf + Sh::Z);
        const int cn = (int)(r.end - n0 < T ? r.end - n0 : T);
        // (the strip with the most blocks left of the diagonal goes round the schedulers)
        const int strip = ((n0 / T) & 1) ? WARPS - 1 - warp : warp, row0 = strip * 16;
        RawStrip<IO, DP> rq;
        rq.load(Q + n0 * D, row0, cn, D, pad);
        {
            RawTile<IO, T, DP, THREADS> rk;
            RawTile<IO, T, MP, THREADS> rv;
            rk.load(K + n0 * D, cn, D, pad);
            rv.load(V + n0 * M, cn, M, 0.f);
            if constexpr (C::BUF == 1) __syncthreads();         // the planes of the chunk before are no longer read
            st.template publish<NS>(buf + Sh::S, sZ);
            with_phi<NQ>(phi, [&](auto f) { rk.template store<NQ>(buf + Sh::X, [&](int, float x) { return f(x); }); });
            rv.template values<NV>(buf + Sh::Y);
        }
        prefetch_rows(Q, n0 + T, r.end, D);
        prefetch_rows(K, n0 + T, r.end, D);
        prefetch_rows(V, n0 + T, r.end, M);
        __syncthreads();
        if (row0 < cn) {
            RawStrip<typename FeatureType<NQ>::type, DP> fq;
            rq.template map<NQ>(phi, fq);
            float d0 = 0.f, d1 = 0.f;           // rows g, g + 8: q . Z, then + the scores
#pragma unroll
            for (int kk = 0; kk < DP / 16; ++kk)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 z = *reinterpret_cast<const float2*>(sZ + kk * 16 + h * 8 + 2 * t);
                    d0 = fmaf(fq.r[kk][2 * h].lo(), z.x, fmaf(fq.r[kk][2 * h].hi(), z.y, d0));
                    d1 = fmaf(fq.r[kk][2 * h + 1].lo(), z.x, fmaf(fq.r[kk][2 * h + 1].hi(), z.y, d1));
                }
            uint32_t qa[DP / 16][NQ][4];
            fq.template planes<NQ>(qa);
            float o[MP / 8][4];
#pragma unroll
            for (int n = 0; n < MP / 16; ++n) {
                Chain c;
#pragma unroll
                for (int kk = 0; kk < DP / 16; ++kk) {
                    uint32_t b[NS][4];
                    load_cols_t<NS, MP>(b, sS, DP * MP * 2, kk * 16, n * 2, lane);
                    c.step<NQ, NS>(qa[kk], b);
                }
                c.put(o[2 * n], o[2 * n + 1]);
            }
#pragma unroll 1
            for (int jb = 0; jb <= strip; ++jb) {
                float s0[4], s1[4];
                {
                    Chain c;
#pragma unroll
                    for (int kk = 0; kk < DP / 16; ++kk) {
                        uint32_t b[NQ][4];
                        load_rows<NQ, DP>(b, sK, T * DP * 2, jb * 16, kk * 2, lane);
                        c.step<NQ, NQ>(qa[kk], b);
                    }
                    c.put(s0, s1);
                }
                if (jb == strip) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int row = g + (j >> 1) * 8, col = 2 * t + (j & 1);
                        if (col > row) s0[j] = 0.f;
                        if (col + 8 > row) s1[j] = 0.f;
                    }
                }
                uint32_t pa[NP][4];
                operand_of<NP>(pa, s0, s1);
                if constexpr (NP == 1) {
                    float u[4] = {0.f, 0.f, 0.f, 0.f};
                    mma16816(u, pa[0], 0x3f803f80u, 0x3f803f80u);       // row sums (in every column; lane 0 of a row counts)
                    d0 += t == 0 ? u[0] : 0.f;
                    d1 += t == 0 ? u[2] : 0.f;
                } else {
                    d0 += (s0[0] + s0[1]) + (s1[0] + s1[1]);
                    d1 += (s0[2] + s0[3]) + (s1[2] + s1[3]);
                }
#pragma unroll
                for (int n = 0; n < MP / 16; ++n) {
                    uint32_t b[NV][4];
                    load_cols_t<NV, MP>(b, sV, T * MP * 2, jb * 16, n * 2, lane);
                    block_mma<NP, NV>(o[2 * n], o[2 * n + 1], pa, b);
                }
            }
            d0 = quad_sum(d0);
            d1 = quad_sum(d1);
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
        flip<C, Sh>(buf, smem);
    }
    zero_rows(O, r.end, r.hi, M);
    if (den) zero_rows(den, r.end, r.hi, 1);
    if (r.piece == p.pieces - 1) st.write(p, p.S1 ? p.S1 + r.bh * D * M : nullptr, p.Z1 ? p.Z1 + r.bh * D : nullptr);
}

// ---- sums over a piece: the forward records [k^T V | k^T 1], or the reverse ones [q^^T G | q^^T dl] -----------------
// Reverse tiles: q^ = phi(Q) / dn and the planes of dl, from the parked dn_i, dl_i.
template <typename IO, int DP, int MP>
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

template <typename C, int DP, int MP, bool EXACT, bool REVERSE>
__global__ void __launch_bounds__(THREADS, C::NP == 1 ? 4 : 2)
causal_mma_sum_kernel(const Params p) {
    using IO = typename C::IO;
    constexpr int NX = REVERSE ? C::NR : C::NQ, NY = C::NV;
    using Sh = Shared<DP, MP, NX, NY, C::NS>;          // (the state planes are not used: the launch asks for less)
    extern __shared__ __align__(128) uint8_t smem[];
    uint8_t* buf = smem;
    const int D = EXACT ? DP : p.D, M = EXACT ? MP : p.M, phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    const Range r = range_of(p, (int)blockIdx.y + (REVERSE ? 1 : 0));
    const IO* X = (const IO*)(REVERSE ? p.Q : p.K) + r.bh * p.N * D;
    const IO* Y = (const IO*)(REVERSE ? p.G : p.V) + r.bh * p.N * M;
    const float* dn = REVERSE ? p.aux + r.bh * 2 * p.N : nullptr;
    const float* delta = REVERSE ? dn + p.N : nullptr;
    State<DP, MP> st;
    st.init(p, nullptr, nullptr, nullptr, 0);
    for (int64_t n0 = r.lo; n0 < r.end; n0 += T) {
        float* w = reinterpret_cast<float*>(buf + Sh::S);
        uint16_t* wpl = reinterpret_cast<uint16_t*>(w + T);
        const int cn = (int)(r.end - n0 < T ? r.end - n0 : T);
        if constexpr (REVERSE) {
            ReverseRows<IO, DP, MP> rr;
            rr.load(X, Y, dn, delta, n0, cn, D, M, pad);
            if constexpr (C::BUF == 1) __syncthreads();
            rr.template store<NX, NY>(buf + Sh::X, buf + Sh::Y, w, wpl, phi);
        } else {
            RawTile<IO, T, DP, THREADS> rx;
            RawTile<IO, T, MP, THREADS> ry;
            rx.load(X + n0 * D, cn, D, pad);
            ry.load(Y + n0 * M, cn, M, 0.f);
            if constexpr (C::BUF == 1) __syncthreads();
            with_phi<NX>(phi, [&](auto f) { rx.template store<NX>(buf + Sh::X, [&](int, float x) { return f(x); }); });
            ry.template values<NY>(buf + Sh::Y);
        }
        prefetch_rows(X, n0 + T, r.end, D);
        prefetch_rows(Y, n0 + T, r.end, M);
        __syncthreads();
        st.template update<NX, NY, !REVERSE>(smem_u32(buf + Sh::X), smem_u32(buf + Sh::Y), wpl);
        flip<C, Sh>(buf, smem);
    }
    float* dst = p.rec + (r.bh * (p.pieces - 1) + blockIdx.y) * (int64_t)(D * M + D);
    st.write(p, dst, dst + D * M);
}

// ---- dQ sweep --------------------------------------------------------------------------------------------------
template <typename C, int DP, int MP, bool EXACT>
__global__ void __launch_bounds__(THREADS, (resident<Shared<DP, MP, C::NQ, C::NV, C::NS>, C>(C::NP == 1 ? 4 : 2)))
causal_mma_dq_kernel(const Params p) {
    using IO = typename C::IO;
    constexpr int NQ = C::NQ, NV = C::NV, NP = C::NP, NS = C::NS;
    using Sh = Shared<DP, MP, NQ, NV, NS>;
    extern __shared__ __align__(128) uint8_t smem[];
    uint8_t* buf = smem;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int D = EXACT ? DP : p.D, M = EXACT ? MP : p.M, phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    const Range r = range_of(p, blockIdx.y);
    const IO* Q = (const IO*)p.Q + r.bh * p.N * D;
    const IO* K = (const IO*)p.K + r.bh * p.N * D;
    const IO* V = (const IO*)p.V + r.bh * p.N * M;
    const IO* G = (const IO*)p.G + r.bh * p.N * M;
    IO* dQ = (IO*)p.dQ + r.bh * p.N * D;
    float* dn_all = p.aux + r.bh * 2 * p.N;
    float* dl_all = dn_all + p.N;

    State<DP, MP> st;
    st.init(p, p.S0 ? p.S0 + r.bh * D * M : nullptr, p.Z0 ? p.Z0 + r.bh * D : nullptr,
            p.rec + r.bh * (p.pieces - 1) * (int64_t)(D * M + D), r.piece);
    for (int64_t n0 = r.lo; n0 < r.end; n0 += T) {
        const uint32_t sK = smem_u32(buf + Sh::X), sV = smem_u32(buf + Sh::Y), sS = smem_u32(buf + Sh::S);
        float* sZ = reinterpret_cast<float*>(buf + Sh::Z);
        const int cn = (int)(r.end - n0 < T ? r.end - n0 : T);
        const int strip = ((n0 / T) & 1) ? WARPS - 1 - warp : warp, row0 = strip * 16;
        uint32_t ga[MP / 16][NV][4];
        {
            RawStrip<IO, MP> rg;
            RawTile<IO, T, DP, THREADS> rk;
            RawTile<IO, T, MP, THREADS> rv;
            rg.load(G + n0 * M, row0, cn, M, 0.f);
            rk.load(K + n0 * D, cn, D, pad);
            rv.load(V + n0 * M, cn, M, 0.f);
            if constexpr (C::BUF == 1) __syncthreads();
            st.template publish<NS>(buf + Sh::S, sZ);
            with_phi<NQ>(phi, [&](auto f) { rk.template store<NQ>(buf + Sh::X, [&](int, float x) { return f(x); }); });
            rv.template values<NV>(buf + Sh::Y);
            rg.template planes<NV>(ga);
        }
        prefetch_rows(Q, n0 + T, r.end, D);
        prefetch_rows(K, n0 + T, r.end, D);
        prefetch_rows(V, n0 + T, r.end, M);
        prefetch_rows(G, n0 + T, r.end, M);
        __syncthreads();
        // The first chunk of a sequence goes through twice, the second time with the G_i . O_i it found taken off the
        // scores: where few terms make up a row, h and (q . h / dn) Zc cancel almost entirely (in row 0 completely).
        float c0 = 0.f, c1 = 0.f;               // G_i . O_i of rows g, g + 8, as far as it is known
        for (int pass = row0 >= cn ? 2 : (n0 == 0 && !p.S0) ? 0 : 1; pass < 2; ++pass) {
            float h[DP / 8][4], zc[DP / 8][4];
#pragma unroll
            for (int n = 0; n < DP / 8; ++n) {
                const float2 z = *reinterpret_cast<const float2*>(sZ + n * 8 + 2 * t);
                zc[n][0] = zc[n][2] = z.x;
                zc[n][1] = zc[n][3] = z.y;
            }
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
#pragma unroll 1
            for (int jb = 0; jb <= strip; ++jb) {
                float s0[4], s1[4];
                {
                    Chain c;
#pragma unroll
                    for (int ee = 0; ee < MP / 16; ++ee) {
                        uint32_t b[NV][4];
                        load_rows<NV, MP>(b, sV, T * MP * 2, jb * 16, ee * 2, lane);
                        c.step<NV, NV>(ga[ee], b);
                    }
                    c.put(s0, s1);
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    s0[j] -= c0; s1[j] -= c0;
                    s0[2 + j] -= c1; s1[2 + j] -= c1;
                }
                uint32_t ones[1][4] = {{0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u}};
                if (jb == strip) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int row = g + (j >> 1) * 8, col = 2 * t + (j & 1);
                        if (col > row) s0[j] = 0.f;
                        if (col + 8 > row) s1[j] = 0.f;
                    }
                    ones[0][0] = ones[0][3] = (2 * t <= g ? 0x3f80u : 0u) | (2 * t + 1 <= g ? 0x3f800000u : 0u);
                    ones[0][2] = 0u;
                }
                uint32_t pa[NP][4];
                operand_of<NP>(pa, s0, s1);
#pragma unroll
                for (int n = 0; n < DP / 16; ++n) {
                    uint32_t b[NQ][4];
                    load_cols_t<NQ, DP>(b, sK, T * DP * 2, jb * 16, n * 2, lane);
                    block_mma<NP, NQ>(h[2 * n], h[2 * n + 1], pa, b);
                    block_mma<1, NQ>(zc[2 * n], zc[2 * n + 1], ones, b);
                }
            }
            RawStrip<IO, DP> rq;                // element j of block kk: result column tile 2 kk + j / 2, row g + 8 (j & 1)
            rq.load(Q + n0 * D, row0, cn, D, pad);
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
                const float inv = 1.f / dn, go = (quad_sum(qh[b]) - (b ? c1 : c0) * p.eps) * inv;    // what is left of G_i . O_i
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
        }
        st.template update<NQ, NV, true>(sK, sV, nullptr);
        flip<C, Sh>(buf, smem);
    }
    zero_rows(dQ, r.end, r.hi, D);
}

// ---- dK, dV sweep ----------------------------------------------------------------------------------------------
template <typename C, int DP, int MP, bool EXACT>
__global__ void __launch_bounds__(THREADS, (resident<Shared<DP, MP, C::NR, C::NV, C::NS>, C>(C::NP == 1 ? 4 : 3)))
causal_mma_dkv_kernel(const Params p) {
    using IO = typename C::IO;
    constexpr int NQ = C::NQ, NV = C::NV, NP = C::NP, NS = C::NS, NR = C::NR;
    using Sh = Shared<DP, MP, NR, NV, NS>;
    extern __shared__ __align__(128) uint8_t smem[];
    uint8_t* buf = smem;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int D = EXACT ? DP : p.D, M = EXACT ? MP : p.M, phi = C::MAPPED ? p.phi : (int)LA_PHI_IDENTITY;
    const float pad = pad_value(phi);
    const Range r = range_of(p, (int)(gridDim.y - 1 - blockIdx.y));
    const IO* Q = (const IO*)p.Q + r.bh * p.N * D;
    const IO* K = (const IO*)p.K + r.bh * p.N * D;
    const IO* V = (const IO*)p.V + r.bh * p.N * M;
    const IO* G = (const IO*)p.G + r.bh * p.N * M;
    IO* dK = (IO*)p.dK + r.bh * p.N * D;
    IO* dV = (IO*)p.dV + r.bh * p.N * M;
    const float* dn = p.aux + r.bh * 2 * p.N;
    const float* delta = dn + p.N;

    State<DP, MP> st;           // record i is the sum of piece i + 1
    st.init(p, p.S0 ? p.S0 + r.bh * D * M : nullptr, p.Z0 ? p.Z0 + r.bh * D : nullptr,
            p.rec + (r.bh * (p.pieces - 1) + r.piece) * (int64_t)(D * M + D), p.pieces - 1 - r.piece);
    const int64_t chunks = (r.end - r.lo + T - 1) / T;
    for (int64_t c = chunks - 1; c >= 0; --c) {
        const uint32_t sQ = smem_u32(buf + Sh::X), sG = smem_u32(buf + Sh::Y), sR = smem_u32(buf + Sh::S);
        float* sr = reinterpret_cast<float*>(buf + Sh::Z);
        float* sdl = reinterpret_cast<float*>(buf + Sh::W);
        uint16_t* wpl = reinterpret_cast<uint16_t*>(buf + Sh::WP);
        const int64_t n0 = r.lo + c * T;
        const int cn = (int)(r.end - n0 < T ? r.end - n0 : T), blocks = (cn + 15) / 16;
        const int strip = (c & 1) ? WARPS - 1 - warp : warp, row0 = strip * 16;
        {
            ReverseRows<IO, DP, MP> rr;
            rr.load(Q, G, dn, delta, n0, cn, D, M, pad);
            if constexpr (C::BUF == 1) __syncthreads();
            st.template publish<NS>(buf + Sh::S, sr);
            rr.template store<NR, NV>(buf + Sh::X, buf + Sh::Y, sdl, wpl, phi);
        }
        if (c > 0) {
            prefetch_rows(Q, n0 - T, r.end, D);
            prefetch_rows(K, n0 - T, r.end, D);
            prefetch_rows(V, n0 - T, r.end, M);
            prefetch_rows(G, n0 - T, r.end, M);
        }
        __syncthreads();
        if (row0 < cn) {
            {
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
                            uint32_t b[NR][4];
                            load_rows<NR, DP>(b, sQ, T * DP * 2, ib * 16, kk * 2, lane);
                            c.step<NQ, NR>(ka[kk], b);
                        }
                        c.put(s0, s1);
                    }
                    if (ib == strip) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int row = g + (j >> 1) * 8, col = 2 * t + (j & 1);
                            if (col < row) s0[j] = 0.f;
                            if (col + 8 < row) s1[j] = 0.f;
                        }
                    }
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
            {
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
                    if (ib == strip) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int row = g + (j >> 1) * 8, col = 2 * t + (j & 1);
                            if (col < row) s0[j] = 0.f;
                            if (col + 8 < row) s1[j] = 0.f;
                        }
                    }
                    uint32_t pa[NP][4];
                    operand_of<NP>(pa, s0, s1);
#pragma unroll
                    for (int n = 0; n < DP / 16; ++n) {
                        uint32_t b[NR][4];
                        load_cols_t<NR, DP>(b, sQ, T * DP * 2, ib * 16, n * 2, lane);
                        block_mma<NP, NR>(gk[2 * n], gk[2 * n + 1], pa, b);
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
        }
        st.template update<NR, NV, false>(sQ, sG, wpl);
        flip<C, Sh>(buf, smem);
    }
    zero_rows(dK, r.end, r.hi, D);
    zero_rows(dV, r.end, r.hi, M);
    if (r.piece == 0) st.write(p, p.S1 ? p.S1 + r.bh * D * M : nullptr, p.Z1 ? p.Z1 + r.bh * D : nullptr);
}

// ---- host ------------------------------------------------------------------------------------------------------
struct Plan { int pieces; int64_t len; };

// Pieces per sequence, by the estimated time in units of one chunk of a main kernel (about 10 us alone on an SM).
// An SM runs two CTAs in 1.25 times the time of one; a CTA's start costs about a chunk, and 0.35 for each record it
// sums, of which it has half of them on average; the pre-pass does 0.35 of a main kernel's work per chunk.  Forward +
// backward in us, fp32, D = M = 64, pieces 1 / 2 / 4 / 8 / 16: B1 H8 N1024 466 / 304 / 172 / 123 / 134;
// B8 H8 N1024 484 / 324 / 245 / 287 / 381; B16 H8 N2048 963 / 815 / 929 / 913 / 1091;
// B32 H8 N4096 2632 / 3318 / 3219 / 3215 / 3645.
Plan choose_plan(const la_problem& p, bool single) {
    const int64_t chunks = (p.N + T - 1) / T, bh = p.B * p.H;
    int64_t best = 1;
    const int forced = tc::causal_pieces_override();
    if (single) {
        best = 1;
    } else if (forced > 0) {
        best = forced < chunks ? forced : chunks;
        if (best > 1024) best = 1024;
    } else {
        auto waves = [](int64_t ctas) {
            const int64_t sm = (ctas + 147) / 148;
            return 1.25 * (double)(sm / 2) + (double)(sm % 2);
        };
        auto cost = [&](int64_t n) {
            const double per = (double)((chunks + n - 1) / n);
            return (per + 1.0 + 0.175 * (n - 1)) * waves(bh * n) + (n > 1 ? 0.35 * (per + 1.0) * waves(bh * (n - 1)) : 0.0);
        };
        for (int64_t n = 2; n <= 16 && n <= chunks; ++n)
            if (cost(n) < cost(best)) best = n;
    }
    const int64_t len = (chunks + best - 1) / best * T;
    return Plan{(int)((p.N + len - 1) / len), len};
}

size_t record_bytes(const la_problem& p, const Plan& pl) {
    return (size_t)(p.B * p.H) * (size_t)(pl.pieces - 1) * (size_t)(p.D * p.M + p.D) * sizeof(float);
}
size_t aux_bytes(const la_problem& p) { return ((size_t)(p.B * p.H) * (size_t)p.N * 2 * sizeof(float) + 15) & ~(size_t)15; }

Params make_params(const la_problem& p, const Plan& pl, const int* lengths) {
    Params a = {};
    a.lengths = lengths;
    a.N = p.N; a.piece_len = pl.len; a.pieces = pl.pieces;
    a.heads = (int)p.H; a.D = (int)p.D; a.M = (int)p.M; a.phi = p.phi; a.eps = p.eps;
    return a;
}

int launch(void (*kern)(const Params), unsigned bh, unsigned y, int smem, const Params& a, cudaStream_t st) {
    if (smem > 48 * 1024) LA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    kern<<<dim3(bh, y), THREADS, smem, st>>>(a);
    LA_LAUNCHED();
    return LA_OK;
}

template <typename C, int DP, int MP, bool EXACT> struct Kernels {
    using Fwd = Shared<DP, MP, C::NQ, C::NV, C::NS>;
    using Rev = Shared<DP, MP, C::NR, C::NV, C::NS>;
    static int sums(const la_problem& p, const Params& a, bool reverse, cudaStream_t st) {
        if (a.pieces == 1) return LA_OK;
        const unsigned bh = (unsigned)(p.B * p.H), y = (unsigned)(a.pieces - 1);
        constexpr int vec = T * 4 + 3 * T * 2;
        if (reverse) return launch(causal_mma_sum_kernel<C, DP, MP, EXACT, true>, bh, y, C::BUF == 2 ? 2 * Rev::BYTES : Rev::S + vec, a, st);
        return launch(causal_mma_sum_kernel<C, DP, MP, EXACT, false>, bh, y, C::BUF == 2 ? 2 * Fwd::BYTES : Fwd::S + vec, a, st);
    }
    static int forward(const la_problem& p, const Params& a, cudaStream_t st) {
        if (int rc = sums(p, a, false, st)) return rc;
        return launch(causal_mma_forward_kernel<C, DP, MP, EXACT>, (unsigned)(p.B * p.H), (unsigned)a.pieces, C::BUF * Fwd::BYTES, a, st);
    }
    static int backward(const la_problem& p, const Params& fwd, const Params& rev, cudaStream_t st) {
        if (int rc = sums(p, fwd, false, st)) return rc;
        if (int rc = launch(causal_mma_dq_kernel<C, DP, MP, EXACT>, (unsigned)(p.B * p.H), (unsigned)fwd.pieces, C::BUF * Fwd::BYTES, fwd, st))
            return rc;
        if (int rc = sums(p, rev, true, st)) return rc;
        return launch(causal_mma_dkv_kernel<C, DP, MP, EXACT>, (unsigned)(p.B * p.H), (unsigned)rev.pieces, C::BUF * Rev::BYTES, rev, st);
    }
};

// Tiles are padded to 32, 64 or (D) 128 columns; EXACT: D and M are those sizes.
template <typename F> int dispatch(const la_problem& p, F f) {
    const bool exact = (p.D == 32 || p.D == 64 || p.D == 128) && p.M == (p.D == 32 ? 32 : 64);
    if (p.dtype == LA_F32) {
        if (p.D <= 32 && p.M <= 32) return exact ? f(Kernels<Fp32, 32, 32, true>()) : f(Kernels<Fp32, 32, 32, false>());
        if (p.D <= 64) return exact ? f(Kernels<Fp32, 64, 64, true>()) : f(Kernels<Fp32, 64, 64, false>());
        return f(Kernels<Fp32, 128, 64, false>());
    }
    if (p.D == 32 && p.M == 32) return f(Kernels<Bf16, 32, 32, true>());
    if (p.phi == LA_PHI_IDENTITY) {
        if (p.D <= 64) return f(Kernels<Bf16Features, 64, 64, false>());
        return exact ? f(Kernels<Bf16Features, 128, 64, true>()) : f(Kernels<Bf16Features, 128, 64, false>());
    }
    return p.D <= 64 ? f(Kernels<Bf16Wide, 64, 64, false>()) : f(Kernels<Bf16Wide, 128, 64, false>());
}

}  // namespace

bool causal_mma_supported(const la_problem& p) {
    static const bool disabled = getenv("LA_DISABLE_TC") != nullptr;
    return !disabled && p.M <= 64;
}

// bf16, D = M = 32, many short sequences: the tcgen05 kernels run one CTA per SM and start up for about three chunks of
// 128 positions in every sequence, and handle 128 scores per row where D is 32.  Forward + backward, us, tcgen05 /
// mma.sync: 1024 heads N 784 373 / 287, 2048 x 300 442 / 234, 512 x 512 131 / 102, 512 x 1024 212 / 192; but
// 512 x 2048 367 / 372, 256 x 512 66 / 70, 128 x 3072 138 / 195.  (D = M = 64: 512 x 512 161 / 265.)
bool causal_mma_preferred(const la_problem& p) {
    return p.dtype == LA_BF16 && p.D == 32 && p.M == 32 && p.B * p.H >= 3 * 148 && p.N <= 1024;
}

size_t causal_mma_workspace(const la_problem& p, bool backward) {
    const size_t rec = record_bytes(p, choose_plan(p, false));
    return backward ? aux_bytes(p) + rec : rec;
}

int causal_mma_forward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const float* S_in,
                       const float* Z_in, void* O, float* den, float* S_out, float* Z_out, void* ws, size_t ws_bytes, cudaStream_t st) {
    Plan pl = choose_plan(p, false);
    if (!ws || !aligned16(ws) || ws_bytes < record_bytes(p, pl)) pl = choose_plan(p, true);       // no room for records: one piece per sequence
    Params a = make_params(p, pl, lengths);
    a.Q = Q; a.K = K; a.V = V; a.O = O; a.den = den;
    a.S0 = S_in; a.Z0 = Z_in; a.S1 = S_out; a.Z1 = Z_out;
    a.rec = (float*)ws;
    return dispatch(p, [&](auto k) { return decltype(k)::forward(p, a, st); });
}

int causal_mma_backward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const void* G,
                        const StateArgs& sa, void* dQ, void* dK, void* dV, void* ws, cudaStream_t st) {
    const Plan pl = choose_plan(p, false);
    Params f = make_params(p, pl, lengths);
    f.Q = Q; f.K = K; f.V = V; f.G = G; f.dQ = dQ; f.dK = dK; f.dV = dV;
    f.aux = (float*)ws;
    f.rec = (float*)((char*)ws + aux_bytes(p));
    Params r = f;
    f.S0 = sa.S_in; f.Z0 = sa.Z_in;
    r.S0 = sa.dS_out; r.Z0 = sa.dZ_out; r.S1 = sa.dS_in; r.Z1 = sa.dZ_in;
    return dispatch(p, [&](auto k) { return decltype(k)::backward(p, f, r, st); });
}

}  // namespace la
