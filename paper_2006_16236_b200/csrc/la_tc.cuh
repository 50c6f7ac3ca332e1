// Tensor-core (tcgen05 / TMA) kernels for bf16 problems: interface to the API layer.
#pragma once
#include "la_common.cuh"

namespace la {

// True when problem p / operation op runs on the tensor-core kernels.
bool tc_supported(const la_problem& p, int op);
size_t tc_workspace_bytes(const la_problem& p, int op);

// pieces, parts, piece_begin[], piece_first_part[], part_begin[], launch_order[] (see la_causal_plan)
int tc_causal_plan(const la_problem& p, int32_t* out, int capacity);

// Causal form on mma.sync (la_causal_mma.cu): at fp32 accuracy, M <= 64, any type and feature map; and bf16 problems with D = M = 32 by a
// warp per piece.  The forward's workspace is optional (without it a sequence is one piece) but for some of the latter.
bool causal_mma_supported(const la_problem& p);
bool causal_mma_preferred(const la_problem& p);      // of the problems that both kinds of kernels take
bool causal_mma_needs_workspace(const la_problem& p);
bool causal_mma_leaves_forward(const la_problem& p); // a forward pass that keeps no sums, of the latter: to the tcgen05 kernels
size_t causal_mma_workspace(const la_problem& p, bool backward);
size_t causal_mma_saved_bytes(const la_problem& p);  // what a forward pass leaves for the backward pass, or 0
int causal_mma_forward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const float* S_in,
                       const float* Z_in, void* O, float* den, float* S_out, float* Z_out, void* saved, void* ws, size_t ws_bytes, cudaStream_t st);
int causal_mma_backward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const void* G,
                        const StateArgs& sa, const void* saved, void* dQ, void* dK, void* dV, void* ws, cudaStream_t st);

// Non-causal form at fp32 accuracy on mma.sync (la_linear_mma.cu): M <= 64, any type and feature map; saved (or null):
// where the forward leaves its sums and the backward finds them.
bool linear_mma_supported(const la_problem& p);
size_t linear_mma_workspace(const la_problem& p, bool backward);
int linear_mma_forward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, void* O, float* den,
                       float* KV, float* Zs, void* saved, void* ws, cudaStream_t st);
int linear_mma_backward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const void* saved,
                        const void* G, void* dQ, void* dK, void* dV, void* ws, cudaStream_t st);

// Short sequences in one launch (la_cluster.cu): ahead of the other kernels where these say so, by the problem's size and by
// whether the context of the stream has room for such a cluster.  saved (or null): filled for the tcgen05 backward kernels,
// except where the size alone says that a cluster does the backward pass: no kernel reads the buffer there, also where the stream
// of the backward call turns out to have no room.
bool causal_cluster_forward_preferred(const la_problem& p, bool saved, bool state, cudaStream_t st);
bool causal_cluster_backward_size(const la_problem& p);
bool causal_cluster_backward_preferred(const la_problem& p, cudaStream_t st);
int causal_cluster_forward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const float* S_in,
                           const float* Z_in, void* O, float* den, float* S_out, float* Z_out, void* saved, cudaStream_t st);
int causal_cluster_backward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const void* G,
                            const StateArgs& sa, void* dQ, void* dK, void* dV, cudaStream_t st);
bool linear_cluster_preferred(const la_problem& p, cudaStream_t st);
int linear_cluster_forward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, void* O, float* den,
                           float* KV, float* Zs, void* saved, cudaStream_t st);

namespace tc {
// process-wide overrides of the automatic plans (see la_plan_override)
void set_plan_override(int causal_pieces, int causal_short, int linear_splits);
int causal_pieces_override();        // -1: automatic
int linear_splits_override();
// In all of these: lengths ([B] int32, device, or null) = real positions per batch element of a right-padded
// ragged batch; saved (or null) = where the forward leaves what the backward pass can reuse.
size_t causal_forward_workspace(const la_problem& p);
size_t causal_saved_bytes(const la_problem& p);
// the part of a saved buffer that a kernel of its own writes: the forward pre-pass's records
int causal_keep_records(const la_problem& p, const void* K, const void* V, const int* lengths, void* saved, cudaStream_t st);
int causal_forward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const float* S_in,
                   const float* Z_in, void* O, float* den, float* S_out, float* Z_out, void* saved, void* ws,
                   cudaStream_t st);
size_t causal_backward_workspace(const la_problem& p);
int causal_backward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, const void* G,
                    const StateArgs& sa, const void* saved, void* dQ, void* dK, void* dV, void* ws, cudaStream_t st);
size_t linear_forward_workspace(const la_problem& p);
size_t linear_backward_workspace(const la_problem& p);
int linear_keep_sums(const la_problem& p, const void* K, const void* V, const int* lengths, void* saved, cudaStream_t st);
int linear_forward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths, void* O,
                   float* den, float* KV, float* Zs, void* saved, void* ws, cudaStream_t st);
int linear_backward(const la_problem& p, const void* Q, const void* K, const void* V, const int* lengths,
                    const void* saved, const void* G, void* dQ, void* dK, void* dV, void* ws, cudaStream_t st);
// random Fourier features (la_rff.cu)
bool rff_supported(int64_t rows, int64_t D, int64_t C, int dtype);
int rff_forward(const void* x, const void* W, void* y, int64_t rows, int D, int C, cudaStream_t st);
int rff_backward(const void* x, const void* W, const void* dy, void* dx, int64_t rows, int D, int C, cudaStream_t st);
}  // namespace tc

}  // namespace la
