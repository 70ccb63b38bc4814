// Host launchers of the surrogate's tcgen05 kernels (pd_mlp_tc.cu).
#pragma once

#include "pd_internal.cuh"

// Training forward: the same kernel also stores Z[l] (BF16 [rows x pad[l+1]], hidden
// layers) and HT[l] (BF16 [pad[l] x ldT], every layer's input transposed), and turns the
// output into the loss (one partial sum a CTA, mlp_forward_tc's return value many) and its
// gradient dY, dYT instead of storing it.  Hidden widths must be multiples of 32.
struct MlpTrain {
    void *const *Z, *const *HT;
    int64_t ldT;
    const float *T;
    float scale;
    void *dY, *dYT;
    float *lpart;
};
// Forward of an MLP whose layers all fit the fused kernel (K, N <= 256): W[l] padded BF16
// weights [pad[l+1] x pad[l]] row-major, bias[l] pad[l+1] floats; tr == nullptr: inference into Y.  Returns the number of CTAs, or -1 (unsupported, nothing launched).
int mlp_forward_tc(int L, const int *dims, const int *pad, void *const *W, const float *const *bias, const float *X,
                   int64_t rows, float *Y, const MlpTrain *tr, unsigned *err, int device, cudaStream_t st);
// The data gradients of a training step: dZT[l] [pad[l+1] x ldT] for the hidden layers l =
// L-2 .. 0 from tr->dY and tr->Z; WT[l]: transposed weights [pad[l] x pad[l+1]].  Returns a
// negative number if it cannot run.
int mlp_backward_tc(int L, const int *pad, void *const *WT, const MlpTrain *tr, void *const *dZT, int64_t rows,
                    unsigned *err, int device, cudaStream_t st);
// Number of splits of the batch that mlp_dw_tc takes.
int mlp_dw_splits(int L, const int *pad, int64_t rows, int device);
// Split-K partials of every layer's dW = dZ^T H and bias gradient dZ^T 1: dZT[l] [pad[l+1] x
// rows], HT[l] [pad[l] x rows] (ld ldT); part[l] [splits x pad[l+1] x pad[l]], partb[l]
// [splits x pad[l+1]], FP32.
int mlp_dw_tc(int L, const int *pad, void *const *dZT, void *const *HT, int64_t rows, int64_t ldT, float *const *part,
              float *const *partb, unsigned *err, int device, cudaStream_t st);
