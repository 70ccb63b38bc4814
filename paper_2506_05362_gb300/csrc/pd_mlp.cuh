// Host launchers of the surrogate's tcgen05 kernels (pd_mlp_tc.cu).
#pragma once

#include "pd_internal.cuh"

// Training forward: the same kernel also stores Z[l] (BF16 [rows x pad[l+1]], hidden
// layers), HT[l] (BF16 [pad[l] x ldT], every layer's input transposed) and the output Y, and
// forms the gradient dY, dYT of the loss.  Hidden widths must be multiples of 32.
struct MlpTrain {
    void *const *Z, *const *HT;
    int64_t ldT;
    float *Y;
    const float *T;
    float scale;
    void *dY, *dYT;
    float *lpart;
    unsigned *next;  // task counter of mlp_dw_tc; the forward clears it
};
// Forward of an MLP whose layers all fit the fused kernel (K, N <= 256): W[l] padded BF16
// weights [pad[l+1] x pad[l]] row-major, bias[l] pad[l+1] floats; tr == nullptr: inference
// into Y.  Returns 0, or -1 (unsupported, nothing launched).
int mlp_forward_tc(int L, const int *dims, const int *pad, void *const *W, const float *const *bias, const float *X,
                   int64_t rows, float *Y, const MlpTrain *tr, unsigned *err, int device, cudaStream_t st);
// The data gradients of a training step: dZT[l] [pad[l+1] x ldT] for the hidden layers l =
// L-2 .. 0 from tr->dY and tr->Z; WT[l]: transposed weights [pad[l] x pad[l+1]].  Returns a
// negative number if it cannot run.
int mlp_backward_tc(int L, const int *pad, void *const *WT, const MlpTrain *tr, void *const *dZT, int64_t rows,
                    unsigned *err, int device, cudaStream_t st);
// Partial sums that mlp_dw_tc leaves of layer l's weight gradient: of at most 8 classes of
// splits, or of every split; kcs, splits (nullable): 64-row chunks per split, splits.
int mlp_dw_parts(int L, const int *pad, int l, int64_t rows, int device, int *kcs, int *splits);
// Sums of a training step over the batch: of every layer the partial weight gradients
// part[l] [parts x pad[l+1] x pad[l]] of dW = dZ^T H and the bias gradient gb[l]
// [dims[l+1]], and the nlp partial sums tr.lpart of (Y - T)^2, all FP32; dZT[l] [pad[l+1] x
// rows], HT[l] [pad[l] x rows] (ld tr.ldT).
int mlp_dw_tc(int L, const int *dims, const int *pad, void *const *dZT, void *const *HT, int64_t rows, const MlpTrain &tr,
              int nlp, float *const *part, float *const *gb, unsigned *err, int device, cudaStream_t st);
