// conv_tc.h -- tensor-core 3x3 convolutions of the learned correction,
// internal to the library.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace mgk {

// what a convolution does with its accumulators
enum ConvEpilogue {
    kHidden,    // + bias, ReLU, BF16 C8 into out
    kResidual,  // + bias, pixel shuffle, times s_out: written to, or added to, res
    kLoss,      // + bias, the loss against target - Pi_F(dC) and its gradient (split) into out
    kBackward   // ReLU mask of the layer's input, the gradient (split) into out
};

struct ConvArgs {
    int n = 0;
    int *status = nullptr;                // a wait that expires records MGENKF_ERR_TIMEOUT here (may be NULL)
    const __nv_bfloat16 *in = nullptr;    // BF16 C8 (split q at in + q in_split)
    size_t in_split = 0;
    const __nv_bfloat16 *wp = nullptr;    // packed weights [9][groups][COUT][8]
    const float *bias = nullptr;
    const float *dC = nullptr, *xs = nullptr;  // the fields (first layer, kLoss)
    const float *stats = nullptr;         // mu_in[8], s_in[8], s_out[4]
    __nv_bfloat16 *a0 = nullptr;          // first layer: the normalised fields, BF16 C8 (NULL: not kept)
    __nv_bfloat16 *out = nullptr;         // BF16 C8 (split q at out + q out_split)
    size_t out_split = 0;
    float *res = nullptr;
    int accumulate = 0;
    bool wide = false;                    // res (target) starts on a 16-byte boundary
    const float *target = nullptr;
    float *loss_part = nullptr;           // one partial per CTA (conv_loss_parts)
    float inv_count = 0.f;
    float pw[16] = {};                    // Lagrange weights of fine offset m at 4 m + t
    const __nv_bfloat16 *mask = nullptr;  // BF16 C8
};

// elements of the packed weights of one CIN -> COUT layer ([9][groups][COUT][8])
int conv_packed_elems(int cin, int cout);
// 3x3 periodic convolution of `batch` n x n maps; CG: input channel groups of
// 8 (1: the normalised fields), NSPLIT: 3 if the input is a split gradient
template <int CG, int NSPLIT, int COUT, int EPI>
cudaError_t launch_conv_tc(const ConvArgs &A, int batch, cudaStream_t s);
int conv_loss_parts(int n, int batch);
// partial weight gradients, part[unit][t][o][i] and db[o], of d (split, COUT
// channels) against in (8 CGI channels)
template <int CGI, int COUT>
cudaError_t launch_conv_wgrad(const __nv_bfloat16 *in, const __nv_bfloat16 *d, size_t d_split, int n, int batch,
                              float *part, int *status, cudaStream_t s);
int wgrad_units(int n, int batch);

}  // namespace mgk
