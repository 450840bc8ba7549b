// cnn.cu -- learned correction of the prolongation (residual CNN over Pi_F).
//
// Network: the 8 coarse channels [dC, x^C*] (normalised with fixed per-channel
// mean and scale) go through three 3x3 convolutions with periodic padding,
// 8 -> 32 -> 32 -> 64 channels, ReLU after the first two; the 64 output
// channels are pixel-shuffled by 4 into 4 fine channels, scaled per channel,
// and added to Pi_F(dC):
//   dF = Pi_F(dC) + s_out[c] * z3[16 c + 4 sy + sx][y][x]   at fine (4y + sy, 4x + sx).
// Training minimises mean(((dF - target) / s_out)^2) with Adam on FP32 master
// weights; the forward and backward passes use BF16 weights and activations
// with FP32 accumulation.
//
// Activations a0 (8 channels), a1, a2 (32) are BF16 in channel groups of 8
// ("C8": element (b, i, p) at ((b C/8 + i/8) n^2 + p) 8 + i % 8); the
// gradients with respect to the layers' outputs are FP32 values held as three
// BF16 maps in that layout (conv_tc.cu).
//
// One training step is nine launches (conv_tc.cu): the three forward
// convolutions, the first normalising the fields, the last going straight
// from its accumulators through the pixel shuffle to the loss and dz3 (z3 is
// never stored); per layer the partial weight gradients and, above the first,
// the adjoint convolution; and
//   k_reduce_grads  the partial sums in unit order, and the loss
//   k_adam          Adam step on FP32 master weights; writes the packed
//                   tensor-core copies of the weights
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <string>
#include <vector>

#include "../../include/mgenkf_ops.h"
#include "analysis.h"
#include "common.cuh"
#include "conv_tc.h"

namespace mgk {

constexpr int kCnnParams = 32 * 8 * 9 + 32 + 32 * 32 * 9 + 32 + 64 * 32 * 9 + 64;  // 30080

struct CnnLayer {
    int cin, cout;
    size_t w_off, b_off;  // offsets into the parameter vector
};
static const CnnLayer kLayers[3] = {{8, 32, 0, 2304}, {32, 32, 2336, 11552}, {32, 64, 11584, 30016}};

// where the packed copies of parameter e live: the forward operand
// [tap][group of i][o][i % 8] and, above the first layer, the adjoint's
// [8 - tap][group of o][i][o % 8]; -1 for a bias / for none
struct PackedAt {
    int fwd, adj;
};
constexpr int kFwdOff[3] = {0, 9 * 2 * 32 * 8, 9 * (2 + 4) * 32 * 8};
constexpr int kAdjOff[3] = {0, 0, 9 * 4 * 32 * 8};
constexpr int kFwdElems = kFwdOff[2] + 9 * 4 * 64 * 8, kAdjElems = kAdjOff[2] + 9 * 8 * 32 * 8;
__device__ __forceinline__ PackedAt packed_at(int e) {
    int l, cin, cout;
    if (e < 2304) {
        l = 0, cin = 8, cout = 32;
    } else if (e >= 2336 && e < 11552) {
        l = 1, cin = 32, cout = 32, e -= 2336;
    } else if (e >= 11584 && e < 30016) {
        l = 2, cin = 32, cout = 64, e -= 11584;
    } else {
        return {-1, -1};
    }
    const int t = e % 9, i = (e / 9) % cin, o = e / (9 * cin);
    const int cgk = cin < 16 ? 2 : cin / 8;
    constexpr int f1 = kFwdOff[1], f2 = kFwdOff[2], a2 = kAdjOff[2];
    const int fo = l == 0 ? 0 : l == 1 ? f1 : f2, ao = l == 2 ? a2 : 0;
    return {fo + ((t * cgk + i / 8) * cout + o) * 8 + i % 8,
            l == 0 ? -1 : ao + (((8 - t) * (cout / 8) + o / 8) * cin + i) * 8 + o % 8};
}

__global__ void k_pack_weights(const float *__restrict__ w, __nv_bfloat16 *__restrict__ fwd,
                               __nv_bfloat16 *__restrict__ adj) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < kCnnParams; e += gridDim.x * blockDim.x) {
        const PackedAt at = packed_at(e);
        if (at.fwd >= 0) fwd[at.fwd] = __float2bfloat16(w[e]);
        if (at.adj >= 0) adj[at.adj] = __float2bfloat16(w[e]);
    }
}

// Gradients: the partials part[unit][t][o][i], db[o] of the three layers summed
// over the units.  A CTA takes 32 consecutive elements (coalesced reads), a
// quarter of the units per group of 32 threads, added in a fixed order; the
// last CTA sums the loss partials.
struct GradParts {
    const float *part[3];
    const float *loss_part;
    float *loss;
    int units, loss_parts;
};
__global__ void __launch_bounds__(128) k_reduce_grads(GradParts P, float *__restrict__ g, const int *status) {
    launch_wait();
    if (*status) return;
    __shared__ float red[128];
    const int tid = threadIdx.x, lane = tid & 31, q = tid >> 5;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    if (blockIdx.x + 1 == gridDim.x) {
        int u = tid;
        for (; u + 3 * 128 < P.loss_parts; u += 4 * 128)
#pragma unroll
            for (int h = 0; h < 4; ++h) s[h] += P.loss_part[u + 128 * h];
        for (; u < P.loss_parts; u += 128) s[0] += P.loss_part[u];
        red[tid] = (s[0] + s[1]) + (s[2] + s[3]);
        __syncthreads();
        for (int h = 64; h > 0; h >>= 1) {
            if (tid < h) red[tid] += red[tid + h];
            __syncthreads();
        }
        if (tid == 0) *P.loss = red[0];
        return;
    }
    // 30080 = 940 x 32, and no 32 elements straddle two layers
    const int e = blockIdx.x * 32 + lane;
    const int l = e < 2336 ? 0 : e < 11584 ? 1 : 2, first = l == 0 ? 0 : l == 1 ? 2336 : 11584;
    const int cin = l == 0 ? 8 : 32, cout = l == 2 ? 64 : 32, k = e - first;
    const int nw = 9 * cin * cout, len = nw + cout;
    const float *p = (l == 0 ? P.part[0] : l == 1 ? P.part[1] : P.part[2]) + k;
    int u = q;
    for (; u + 12 < P.units; u += 16)
#pragma unroll
        for (int h = 0; h < 4; ++h) s[h] += p[(size_t)(u + 4 * h) * len];
    for (; u < P.units; u += 4) s[0] += p[(size_t)u * len];
    red[tid] = (s[0] + s[1]) + (s[2] + s[3]);
    __syncthreads();
    if (q) return;
    // (t, o, i) -> (o, i, t)
    const int to = first + (k < nw ? (k % (cin * cout)) * 9 + k / (cin * cout) : k);
    g[to] = (red[lane] + red[lane + 32]) + (red[lane + 64] + red[lane + 96]);
}

__global__ void k_adam(float *__restrict__ w, float *__restrict__ m, float *__restrict__ v,
                       const float *__restrict__ g, __nv_bfloat16 *__restrict__ fwd, __nv_bfloat16 *__restrict__ adj,
                       float lr, float b1, float b2, float eps, float c1, float c2) {
    launch_wait();
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < kCnnParams; e += gridDim.x * blockDim.x) {
        const float gi = g[e];
        const float mi = b1 * m[e] + (1.f - b1) * gi;
        const float vi = b2 * v[e] + (1.f - b2) * gi * gi;
        m[e] = mi;
        v[e] = vi;
        const float wi = w[e] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        w[e] = wi;
        const PackedAt at = packed_at(e);
        if (at.fwd >= 0) fwd[at.fwd] = __float2bfloat16(wi);
        if (at.adj >= 0) adj[at.adj] = __float2bfloat16(wi);
    }
}

}  // namespace mgk

// ===========================================================================
// C ABI: the learned-correction object
// ===========================================================================
using namespace mgk;

struct mgk_cnn {
    int nc, bmax;
    float *w = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;  // FP32 master, Adam, grads
    float *stats = nullptr;  // mu_in[8], s_in[8], s_out[4]
    __nv_bfloat16 *a0 = nullptr, *a1 = nullptr, *a2 = nullptr;
    __nv_bfloat16 *d3 = nullptr, *d2 = nullptr, *d1 = nullptr;  // gradients of the layers' outputs, three splits each
    float *part = nullptr, *loss_part = nullptr, *loss = nullptr;
    __nv_bfloat16 *fwd = nullptr, *adj = nullptr;  // tensor-core copies of the weights (packed_at)
    int *status = nullptr;       // MGENKF_ERR_TIMEOUT from a tensor-core wait, sticky
    int step = 0;
    std::string err;
};

static void cnn_free(mgk_cnn *c) {
    void *ptrs[] = {c->w, c->m, c->v, c->g, c->stats, c->a0, c->a1, c->a2, c->d3, c->d2,
                    c->d1, c->part, c->loss_part, c->loss, c->fwd, c->adj, c->status};
    for (void *p : ptrs)
        if (p) cudaFree(p);
}

extern "C" mgenkf_status mgk_cnn_create(int32_t n_coarse, int32_t batch_max, mgk_cnn_t *out) {
    if (!out) return MGENKF_ERR_INVALID_ARG;
    *out = nullptr;
    if (n_coarse < 1 || n_coarse > 1024 || batch_max < 1 || batch_max > 256) {
        mgk_set_error("mgk_cnn_create: n_coarse must be in [1, 1024] and batch_max in [1, 256]");
        return MGENKF_ERR_INVALID_ARG;
    }
    mgk_cnn *c = new mgk_cnn();
    c->nc = n_coarse;
    c->bmax = batch_max;
    const size_t pl = (size_t)n_coarse * n_coarse, B = batch_max;
    // the partial sums of any batch up to batch_max
    size_t units = 0, ctas = 0;
    for (int q = 1; q <= batch_max; ++q) {
        units = std::max(units, (size_t)wgrad_units(n_coarse, q));
        ctas = std::max(ctas, (size_t)conv_loss_parts(n_coarse, q));
    }
    struct A {
        void **p;
        size_t bytes;
    } allocs[] = {
        {(void **)&c->w, kCnnParams * sizeof(float)},   {(void **)&c->m, kCnnParams * sizeof(float)},
        {(void **)&c->v, kCnnParams * sizeof(float)},   {(void **)&c->g, kCnnParams * sizeof(float)},
        {(void **)&c->stats, 20 * sizeof(float)},       {(void **)&c->a0, B * 8 * pl * 2},
        {(void **)&c->a1, B * 32 * pl * 2},             {(void **)&c->a2, B * 32 * pl * 2},
        {(void **)&c->d3, B * 64 * pl * 6},             {(void **)&c->d2, B * 32 * pl * 6},
        {(void **)&c->d1, B * 32 * pl * 6},             {(void **)&c->part, units * kCnnParams * sizeof(float)},
        {(void **)&c->loss_part, ctas * sizeof(float)}, {(void **)&c->loss, sizeof(float)},
        {(void **)&c->fwd, kFwdElems * 2},              {(void **)&c->adj, kAdjElems * 2},
        {(void **)&c->status, sizeof(int)},
    };
    for (auto &a : allocs) {
        if (cudaMalloc(a.p, a.bytes) != cudaSuccess) {
            cudaGetLastError();
            mgk_set_error("mgk_cnn_create: device allocation failed");
            cnn_free(c);
            delete c;
            return MGENKF_ERR_OOM;
        }
    }
    cudaMemset(c->w, 0, kCnnParams * sizeof(float));
    cudaMemset(c->m, 0, kCnnParams * sizeof(float));
    cudaMemset(c->v, 0, kCnnParams * sizeof(float));
    cudaMemset(c->status, 0, sizeof(int));
    cudaMemset(c->fwd, 0, kFwdElems * 2);  // the K padding of the first layer stays zero
    cudaMemset(c->adj, 0, kAdjElems * 2);
    const float st[20] = {0, 0, 0, 0, 0, 0, 0, 0, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1};
    cudaMemcpy(c->stats, st, sizeof(st), cudaMemcpyHostToDevice);
    if (cudaDeviceSynchronize() != cudaSuccess) {
        mgk_set_error("mgk_cnn_create: CUDA error during set-up");
        cnn_free(c);
        delete c;
        return MGENKF_ERR_CUDA;
    }
    *out = c;
    return MGENKF_OK;
}

extern "C" int32_t mgk_cnn_coarse_size(mgk_cnn_t c) { return c ? c->nc : 0; }

extern "C" mgenkf_status mgk_cnn_destroy(mgk_cnn_t c) {
    if (!c) return MGENKF_OK;
    cudaDeviceSynchronize();
    cnn_free(c);
    delete c;
    return MGENKF_OK;
}

extern "C" mgenkf_status mgk_cnn_set_params(mgk_cnn_t c, const float *params, const float *stats) {
    if (!c) return MGENKF_ERR_INVALID_ARG;
    if (params) {
        if (cudaMemcpy(c->w, params, kCnnParams * sizeof(float), cudaMemcpyDefault) != cudaSuccess) return MGENKF_ERR_CUDA;
        cudaMemset(c->m, 0, kCnnParams * sizeof(float));
        cudaMemset(c->v, 0, kCnnParams * sizeof(float));
        c->step = 0;
        count_launches(1);
        k_pack_weights<<<118, 256>>>(c->w, c->fwd, c->adj);
    }
    if (stats && cudaMemcpy(c->stats, stats, 20 * sizeof(float), cudaMemcpyDefault) != cudaSuccess)
        return MGENKF_ERR_CUDA;
    return cudaDeviceSynchronize() == cudaSuccess ? MGENKF_OK : MGENKF_ERR_CUDA;
}

extern "C" mgenkf_status mgk_cnn_get_params(mgk_cnn_t c, float *params, float *grads) {
    if (!c) return MGENKF_ERR_INVALID_ARG;
    if (cudaDeviceSynchronize() != cudaSuccess) return MGENKF_ERR_CUDA;  // training launches on any stream
    int st = 0;
    if (cudaMemcpy(&st, c->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return MGENKF_ERR_CUDA;
    if (st) {
        mgk_set_error("mgk_cnn: a tensor-core wait expired in an earlier call");
        return (mgenkf_status)st;
    }
    if (params && cudaMemcpy(params, c->w, kCnnParams * sizeof(float), cudaMemcpyDefault) != cudaSuccess)
        return MGENKF_ERR_CUDA;
    if (grads && cudaMemcpy(grads, c->g, kCnnParams * sizeof(float), cudaMemcpyDefault) != cudaSuccess)
        return MGENKF_ERR_CUDA;
    return MGENKF_OK;
}

// the hidden layers of B samples: a1, a2 (and a0 if `keep`)
static void cnn_hidden(mgk_cnn *c, const float *dC, const float *xs, int B, bool keep, int *status, cudaStream_t s) {
    ConvArgs A;
    A.n = c->nc;
    A.status = status;
    A.stats = c->stats;
    A.dC = dC;
    A.xs = xs;
    A.a0 = keep ? c->a0 : nullptr;
    A.wp = c->fwd + kFwdOff[0];
    A.bias = c->w + kLayers[0].b_off;
    A.out = c->a1;
    launch_conv_tc<1, 1, 32, kHidden>(A, B, s);
    A.in = c->a1;
    A.wp = c->fwd + kFwdOff[1];
    A.bias = c->w + kLayers[1].b_off;
    A.out = c->a2;
    launch_conv_tc<4, 1, 32, kHidden>(A, B, s);
}

// the last layer's arguments
static ConvArgs cnn_last(mgk_cnn *c, int *status) {
    ConvArgs A;
    A.n = c->nc;
    A.status = status;
    A.stats = c->stats;
    A.in = c->a2;
    A.wp = c->fwd + kFwdOff[2];
    A.bias = c->w + kLayers[2].b_off;
    return A;
}

namespace mgk {
mgenkf_status cnn_forward_status(mgk_cnn_t c, const float *dC, const float *xstar, int batch, float *residual,
                                 int accumulate, int *status, cudaStream_t s) {
    if (!c || !dC || !xstar || !residual || batch < 1 || batch > c->bmax) return MGENKF_ERR_INVALID_ARG;
    cnn_hidden(c, dC, xstar, batch, false, status, s);
    ConvArgs A = cnn_last(c, status);
    A.res = residual;
    A.accumulate = accumulate;
    A.wide = (reinterpret_cast<uintptr_t>(residual) & 15) == 0;
    launch_conv_tc<4, 1, 64, kResidual>(A, batch, s);
    return cudaGetLastError() == cudaSuccess ? MGENKF_OK : MGENKF_ERR_CUDA;
}
}  // namespace mgk

extern "C" mgenkf_status mgk_cnn_forward(mgk_cnn_t c, const float *dC, const float *xstar, int32_t batch,
                                         float *residual, int32_t accumulate, void *stream) {
    if (!c) return MGENKF_ERR_INVALID_ARG;
    return cnn_forward_status(c, dC, xstar, batch, residual, accumulate, c->status, (cudaStream_t)stream);
}

extern "C" mgenkf_status mgk_cnn_loss_grad(mgk_cnn_t c, const float *dC, const float *xstar, const float *target,
                                           int32_t batch, float *loss_out, void *stream) {
    if (!c || !dC || !xstar || !target || batch < 1 || batch > c->bmax) return MGENKF_ERR_INVALID_ARG;
    const cudaStream_t s = (cudaStream_t)stream;
    const int n = c->nc, B = batch;
    const size_t pl = (size_t)n * n, s3 = (size_t)B * 64 * pl, s2 = (size_t)B * 32 * pl;  // elements of one split
    cnn_hidden(c, dC, xstar, B, true, c->status, s);
    ConvArgs A = cnn_last(c, c->status);
    A.dC = dC;
    A.target = target;
    A.wide = (reinterpret_cast<uintptr_t>(target) & 15) == 0;
    A.loss_part = c->loss_part;
    A.inv_count = 1.f / (float)((size_t)B * 4 * 16 * pl);
    for (int m = 0; m < 4; ++m) {
        const double sv = m / 4.0;
        A.pw[4 * m + 0] = (float)(-sv * (sv - 1.0) * (sv - 2.0) / 6.0);
        A.pw[4 * m + 1] = (float)((sv + 1.0) * (sv - 1.0) * (sv - 2.0) / 2.0);
        A.pw[4 * m + 2] = (float)(-(sv + 1.0) * sv * (sv - 2.0) / 2.0);
        A.pw[4 * m + 3] = (float)((sv + 1.0) * sv * (sv - 1.0) / 6.0);
    }
    A.out = c->d3;
    A.out_split = s3;
    launch_conv_tc<4, 1, 64, kLoss>(A, B, s);
    const int units = wgrad_units(n, B);
    float *part[3] = {c->part, c->part + (size_t)units * 2336, c->part + (size_t)units * 11584};
    // layer 3: dW3, db3, and the gradient of z2, masked by a2 > 0
    launch_conv_wgrad<4, 64>(c->a2, c->d3, s3, n, B, part[2], c->status, s);
    ConvArgs D;
    D.n = n;
    D.status = c->status;
    D.in = c->d3;
    D.in_split = s3;
    D.wp = c->adj + kAdjOff[2];
    D.mask = c->a2;
    D.out = c->d2;
    D.out_split = s2;
    launch_conv_tc<8, 3, 32, kBackward>(D, B, s);
    // layer 2
    launch_conv_wgrad<4, 32>(c->a1, c->d2, s2, n, B, part[1], c->status, s);
    D.in = c->d2;
    D.in_split = s2;
    D.wp = c->adj + kAdjOff[1];
    D.mask = c->a1;
    D.out = c->d1;
    launch_conv_tc<4, 3, 32, kBackward>(D, B, s);
    // layer 1 (no input gradient)
    launch_conv_wgrad<1, 32>(c->a0, c->d1, s2, n, B, part[0], c->status, s);
    const GradParts P{{part[0], part[1], part[2]}, c->loss_part, c->loss, units, conv_loss_parts(n, B)};
    count_launches(1);
    launch_kernel(k_reduce_grads, kCnnParams / 32 + 1, 128, 0, s, LaunchHow{}, P, c->g, c->status);
    if (loss_out) {
        if (cudaMemcpyAsync(loss_out, c->loss, sizeof(float), cudaMemcpyDefault, s) != cudaSuccess)
            return MGENKF_ERR_CUDA;
    }
    return cudaGetLastError() == cudaSuccess ? MGENKF_OK : MGENKF_ERR_CUDA;
}

extern "C" mgenkf_status mgk_cnn_adam_step(mgk_cnn_t c, float lr, void *stream) {
    if (!c || !(lr > 0.f)) return MGENKF_ERR_INVALID_ARG;
    c->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)c->step), c2 = 1.f - powf(b2, (float)c->step);
    count_launches(1);
    launch_kernel(k_adam, 118, 256, 0, (cudaStream_t)stream, LaunchHow{},
                  c->w, c->m, c->v, c->g, c->fwd, c->adj, lr, b1, b2, 1e-8f, c1, c2);
    return cudaGetLastError() == cudaSuccess ? MGENKF_OK : MGENKF_ERR_CUDA;
}
