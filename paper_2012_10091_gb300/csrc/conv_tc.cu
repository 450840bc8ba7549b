// conv_tc.cu -- the 3x3 periodic convolutions of the learned correction, forward
// and backward, on the tensor cores (tcgen05), as implicit GEMMs with no
// im2col copy.
//
// Activations are stored in channel groups of 8 ("C8"): element (b, i, p) of a
// C-channel n x n map sits at ((b C/8 + i/8) n^2 + p) 8 + i % 8, so the 8
// channels of one group at one pixel are 16 contiguous bytes.  Gradients are
// FP32 values held as three BF16 maps in that layout, x = hi + mid + lo: 24
// significand bits, so every product of a gradient with a BF16 weight or
// activation is exact in the tensor cores and sums in FP32, as on the FP32
// pipes before.
//
// k_conv_tc (forward layers and the adjoint convolutions): a CTA computes ROWS
// output rows x 128 pixels x COUT channels of one sample:
//   * the input block (ROWS + 2 rows x 130 pixels, periodic wrap) comes to
//     shared memory (a gradient 16 channels of one split at a time), one plane
//     per channel group with pixels 16 bytes apart.  That is the no-swizzle
//     K-major operand layout (a core matrix = 8 pixels x 8 channels = 128
//     contiguous bytes; the next 8 pixels 128 bytes on, the next 8 channels
//     one plane on), so the A operand of tap (dy, dx) for output row r is the
//     same planes with the start moved to pixel (r + dy, dx): nine taps, nine
//     start addresses, no copies;
//   * the packed weights [tap][group][COUT][8] are the B operands in the same
//     layout; the three splits of a gradient share them;
//   * one warp per output row issues the row's 9 MMAs per 16 channels (M = 128
//     pixels, N = COUT, K = 16) into its own TMEM columns; the next chunks are
//     copied while chunk c multiplies.  MMAs this small are bound by their
//     issue when one thread issues all of them (about 80 cycles each), hence
//     several warps, each with its descriptors in uniform registers (the last
//     layer's adjoint 185 -> 112 us);
//   * eight warps read the accumulators back and finish in registers: bias,
//     ReLU and BF16 C8 (hidden layers); the pixel shuffle into the residual,
//     or the loss and its gradient (last layer); the ReLU mask (backward).
//
// k_conv_wgrad (weight gradients): dW_t = sum over pixels of d[p] in[p + t],
// a GEMM whose K dimension is the pixels, with both operands MN-major in the
// same C8 rows (a core matrix = 8 pixels x 8 channels; the next 8 pixels 128
// bytes on, the next 8 channels one plane on): M = 128 = the splits of d
// stacked (their rows are added at the end), N = the input channels of one
// tap, all nine taps and the bias column (ones) in TMEM for the whole run of
// rows of a CTA.  Input rows live in a ring, so each is loaded once (two of eight
// twice, see WgradShape).  An MMA takes the three taps of one dx, the channel
// groups of three consecutive rows being evenly spaced: N = 96 instead of 32
// for the same 4 KB of A read from shared memory (32 cycles of the 54 an MMA of
// N = 32 takes; one warp per dx and one for the bias issue).  8 x 256^2:
// last layer 97 us, one tap at a time 147; middle 56 (80), first 49 (74).  Every FLUSH rows the accumulators are
// added to sums in registers (10 us more for the last layer): the tensor cores
// truncate, and over a whole run of rows the bias grew to 2e-6 of the gradient
// against 9e-7 now and 8e-7 on the FP32 pipes.
//
// Measured, 8 samples of 256^2 coarse points: the loss and all gradients 5.4 ms
// with the backward pass on the CUDA cores, 0.58 ms here; inference of one
// sample 80 us, 20 us here.
//
// Rows and pixels past the map's edge are computed from wrapped inputs (zeros
// in the gradients) and not stored.  Every mbarrier wait is bounded; on expiry
// the kernel records MGENKF_ERR_TIMEOUT in the status word, frees its TMEM and
// returns.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "conv_tc.h"
#include "tc_common.cuh"

namespace mgk {

namespace {

constexpr int kPix = 128;   // output pixels per MMA (M), or pixels of K per row
constexpr int kRowW = 136;  // smem pixels per input row (130 used)
constexpr int kConvThreads = 256;

__device__ __forceinline__ int wrap_c8(int v, int n) {
    while (v < 0) v += n;
    while (v >= n) v -= n;
    return v;
}

__device__ __forceinline__ void cp_async16_cg(uint32_t smem, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem), "l"(gmem) : "memory");
}
// 16 bytes, or zeros (nothing is read) if !ok
__device__ __forceinline__ void cp_async16_zfill(uint32_t smem, const void *gmem, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem), "l"(gmem), "r"(ok ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 two = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&two);
}

// the three BF16 parts of 8 FP32 values, 16 bytes each; the remainders are exact
__device__ __forceinline__ void split8(const float *x, uint4 (&part)[3]) {
    uint32_t *w[3] = {reinterpret_cast<uint32_t *>(&part[0]), reinterpret_cast<uint32_t *>(&part[1]),
                      reinterpret_cast<uint32_t *>(&part[2])};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float r0 = x[2 * q], r1 = x[2 * q + 1];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const __nv_bfloat162 two = __floats2bfloat162_rn(r0, r1);
            w[s][q] = *reinterpret_cast<const uint32_t *>(&two);
            r0 -= __bfloat162float(two.x);
            r1 -= __bfloat162float(two.y);
        }
    }
}

// four consecutive values, as one 16-byte load where the array starts on a
// 16-byte boundary (`wide`)
__device__ __forceinline__ void load4(const float *p, bool wide, float (&v)[4]) {
    if (wide) {
        const float4 f = *reinterpret_cast<const float4 *>(p);
        v[0] = f.x, v[1] = f.y, v[2] = f.z, v[3] = f.w;
    } else {
#pragma unroll
        for (int m = 0; m < 4; ++m) v[m] = p[m];
    }
}

constexpr int tmem_cols(int used) { return used <= 32 ? 32 : used <= 64 ? 64 : used <= 128 ? 128 : used <= 256 ? 256 : 512; }
// at most 512 / cols CTAs may share an SM's TMEM: ask for enough shared memory
// that no more are resident, so no CTA waits in alloc
constexpr int tmem_min_smem(int cols) { return 228 * 1024 / (512 / cols + 1) + 2048; }

// The tensor cores truncate their FP32 sums, a bias of up to one ulp of the
// accumulator per MMA.  A gradient's leading split therefore has an accumulator
// per row of taps (12 MMAs at most), its two remainders one of their own (2^-8
// of the size), and the four are added in registers.
template <int CG, int NSPLIT, int COUT, int ROWS>
struct ConvShape {
    static constexpr int NACC = NSPLIT == 1 ? 1 : 4;
    static constexpr int CGK = CG < 2 ? 2 : CG;               // channel groups of K (padded to 16 channels)
    // channel groups per chunk: a forward layer is one chunk (its MMAs run tap by
    // tap, and the order decides the FP32 sums that the BF16 activations round);
    // the splits of a gradient go 16 channels at a time
    static constexpr int GPC = NSPLIT == 1 ? CGK : 2;
    static constexpr int NC = NSPLIT * CGK / GPC;
    static constexpr int PLANE = (ROWS + 2) * kRowW * 16;     // bytes per channel-group plane
    static constexpr int STAGE = GPC * PLANE;
    static constexpr int NST = NC < 4 ? NC : 4;
    static constexpr int W_BYTES = 9 * CGK * COUT * 16;
    static constexpr int TMEM_COLS = tmem_cols(ROWS * NACC * COUT);
    static constexpr int NEED = 1024 + NST * STAGE + W_BYTES;
    static constexpr int SMEM = NEED > tmem_min_smem(TMEM_COLS) ? NEED : tmem_min_smem(TMEM_COLS);
    static_assert(ROWS * NACC * COUT <= 512, "accumulators of one CTA fit TMEM");
    static_assert(COUT % 16 == 0 && COUT >= 16 && COUT <= 256, "N of an M = 128 MMA");
    static_assert(CGK % 2 == 0, "K steps of 16 channels");
};

}  // namespace

// CG: channel groups of the input (1: the fields, normalised here); NSPLIT: 3
// for a gradient; EPI: kHidden, kResidual, kLoss or kBackward (conv_tc.h)
template <int CG, int NSPLIT, int COUT, int EPI, int ROWS>
__global__ void __launch_bounds__(kConvThreads, EPI == kLoss ? 3 : 2) k_conv_tc(ConvArgs A) {
    using S = ConvShape<CG, NSPLIT, COUT, ROWS>;
    launch_wait();
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sin = base;                       // NST stages of two planes of (ROWS + 2) x kRowW pixels
    unsigned char *sw = base + S::NST * S::STAGE;    // [9][CGK][COUT][8] bf16
    __shared__ uint64_t bar[S::NST];
    __shared__ uint32_t tmem_slot;
    __shared__ int s_fail;
    __shared__ float s_loss[kConvThreads / 32];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b = blockIdx.z, x0 = blockIdx.x * kPix, y0 = blockIdx.y * ROWS, n = A.n;
    const size_t pl = (size_t)n * n;
    if (tid == 0) {
        s_fail = A.status ? *A.status : 0;  // one read: the whole CTA leaves or none of it
        for (int q = 0; q < S::NST; ++q) tc::mbar_init(&bar[q], ROWS);
        fence_async_proxy();
    }
    __syncthreads();
    if (s_fail) return;
    if (warp == 0) tc::tmem_alloc(&tmem_slot, S::TMEM_COLS);
    const int uwarp = __shfl_sync(0xffffffffu, warp, 0);  // known to be uniform
    // the columns this lane copies of every input row
    constexpr int XC = (kPix + 2 + 31) / 32;
    int gx[XC];
#pragma unroll
    for (int q = 0; q < XC; ++q) gx[q] = wrap_c8(x0 - 1 + lane + 32 * q, n);
    // chunk c: GPC channel groups from GPC (c mod CGK/GPC) of split c / (CGK/GPC)
    auto load = [&](int c) {
        const int split = c / (S::CGK / S::GPC), g0 = S::GPC * (c % (S::CGK / S::GPC));
        unsigned char *st = sin + (c % S::NST) * S::STAGE;
        for (int rg = warp; rg < S::GPC * (ROWS + 2); rg += kConvThreads / 32) {
            const int g = rg / (ROWS + 2), r = rg - g * (ROWS + 2);
            const int gy = wrap_c8(y0 - 1 + r, n);
            unsigned char *dst = st + g * S::PLANE + r * kRowW * 16;
            const __nv_bfloat16 *src =
                A.in + (size_t)split * A.in_split + (((size_t)b * CG + g0 + g) * pl + (size_t)gy * n) * 8;
            const uint32_t d = tc::smem_u32(dst);
#pragma unroll
            for (int q = 0; q < XC; ++q)
                if (q < XC - 1 || lane + 32 * q < kPix + 2)
                    cp_async16_cg(d + (lane + 32 * q) * 16, src + (size_t)gx[q] * 8);
        }
    };
    // the normalised fields [dC, x^C*] as BF16 (group 1 is the K padding); every
    // load of a thread is issued before the first is used
    auto load_fields = [&]() {
        constexpr int TOT = (ROWS + 2) * (kPix + 2), IT = (TOT + kConvThreads - 1) / kConvThreads;
        float x[IT][8];
        size_t at[IT];
#pragma unroll
        for (int q = 0; q < IT; ++q) {
            const int e = min(tid + q * kConvThreads, TOT - 1), r = e / (kPix + 2), j = e - r * (kPix + 2);
            at[q] = (size_t)wrap_c8(y0 - 1 + r, n) * n + wrap_c8(x0 - 1 + j, n);
#pragma unroll
            for (int ch = 0; ch < 8; ++ch)
                x[q][ch] = __ldg((ch < 4 ? A.dC : A.xs) + ((size_t)b * 4 + (ch & 3)) * pl + at[q]);
        }
#pragma unroll
        for (int q = 0; q < IT; ++q) {
            const int e = tid + q * kConvThreads, r = e / (kPix + 2), j = e - r * (kPix + 2);
            if (e >= TOT) continue;
            uint4 pk;
            uint32_t *w = reinterpret_cast<uint32_t *>(&pk);
#pragma unroll
            for (int h = 0; h < 4; ++h)
                w[h] = pack2((x[q][2 * h] - __ldg(A.stats + 2 * h)) / __ldg(A.stats + 8 + 2 * h),
                             (x[q][2 * h + 1] - __ldg(A.stats + 2 * h + 1)) / __ldg(A.stats + 9 + 2 * h));
            unsigned char *dst = sin + (r * kRowW + j) * 16;
            *reinterpret_cast<uint4 *>(dst) = pk;
            *reinterpret_cast<uint4 *>(dst + S::PLANE) = make_uint4(0, 0, 0, 0);
            if (A.a0 && r >= 1 && r <= ROWS && j >= 1 && j <= kPix && y0 + r - 1 < n && x0 + j - 1 < n)
                reinterpret_cast<uint4 *>(A.a0)[(size_t)b * pl + at[q]] = pk;
        }
    };
    for (int e = tid; e < S::W_BYTES / 16; e += kConvThreads)
        cp_async16_cg(tc::smem_u32(sw) + e * 16, A.wp + (size_t)e * 8);
    for (int c = 0; c < S::NST; ++c) {
        if (CG == 1)
            load_fields();
        else
            load(c);
        cp_async_commit();
    }
    const int rows = min(ROWS, n - y0);
    if (EPI == kLoss) {
        // the target values of this thread's pixel on their way to L2 while the
        // tensor cores work (a line holds eight lanes' 16 bytes)
        const int x = x0 + (warp & 3) * 32 + lane, nf = 4 * n;
        for (int r = warp >> 2; r < rows; r += 2)
            if (x < n && (lane & 7) == 0)
                for (int q = 0; q < 16; ++q) {
                    const float *t = A.target + (((size_t)b * 4 + (q >> 2)) * nf + 4 * (y0 + r) + (q & 3)) * (size_t)nf +
                                     4 * (size_t)x;
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(t));
                }
    }
    const uint32_t a0 = tc::smem_u32(sin), b0 = tc::smem_u32(sw);
    uint32_t tmem = 0;
    bool ok = true;
    for (int c = 0; c < S::NC; ++c) {
        cp_async_wait<(S::NST > 1 ? S::NST - 2 : 0)>();  // chunk c has landed (one group per iteration below)
        fence_async_proxy();                             // written by the generic proxy, read by the tensor cores
        tc::fence_before_sync();
        if (__syncthreads_or(!ok)) {
            ok = false;
            break;
        }
        tc::fence_after_sync();
        tmem = tmem_slot;
        if (uwarp < ROWS) {
            constexpr uint32_t idesc = tc::idesc_bf16(kPix, COUT);
            const bool lead = tc::elect_one();
            const uint32_t ac = a0 + (uint32_t)((c % S::NST) * S::STAGE + uwarp * kRowW * 16);
            const uint32_t bc = b0 + (uint32_t)(S::GPC * (c % (S::CGK / S::GPC)) * COUT * 16);
            const uint32_t acc = tmem + (uint32_t)(uwarp * S::NACC * COUT);
            constexpr int CPS = S::CGK / S::GPC;  // chunks per split
            if (uwarp < rows) {
#pragma unroll
                for (int t = 0; t < 9; ++t) {
#pragma unroll
                    for (int k = 0; k < S::GPC / 2; ++k) {
                        const uint64_t ad = tc::smem_desc_interleave(
                            ac + (uint32_t)(2 * k * S::PLANE + ((t / 3) * kRowW + t % 3) * 16), S::PLANE, 128);
                        const uint64_t bd = tc::smem_desc_interleave(
                            bc + (uint32_t)((t * S::CGK + 2 * k) * COUT * 16), COUT * 16, 128);
                        if (NSPLIT == 1) {
                            tc::mma_bf16_lead(lead, acc, ad, bd, idesc, (c | t | k) ? 1u : 0u);
                        } else {
                            const bool first = c < CPS;  // the leading split
                            tc::mma_bf16_lead(lead, acc + (uint32_t)((first ? t / 3 : 3) * COUT), ad, bd, idesc,
                                              (first ? (c | (t % 3) | k) : ((c - CPS) | t | k)) ? 1u : 0u);
                        }
                    }
                }
            }
            if (lead) tc::mma_commit(&bar[c % S::NST]);
        }
        if (c >= 1 && c - 1 + S::NST < S::NC) {  // refill the stage that chunk c - 1 has left
            ok = tc::mbar_wait(&bar[(c - 1) % S::NST], ((c - 1) / S::NST) & 1);
            if (ok) load(c - 1 + S::NST);
        }
        cp_async_commit();
    }
    cp_async_wait<0>();
    if (ok) ok = tc::mbar_wait(&bar[(S::NC - 1) % S::NST], ((S::NC - 1) / S::NST) & 1);
    // uniform over the CTA: the TMEM loads below are warp-collective
    ok = !__syncthreads_or(!ok);
    float lsum = 0.f;
    if (!ok) {
        if (tid == 0 && A.status) atomicCAS(A.status, 0, tc::kStTimeout);
    } else {
        tc::fence_after_sync();
        const int x = x0 + (warp & 3) * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        int cx[4];  // kLoss: the columns of the pixel's Lagrange stencil
        if (EPI == kLoss)
#pragma unroll
            for (int t = 0; t < 4; ++t) cx[t] = wrap_c8(x - 1 + t, n);
        for (int r = warp >> 2; r < rows; r += 2) {
            const int y = y0 + r;
            const size_t p = (size_t)y * n + x;
            int cy[4];
            if (EPI == kLoss)
#pragma unroll
                for (int t = 0; t < 4; ++t) cy[t] = wrap_c8(y - 1 + t, n) * n;
#pragma unroll
            for (int c0 = 0; c0 < COUT; c0 += 16) {
                float v[16];
                __syncwarp();
                tc::tmem_ld16(lane_base + (uint32_t)(r * S::NACC * COUT + c0), v);
#pragma unroll
                for (int h = 1; h < S::NACC; ++h) {
                    float v1[16];
                    tc::tmem_ld16(lane_base + (uint32_t)((r * S::NACC + h) * COUT + c0), v1);
#pragma unroll
                    for (int q = 0; q < 16; ++q) v[q] += v1[q];
                }
                if (x < n) {
                    if (EPI != kBackward) {
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            v[q] += __ldg(A.bias + c0 + q);
                            if (EPI == kHidden) v[q] = fmaxf(v[q], 0.f);
                        }
                    }
                    if (EPI == kHidden) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint4 pk;
                            uint32_t *w = reinterpret_cast<uint32_t *>(&pk);
#pragma unroll
                            for (int q = 0; q < 4; ++q) w[q] = pack2(v[8 * h + 2 * q], v[8 * h + 2 * q + 1]);
                            reinterpret_cast<uint4 *>(A.out)[((size_t)b * (COUT / 8) + (c0 >> 3) + h) * pl + p] = pk;
                        }
                    } else if (EPI == kResidual) {
                        // channel 16 c + 4 sy + sx is fine point (4 y + sy, 4 x + sx) of fine channel c
                        const int c = c0 >> 4, nf = 4 * n;
                        const float s = __ldg(A.stats + 16 + c);
#pragma unroll
                        for (int sy = 0; sy < 4; ++sy) {
                            float *o = A.res + (((size_t)b * 4 + c) * nf + 4 * y + sy) * (size_t)nf + 4 * (size_t)x;
                            float f[4], old[4] = {0.f, 0.f, 0.f, 0.f};
                            if (A.accumulate) load4(o, A.wide, old);
#pragma unroll
                            for (int m = 0; m < 4; ++m) {
                                const float r1 = s * v[4 * sy + m];
                                f[m] = A.accumulate ? old[m] + r1 : r1;
                            }
                            if (A.wide) {
                                *reinterpret_cast<float4 *>(o) = make_float4(f[0], f[1], f[2], f[3]);
                            } else {
#pragma unroll
                                for (int m = 0; m < 4; ++m) o[m] = f[m];
                            }
                        }
                    } else if (EPI == kLoss) {
                        const int c = c0 >> 4, nf = 4 * n;
                        const float s = __ldg(A.stats + 16 + c);
                        // s and the differences times 2^+-64 where the reciprocal would
                        // over- or underflow
                        const float f = fabsf(s) < 0x1p-60f ? 0x1p64f : fabsf(s) > 0x1p60f ? 0x1p-64f : 1.f;
                        const float sf = s * f, rs = 1.f / sf;
                        // Pi_F(dC) at the pixel's 16 fine points: 4-tap sums along x, then along y
                        const float *d = A.dC + ((size_t)b * 4 + c) * pl;
                        float sx[4][4];
#pragma unroll
                        for (int ty = 0; ty < 4; ++ty) {
                            const float *dr = d + cy[ty];
                            float e[4];
#pragma unroll
                            for (int t = 0; t < 4; ++t) e[t] = __ldg(dr + cx[t]);
#pragma unroll
                            for (int m = 0; m < 4; ++m) {
                                float a = 0.f;
#pragma unroll
                                for (int t = 0; t < 4; ++t) a = fmaf(A.pw[4 * m + t], e[t], a);
                                sx[ty][m] = a;
                            }
                        }
#pragma unroll
                        for (int sy = 0; sy < 4; ++sy) {
                            float tv[4];
                            load4(A.target + (((size_t)b * 4 + c) * nf + 4 * y + sy) * (size_t)nf + 4 * (size_t)x,
                                  A.wide, tv);
#pragma unroll
                            for (int m = 0; m < 4; ++m) {
                                float pf = 0.f;
#pragma unroll
                                for (int ty = 0; ty < 4; ++ty) pf = fmaf(A.pw[4 * sy + ty], sx[ty][m], pf);
                                // the quotient by s: a product with the reciprocal and one
                                // correction by its remainder (a Newton step for the quotient);
                                // the remainder of an infinite quotient is not a number and
                                // becomes a finite one here
                                const float x1 = s * v[4 * sy + m] - (tv[m] - pf), x2 = x1 * f, q1 = x2 * rs;
                                const float dv = fmaf(fminf(fmaf(-q1, sf, x2), 3e38f), rs, q1);
                                lsum += dv * dv;
                                v[4 * sy + m] = 2.f * dv * A.inv_count;
                            }
                        }
                    } else {  // kBackward: ReLU mask of the layer's input
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint4 mk = reinterpret_cast<const uint4 *>(
                                A.mask)[((size_t)b * (COUT / 8) + (c0 >> 3) + h) * pl + p];
                            const __nv_bfloat16 *mv = reinterpret_cast<const __nv_bfloat16 *>(&mk);
#pragma unroll
                            for (int q = 0; q < 8; ++q)
                                if (!(__bfloat162float(mv[q]) > 0.f)) v[8 * h + q] = 0.f;
                        }
                    }
                    if (EPI == kLoss || EPI == kBackward) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint4 part[3];
                            split8(v + 8 * h, part);
                            const size_t o = (((size_t)b * (COUT / 8) + (c0 >> 3) + h) * pl + p) * 8;
#pragma unroll
                            for (int q = 0; q < 3; ++q) *reinterpret_cast<uint4 *>(A.out + q * A.out_split + o) = part[q];
                        }
                    }
                }
            }
        }
    }
    if (EPI == kLoss) {
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, o);
        if (lane == 0) s_loss[warp] = lsum;
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem_slot, S::TMEM_COLS);
    if (EPI == kLoss && tid == 0) {
        float t = 0.f;
        for (int q = 0; q < kConvThreads / 32; ++q) t += s_loss[q];
        A.loss_part[((size_t)b * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t * A.inv_count;
    }
}

template <int CG, int NSPLIT, int COUT, int EPI, int ROWS>
static cudaError_t conv_launch(const ConvArgs &A, int batch, cudaStream_t s) {
    using S = ConvShape<CG, NSPLIT, COUT, ROWS>;
    static OncePerDevice attr;
    attr.run([](int) {
        return cudaFuncSetAttribute(k_conv_tc<CG, NSPLIT, COUT, EPI, ROWS>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM);
    });
    count_launches(1);
    const dim3 grid(ceil_div(A.n, kPix), ceil_div(A.n, ROWS), batch);
    return launch_kernel(k_conv_tc<CG, NSPLIT, COUT, EPI, ROWS>, grid, kConvThreads, S::SMEM, s, LaunchHow{}, A);
}

// Four output rows per CTA read 1.5 input rows per output row, two read 2, but
// two rows give twice the CTAs (taken by the forward layers while four would
// leave SMs without two CTAs: one 256^2 sample has 128 CTAs of four rows) and
// need less shared memory and TMEM: a ring of four stages instead of two in the
// backward layers (the last layer's adjoint at 8 x 256^2: 210 us with four rows,
// 185 with two), three CTAs per SM instead of two in the loss (190 and 95 us).
static int conv_rows(int n, int batch, int epi) {
    if (epi == kLoss || epi == kBackward) return 2;
    return (long long)ceil_div(n, kPix) * ceil_div(n, 4) * batch >= 2 * kNumSMs ? 4 : 2;
}

template <int CG, int NSPLIT, int COUT, int EPI>
cudaError_t launch_conv_tc(const ConvArgs &A, int batch, cudaStream_t s) {
    if constexpr (EPI == kHidden || EPI == kResidual)
        if (conv_rows(A.n, batch, EPI) == 4) return conv_launch<CG, NSPLIT, COUT, EPI, 4>(A, batch, s);
    return conv_launch<CG, NSPLIT, COUT, EPI, 2>(A, batch, s);
}

int conv_loss_parts(int n, int batch) { return ceil_div(n, kPix) * ceil_div(n, conv_rows(n, batch, kLoss)) * batch; }

// ---------------------------------------------------------------------------
// weight gradients
// ---------------------------------------------------------------------------
namespace {

template <int CGI, int COUT>
struct WgradShape {
    static constexpr int CGB = CGI < 2 ? 2 : CGI;           // channel groups of N (padded to 16 channels)
    static constexpr int N = 8 * CGB;
    static constexpr int AG = COUT / 8;                     // channel groups of one split
    static constexpr int PXS = COUT == 64 ? kPix / 2 : kPix;  // pixels of a row of d per stage
    static constexpr int APL = PXS * 16;                    // bytes of one group's plane of a stage
    static constexpr int A_STAGE = 4 * AG * APL;            // COUT 32: [hi][mid][lo][zeros], 64: [hi][mid][zeros][lo]
    static constexpr int NST = 4;                           // stages: three in flight beside the one in use
    // M = 128 MMAs per K step: (hi, mid, lo, 0), or (hi, mid) and (0, lo) into the
    // same accumulator rows (the remainders together: see ConvShape)
    static constexpr int NM = COUT / 32;
    static constexpr int LO = COUT == 64 ? 3 : 2, ZERO = 5 - LO;  // which quarter of a stage holds lo, zeros
    static constexpr int FLUSH = 2;                         // rows of d summed in TMEM before the registers
    static constexpr int BPL = kRowW * 16;
    static constexpr int B_ROW = CGB * BPL;                 // one row of the input
    static constexpr int USED = 9 * N + 16;                 // TMEM columns: nine taps and the bias
    static constexpr int TMEM_COLS = tmem_cols(USED);
    // a ring of eight input rows, the first two once more behind them: the three
    // rows around a gradient row are always consecutive in memory
    static constexpr int NEED = 1024 + NST * A_STAGE + 10 * B_ROW + 2 * APL;
    static constexpr int SMEM = NEED > tmem_min_smem(TMEM_COLS) ? NEED : tmem_min_smem(TMEM_COLS);
    static_assert(COUT == 32 || COUT == 64, "the stacked splits fill one or two M = 128 operands");
    static_assert(NST * A_STAGE >= 128 * (N + 1) * 4, "the epilogue's tile of one tap reuses the stages");
};

}  // namespace

// unit = a run of `rs` rows of one 128-pixel column strip of one sample;
// part[unit][t][o][i], then db[o]
template <int CGI, int COUT>
__global__ void __launch_bounds__(kConvThreads, 1) k_conv_wgrad(const __nv_bfloat16 *__restrict__ in,
                                                                const __nv_bfloat16 *__restrict__ d, size_t d_split,
                                                                int n, int rs, float *__restrict__ part,
                                                                int *status) {
    using S = WgradShape<CGI, COUT>;
    constexpr int CIN = 8 * CGI;
    launch_wait();
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *sa = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char *sb = sa + S::NST * S::A_STAGE;  // ring of eight input rows, and two again
    unsigned char *s1 = sb + 10 * S::B_ROW;        // two planes of ones: the bias operand
    __shared__ uint64_t bar[S::NST];
    __shared__ uint32_t tmem_slot;
    __shared__ int s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        s_fail = status ? *status : 0;
        for (int q = 0; q < S::NST; ++q) tc::mbar_init(&bar[q], 4);
        fence_async_proxy();
    }
    __syncthreads();
    if (s_fail) return;
    if (warp == 0) tc::tmem_alloc(&tmem_slot, S::TMEM_COLS);
    const int uwarp = __shfl_sync(0xffffffffu, warp, 0);  // known to be uniform
    const int xb = ceil_div(n, kPix), segs = ceil_div(n, rs);
    const int strip = blockIdx.x / segs, seg = blockIdx.x - strip * segs;
    const int b = strip / xb, x0 = (strip - b * xb) * kPix;
    const int r0 = seg * rs, rows = min(rs, n - r0);
    const size_t pl = (size_t)n * n;
    // constant parts: the zero planes of the stages, the padded input group, the ones
    for (int e = tid; e < S::NST * S::AG * S::PXS; e += kConvThreads) {
        const int st = e / (S::AG * S::PXS), k = e - st * (S::AG * S::PXS);
        reinterpret_cast<uint4 *>(sa + st * S::A_STAGE + S::ZERO * S::AG * S::APL)[k] = make_uint4(0, 0, 0, 0);
    }
    if (CGI < 2)
        for (int e = tid; e < 10 * kRowW; e += kConvThreads)
            reinterpret_cast<uint4 *>(sb + (e / kRowW) * S::B_ROW + S::BPL)[e % kRowW] = make_uint4(0, 0, 0, 0);
    for (int e = tid; e < 2 * S::PXS; e += kConvThreads) {
        const uint32_t one2 = 0x3F803F80u;  // two BF16 ones
        reinterpret_cast<uint4 *>(s1)[e] = make_uint4(one2, one2, one2, one2);
    }
    constexpr int XC = (kPix + 2 + 31) / 32;
    int gx[XC];
#pragma unroll
    for (int q = 0; q < XC; ++q) gx[q] = wrap_c8(x0 - 1 + lane + 32 * q, n);
    // input row y (map row, may be -1 .. n) into ring slot s = (y - r0 + 1) mod 8
    // (and s + 8)
    auto load_in = [&](int y) {
        const int gy = wrap_c8(y, n), slot = (y - r0 + 1) & 7;
        const uint32_t dst = tc::smem_u32(sb + slot * S::B_ROW);
        for (int g = warp; g < CGI; g += kConvThreads / 32) {
            const __nv_bfloat16 *src = in + (((size_t)b * CGI + g) * pl + (size_t)gy * n) * 8;
#pragma unroll
            for (int q = 0; q < XC; ++q)
                if (q < XC - 1 || lane + 32 * q < kPix + 2) {
                    cp_async16_cg(dst + g * S::BPL + (lane + 32 * q) * 16, src + (size_t)gx[q] * 8);
                    if (slot < 2)
                        cp_async16_cg(dst + 8 * S::B_ROW + g * S::BPL + (lane + 32 * q) * 16, src + (size_t)gx[q] * 8);
                }
        }
    };
    // step q: pixels PXS (q mod SPR) .. of gradient row r0 + q / SPR into stage
    // q mod NST (zeros past the map's edge), and with a row's first step the
    // input row below it
    constexpr int SPR = kPix / S::PXS;
    const int steps = rows * SPR;
    auto load_step = [&](int q) {
        const int i = q / SPR, px = (q % SPR) * S::PXS;
        const uint32_t dst = tc::smem_u32(sa + (q % S::NST) * S::A_STAGE);
        for (int e = tid; e < 3 * S::AG * S::PXS; e += kConvThreads) {
            const int g = e / S::PXS, j = px + e % S::PXS, split = g / S::AG;
            const bool in_map = x0 + j < n;
            const __nv_bfloat16 *src = d + (size_t)split * d_split +
                                       (((size_t)b * S::AG + (g - split * S::AG)) * pl + (size_t)(r0 + i) * n +
                                        (in_map ? x0 + j : 0)) * 8;
            const int shift = split == 2 ? (S::LO - 2) * S::AG * S::APL : 0;
            cp_async16_zfill(dst + e * 16 + shift, src, in_map);
        }
        if (q % SPR == 0) load_in(r0 + i + 1);
    };
    load_in(r0 - 1);
    load_in(r0);
    for (int q = 0; q < S::NST; ++q) {
        if (q < steps) load_step(q);
        cp_async_commit();
    }
    uint32_t tmem = 0;
    bool ok = true;
    // the running sums: warps 0-3 hold five taps of their 32 accumulator rows,
    // warps 4-7 four and the bias; block t of the accumulators is tap
    // (t mod 3, t / 3)
    const int half = warp >> 2;
    constexpr int HT = 5;
    float sum[HT * S::N];
#pragma unroll
    for (int e = 0; e < HT * S::N; ++e) sum[e] = 0.f;
    for (int q = 0; q < steps; ++q) {
        cp_async_wait<S::NST - 2>();  // step q has landed (one group per iteration below)
        fence_async_proxy();
        tc::fence_before_sync();
        if (__syncthreads_or(!ok)) {
            ok = false;
            break;
        }
        tc::fence_after_sync();
        tmem = tmem_slot;
        if (uwarp < 4) {
            // both operands MN-major (instruction bits 15, 16); K groups 128 bytes
            // apart, channel groups one plane apart.  Warp w < 3 issues the taps
            // (0 .. 2, w), whose operands are the channel groups of three
            // consecutive rows; warp 3 the bias
            constexpr uint32_t mn = (1u << 15) | (1u << 16);
            const uint32_t idesc = (uwarp == 3 ? tc::idesc_bf16(128, 16) : tc::idesc_bf16(128, 3 * S::N)) | mn;
            const bool lead = tc::elect_one();
            const int i = q / SPR, px = (q % SPR) * S::PXS;
            const uint32_t aa = tc::smem_u32(sa + (q % S::NST) * S::A_STAGE);
            // row r0 + i - 1 + dy sits in slot i mod 8 + dy
            const uint32_t bt = uwarp == 3 ? tc::smem_u32(s1)
                                           : tc::smem_u32(sb) + (uint32_t)((i & 7) * S::B_ROW + (px + uwarp) * 16);
            const uint32_t pitch = uwarp == 3 ? S::APL : S::BPL;
            const uint32_t dt = tmem + (uint32_t)(3 * uwarp * S::N);
#pragma unroll
            for (int k = 0; k < S::PXS / 16; ++k) {
#pragma unroll
                for (int m = 0; m < S::NM; ++m) {
                    const uint64_t ad =
                        tc::smem_desc_interleave(aa + (uint32_t)(m * 16 * S::APL + k * 256), 128, S::APL);
                    const uint32_t acc = ((q % (S::FLUSH * SPR)) | k | m) ? 1u : 0u;
                    tc::mma_bf16_lead(lead, dt, ad, tc::smem_desc_interleave(bt + k * 256, 128, pitch), idesc, acc);
                }
            }
            if (lead) tc::mma_commit(&bar[q % S::NST]);
        }
        if (q >= 1 && q - 1 + S::NST < steps) {  // refill the stage (and the ring slot) that step q - 1 has left
            ok = tc::mbar_wait(&bar[(q - 1) % S::NST], ((q - 1) / S::NST) & 1);
            if (ok) load_step(q - 1 + S::NST);
        }
        cp_async_commit();
        if ((q + 1) % (S::FLUSH * SPR) == 0 || q + 1 == steps) {
            // the sums of these rows into the registers; the next step's MMAs
            // start anew (after the barrier at the top)
            ok = ok && tc::mbar_wait(&bar[q % S::NST], (q / S::NST) & 1);
            if (__syncthreads_or(!ok)) {
                ok = false;
                break;
            }
            tc::fence_after_sync();
            const uint32_t src = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(half * HT * S::N);
#pragma unroll
            for (int t = 0; t < HT; ++t) {
                if (half && t == HT - 1) {
                    float v[16];
                    tc::tmem_ld16(src + (uint32_t)(t * S::N), v);
                    sum[t * S::N] += v[0];
                } else {
#pragma unroll
                    for (int c0 = 0; c0 < S::N; c0 += 16) {
                        float v[16];
                        tc::tmem_ld16(src + (uint32_t)(t * S::N + c0), v);
#pragma unroll
                        for (int e = 0; e < 16; ++e) sum[t * S::N + c0 + e] += v[e];
                    }
                }
            }
        }
    }
    cp_async_wait<0>();
    ok = !__syncthreads_or(!ok);
    if (!ok) {
        if (tid == 0 && status) atomicCAS(status, 0, tc::kStTimeout);
    } else {
        // per tap: the 128 accumulator rows to shared memory, the splits' rows
        // added (hi + mid) + lo in order
        float *tile = reinterpret_cast<float *>(sa);
        constexpr int LD = S::N + 1;
        float *out = part + (size_t)blockIdx.x * (9 * COUT * CIN + COUT);
        const int m = (warp & 3) * 32 + lane;
#pragma unroll
        for (int t = 0; t <= 9; ++t) {
            if (half == t / HT) {
#pragma unroll
                for (int c = 0; c < (t < 9 ? S::N : 1); ++c) tile[m * LD + c] = sum[(t % HT) * S::N + c];
            }
            __syncthreads();
            const int count = t < 9 ? COUT * CIN : COUT, width = t < 9 ? CIN : 1;
            for (int e = tid; e < count; e += kConvThreads) {
                const int o = e / width, c = e - o * width;
                float v = tile[o * LD + c] + tile[(o + COUT) * LD + c];
                if (COUT == 32) v += tile[(o + 2 * COUT) * LD + c];
                out[(size_t)(t < 9 ? t % 3 * 3 + t / 3 : t) * COUT * CIN + e] = v;
            }
            __syncthreads();
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem_slot, S::TMEM_COLS);
}

// rows per unit: as many units as fit one CTA per SM (its TMEM) in one wave,
// a whole strip where there are more strips than SMs
static int wgrad_rows(int n, int batch) {
    const int strips = ceil_div(n, kPix) * batch;
    return ceil_div(n, std::max(1, std::min(n, kNumSMs / strips)));
}
int wgrad_units(int n, int batch) { return ceil_div(n, kPix) * batch * ceil_div(n, wgrad_rows(n, batch)); }

template <int CGI, int COUT>
cudaError_t launch_conv_wgrad(const __nv_bfloat16 *in, const __nv_bfloat16 *d, size_t d_split, int n, int batch,
                              float *part, int *status, cudaStream_t s) {
    using S = WgradShape<CGI, COUT>;
    static OncePerDevice attr;
    attr.run([](int) {
        return cudaFuncSetAttribute(k_conv_wgrad<CGI, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM);
    });
    count_launches(1);
    return launch_kernel(k_conv_wgrad<CGI, COUT>, wgrad_units(n, batch), kConvThreads, S::SMEM, s, LaunchHow{}, in, d,
                         d_split, n, wgrad_rows(n, batch), part, status);
}

int conv_packed_elems(int cin, int cout) { return 9 * (cin < 16 ? 2 : cin / 8) * cout * 8; }

template cudaError_t launch_conv_tc<1, 1, 32, kHidden>(const ConvArgs &, int, cudaStream_t);
template cudaError_t launch_conv_tc<4, 1, 32, kHidden>(const ConvArgs &, int, cudaStream_t);
template cudaError_t launch_conv_tc<4, 1, 64, kResidual>(const ConvArgs &, int, cudaStream_t);
template cudaError_t launch_conv_tc<4, 1, 64, kLoss>(const ConvArgs &, int, cudaStream_t);
template cudaError_t launch_conv_tc<8, 3, 32, kBackward>(const ConvArgs &, int, cudaStream_t);
template cudaError_t launch_conv_tc<4, 3, 32, kBackward>(const ConvArgs &, int, cudaStream_t);
template cudaError_t launch_conv_wgrad<4, 64>(const __nv_bfloat16 *, const __nv_bfloat16 *, size_t, int, int, float *,
                                              int *, cudaStream_t);
template cudaError_t launch_conv_wgrad<4, 32>(const __nv_bfloat16 *, const __nv_bfloat16 *, size_t, int, int, float *,
                                              int *, cudaStream_t);
template cudaError_t launch_conv_wgrad<1, 32>(const __nv_bfloat16 *, const __nv_bfloat16 *, size_t, int, int, float *,
                                              int *, cudaStream_t);

}  // namespace mgk
