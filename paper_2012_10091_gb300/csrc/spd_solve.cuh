// spd_solve.cuh -- FP64 solve of a small SPD system with many right-hand sides
// (the gain solve, Algorithm 3 step 8), device bodies shared by the launches
// over one problem and over many.
//
// GB300 issues one FP64 instruction of a warp per SM sub-partition in 64 cycles,
// whatever its lanes do, and with no further latency: a step that depends on
// the previous one costs its FP64 instructions, and work costs its warp
// instructions divided by the sub-partitions it is spread over.  So
//   * the factorisation S = L D L^T (unit L) and its inverse W = L^-1 run on a
//     cluster of C CTAs.  The matrix is cut into 16 x 16 blocks; CTA 0 does
//     nothing but the serial chain (the diagonal blocks), the others own the
//     blocks of the lower triangle and do the products.  A block (i, j) of
//     row i holds A_ij until panel j is done and the running X_ij of
//     L W = I from then on, so one elimination yields L, D and W in place;
//   * the solves are then products with W, S^-1 b = W^T D^-1 W b: no
//     substitution chain, one or a few columns per CTA over the whole GPU.
// Measured, n = 128 (129 columns): Cholesky by column panels on eight CTAs and
// one warp of substitution per column 150 + 43 us, this 73 + 19 us; n = 64: 62 + 22
// and 36 + 10 us.  The chain bounds the factorisation: about 600 cycles per pivot
// (five dependent FP64 instructions, a barrier, shared-memory latency) and 6 k
// per panel for the blocks that lead to the next diagonal block.
#pragma once

#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"

namespace mgk {

constexpr int kSpdMax = 256;      // largest order
constexpr int kSpdThreads = 256;
constexpr int kSpdB = 16;         // block order
constexpr int kSpdLd = 17;        // row pitch of a block in shared memory
constexpr int kSpdBlk = kSpdB * kSpdLd;
constexpr int kSpdMaxBlocks = kSpdMax / kSpdB;

// C = 8 CTAs per problem (a portable cluster; many problems share the GPU), 16
// for one larger problem, where seven workers cannot keep up with the chain
// (n = 100: 62 us with either, 128: 82 and 73 us, 256: 398 and 235 us).
constexpr int kSpdGroupCluster = 8;
constexpr int spd_cluster(int n) { return n > 112 ? 16 : 8; }

// the worker that owns block (i, j), j <= i: 1 .. C - 1.  Within a column (and a
// row) consecutive blocks have different owners.
template <int C>
__device__ __forceinline__ int spd_owner(int i, int j) {
    return 1 + (i + j) % (C - 1);
}
// block slots per CTA for nb block rows: a worker owns at most i / (C - 1) + 1
// blocks of row i; CTA 0 keeps nb inverse diagonal blocks and its two work blocks
__host__ __device__ inline int spd_slots(int nb, int C) {
    int c = 0;
    for (int i = 0; i < nb; ++i) c += i / (C - 1) + 1;
    return c > nb + 2 ? c : nb + 2;
}
// dynamic shared memory of the factorisation of order n: the slots, the
// published Q and P of up to three blocks of a column, two pairs of operands,
// the reciprocal pivots
inline size_t spd_factor_smem(int n, int C) {
    return sizeof(double) * ((size_t)(spd_slots((n + kSpdB - 1) / kSpdB, C) + 6 + 4) * kSpdBlk + kSpdMax);
}

// 1 / d of a pivot, to about one unit in the last place: with e = 1 - d y of an
// approximate reciprocal y, y (1 + e + e^2) = (1 - e^3) / d (third-order
// Newton iteration).  A pivot that is not positive and finite raises *fail and
// yields 1, so that the factorisation runs on.
__device__ __forceinline__ double spd_pivot(double d, int *fail) {
    // comparisons of doubles would take the FP64 pipe (64 cycles each): a high
    // word in this range is a positive number between about 1e-300 and 1e300
    const int hi = __double2hiint(d);
    if (hi < 0x01c00000 || hi > 0x7e000000) {
        if (!(d > 0.0) || !isfinite(d)) {
            *fail = 1;
            return 1.0;
        }
        return 1.0 / d;
    }
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-d, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// A diagonal block by warps 0-3 (128 threads): e[0] holds it (both triangles); W = L^-1 of the block into `linv` (unit diagonal, zeros
// above) and 1 / D into `dinv`.  Pivot k takes one barrier: warp 0 updates the
// next diagonal entry by itself and forms its reciprocal (two and three
// dependent FP64 instructions, the chain) while warps 1-3, on the other three
// sub-partitions, eliminate column k from the rows below in one of two buffers.
__device__ __forceinline__ void spd_diag(double (*e)[kSpdBlk], double *linv, double *dinv, int *fail) {
    __shared__ double s_y[2];
    const int tid = threadIdx.x;
    if (tid == 0) s_y[0] = spd_pivot(e[0][0], fail);
    const int r = (tid - 32) & 15, g = (tid - 32) >> 4;
#pragma unroll
    for (int k = 0; k < kSpdB; ++k) {
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const double *cur = e[k & 1];
        double *nxt = e[(k + 1) & 1];
        const double y = s_y[k & 1];
        if (tid < 32) {
            if (tid == 0) dinv[k] = y;
            if (k + 1 < kSpdB) {
                const double a = cur[(k + 1) * kSpdLd + k], d = cur[(k + 1) * kSpdLd + k + 1];
                const double yn = spd_pivot(fma(-(a * y), a, d), fail);
                if (tid == 0) s_y[(k + 1) & 1] = yn;
            }
        } else {
            // element (r, c), c = g, g + 6, g + 12: a column c > k of A or c < k of X
            const double nl = -(cur[r * kSpdLd + k] * y);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int c = g + 6 * q;
                if (c < kSpdB) {
                    double v = cur[r * kSpdLd + c];
                    if (r > k) v = c == k ? nl : fma(nl, cur[k * kSpdLd + c], v);
                    nxt[r * kSpdLd + c] = v;
                }
            }
        }
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    for (int q = tid; q < kSpdB * kSpdB; q += 128) {
        const int r = q >> 4, c = q & 15;
        linv[r * kSpdLd + c] = r > c ? e[0][r * kSpdLd + c] : (r == c ? 1.0 : 0.0);
    }
}

// S (n x n row-major, lower triangle read) -> A: W = L^-1 below the diagonal,
// 1 / D on it; At: the transpose of W below.  A pivot that is not positive and
// finite sets the status and leaves A and At as they were.  One cluster of C
// CTAs; the arithmetic does not depend on C.
template <int C>
__device__ __forceinline__ void spd_factor_body(double *A, double *At, int n, int *status) {
    namespace cg = cooperative_groups;
    extern __shared__ double spd_sm[];
    __shared__ int s_fail;
    __shared__ unsigned char s_slot[kSpdMaxBlocks][kSpdMaxBlocks];
    __shared__ unsigned char s_i[32], s_j[32];
    __shared__ int s_n;
    cg::cluster_group cl = cg::this_cluster();
    const int q = (int)cl.block_rank(), nb = (n + kSpdB - 1) / kSpdB, tid = threadIdx.x;
    if (*status) return;          // written only at the end of a launch
    if (nb == 1 && q > 0) return;  // one diagonal block: no worker
    const int slots = spd_slots(nb, C);
    double *blk = spd_sm;                        // worker: its blocks; CTA 0: linv[nb], then e[2] and a spare
    double *pub = blk + slots * kSpdBlk;         // worker: Q, P of its blocks of the panel's column
    double *op = pub + 6 * kSpdBlk;              // two pairs of operands
    double *dv = op + 4 * kSpdBlk;               // CTA 0: 1 / D of every panel; worker: of the current one
    double(*e)[kSpdBlk] = reinterpret_cast<double(*)[kSpdBlk]>(blk + nb * kSpdBlk);
    const int lr = tid >> 4, lc = tid & 15;      // element in row order (loads, stores)
    const int ur = tid & 15, uc = tid >> 4;      // element of a product: a warp has all rows of two columns
    const int warp = tid >> 5, lane = tid & 31;
    // two columns (or rows) per warp, so that the four sub-partitions get equal
    // triangles: pairs w and 7 - w share one
    const int pr = warp < 4 ? warp : 11 - warp, px = 2 * pr + (lane >> 4), py = lane & 15;
    if (tid == 0) {
        s_fail = 0;
        s_n = 0;
    }
    __syncthreads();
    if (lc <= lr && lr < nb) {  // thread (lr, lc) places block (lr, lc)
        const int own = spd_owner<C>(lr, lc);
        int s = 0;  // the blocks of its owner before it, row by row: every seventh of a row
        for (int i = 0; i <= lr; ++i) {
            const int first = (own - 1 + 2 * kSpdMaxBlocks * (C - 1) - i) % (C - 1), end = i < lr ? i + 1 : lc;
            if (first < end) s += (end - 1 - first) / (C - 1) + 1;
        }
        s_slot[lr][lc] = (unsigned char)s;
        if (own == q) {
            s_i[s] = (unsigned char)lr;
            s_j[s] = (unsigned char)lc;
            atomicAdd(&s_n, 1);
        }
    }
    __syncthreads();
    // element (r, c) of block (i, j), from the lower triangle; the identity past
    // the matrix' edge
    auto entry = [&](int i, int j, int r, int c) {
        const int gi = kSpdB * i + r, gj = kSpdB * j + c;
        return max(gi, gj) < n ? A[(size_t)max(gi, gj) * n + min(gi, gj)] : (gi == gj ? 1.0 : 0.0);
    };
    const int owned = q > 0 ? s_n : 0;
    for (int s = 0; s < owned; ++s) blk[s * kSpdBlk + lr * kSpdLd + lc] = entry(s_i[s], s_j[s], lr, lc);
    if (q == 0) e[0][lr * kSpdLd + lc] = entry(0, 0, lr, lc);
    __syncthreads();
    for (int p = 0; p < nb; ++p) {
        if (q == 0 && tid < 128) spd_diag(e, blk + p * kSpdBlk, dv + kSpdB * p, &s_fail);
        if (nb == 1) break;
        // CTA 0 arrived at the barrier in the middle of panel p - 1 long ago
        if (q == 0 && p > 0) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        cl.sync();  // W_pp and 1 / D_p are published, every product of panel p - 1 is done
        if (q == 0) {
            if (p + 1 == nb) break;
            // the next diagonal block without waiting for the workers: its blocks
            // A_{p+1,p} and A_{p+1,p+1} as they left them, Q and P of the first
            // and A_{p+1,p+1} - P Q^T, formed here
            const double a0 = cl.map_shared_rank(blk, spd_owner<C>(p + 1, p))[s_slot[p + 1][p] * kSpdBlk + lr * kSpdLd + lc];
            const double a1 =
                cl.map_shared_rank(blk, spd_owner<C>(p + 1, p + 1))[s_slot[p + 1][p + 1] * kSpdBlk + lr * kSpdLd + lc];
            op[lr * kSpdLd + lc] = a0;
            e[1][lr * kSpdLd + lc] = a1;
            __syncthreads();
            asm volatile("barrier.cluster.arrive.release;" ::: "memory");  // they may overwrite A_{p+1,p}
            const double *lin = blk + p * kSpdBlk;
            double v = 0.0;
#pragma unroll 4
            for (int k = 0; k < 2 * pr + 2; ++k) v = fma(op[py * kSpdLd + k], lin[px * kSpdLd + k], v);
            double *Q = op + kSpdBlk, *P = op + 2 * kSpdBlk;
            Q[py * kSpdLd + px] = v;
            P[py * kSpdLd + px] = v * dv[kSpdB * p + px];
            __syncthreads();
            // the 136 entries of the lower triangle on five warps
            if (tid < 136) {
                int r = (int)((sqrtf(8.f * tid + 1.f) - 1.f) * 0.5f);
                while ((r + 1) * (r + 2) / 2 <= tid) ++r;
                while (r * (r + 1) / 2 > tid) --r;
                const int c = tid - r * (r + 1) / 2;
                double w = e[1][r * kSpdLd + c];
#pragma unroll
                for (int k = 0; k < kSpdB; ++k) w = fma(-P[r * kSpdLd + k], Q[c * kSpdLd + k], w);
                e[0][r * kSpdLd + c] = w;
                e[0][c * kSpdLd + r] = w;  // the elimination reads row k right of the diagonal
            }
            __syncthreads();
            continue;
        }
        {
            // W_pp and 1 / D_p here, then Q_i = A_ip W_pp^T, P_i = Q_i / D_p of the
            // column's blocks and W_pj = W_pp X_pj of the row's
            double *lin = op;
            lin[lr * kSpdLd + lc] = cl.map_shared_rank(blk, 0)[p * kSpdBlk + lr * kSpdLd + lc];
            if (tid < kSpdB) dv[tid] = cl.map_shared_rank(dv, 0)[kSpdB * p + tid];
            if (tid == 0 && p + 1 == nb) s_fail = *cl.map_shared_rank(&s_fail, 0);
            __syncthreads();
            for (int s = 0; s < owned; ++s) {
                const int i = s_i[s], j = s_j[s];
                double *b = blk + s * kSpdBlk;
                if (j == p && i > p) {
                    double v = 0.0;
#pragma unroll 4
                    for (int k = 0; k < 2 * pr + 2; ++k) v = fma(b[py * kSpdLd + k], lin[px * kSpdLd + k], v);
                    double *o = pub + 2 * ((i - p - 1) / (C - 1)) * kSpdBlk;
                    o[py * kSpdLd + px] = v;
                    o[kSpdBlk + py * kSpdLd + px] = v * dv[px];
                } else if (i == p && j < p) {
                    double v = 0.0;
#pragma unroll 4
                    for (int k = 0; k < 2 * pr + 2; ++k) v = fma(lin[px * kSpdLd + k], b[k * kSpdLd + py], v);
                    __syncthreads();
                    b[px * kSpdLd + py] = v;
                }
            }
        }
        if (p + 1 == nb) break;
        cl.sync();  // Q, P and row p of W are published
        // address of Q_i (P_i one block on)
        auto qp = [&](int i) {
            return cl.map_shared_rank(pub, spd_owner<C>(i, p)) + 2 * ((i - p - 1) / (C - 1)) * kSpdBlk;
        };
        const int le = lr * kSpdLd + lc;
        {
            // block (i, j) -= P_i Q_j^T (j > p), P_i W_pj (j <= p; the block starts
            // from zero at j = p); the operands of the next block are fetched
            // during the products of this one
            auto active = [&](int s) {
                return s < owned && s_i[s] > p && !(s_i[s] == p + 1 && s_j[s] == p + 1);
            };
            auto next = [&](int s) {
                while (s < owned && !active(s)) ++s;
                return s;
            };
            double f0 = 0.0, f1 = 0.0;
            auto fetch = [&](int s) {
                const int i = s_i[s], j = s_j[s];
                f0 = qp(i)[kSpdBlk + le];
                const double *b = j > p ? qp(j)
                                        : j < p ? cl.map_shared_rank(blk, spd_owner<C>(p, j)) + s_slot[p][j] * kSpdBlk
                                                : cl.map_shared_rank(blk, 0) + p * kSpdBlk;
                f1 = b[le];
            };
            int s = next(0), w = 0;
            if (s < owned) fetch(s);
            while (s < owned) {
                double *o = op + 2 * w * kSpdBlk;
                o[le] = f0;
                o[kSpdBlk + le] = f1;
                __syncthreads();
                const int t = next(s + 1);
                if (t < owned) fetch(t);
                double *b = blk + s * kSpdBlk + ur * kSpdLd + uc;
                double v = s_j[s] == p ? 0.0 : *b;
                if (s_j[s] > p) {
#pragma unroll
                    for (int k = 0; k < kSpdB; ++k) v = fma(-o[ur * kSpdLd + k], o[kSpdBlk + uc * kSpdLd + k], v);
                } else {
#pragma unroll
                    for (int k = 0; k < kSpdB; ++k) v = fma(-o[ur * kSpdLd + k], o[kSpdBlk + k * kSpdLd + uc], v);
                }
                *b = v;
                s = t;
                w ^= 1;
            }
        }
    }
    __syncthreads();
    if (!s_fail) {
        // W below the diagonal and its transpose, 1 / D on the diagonal of A
        auto put = [&](const double *b, int i, int j, bool diag) {
            const int gi = kSpdB * i + lr, gj = kSpdB * j + lc;
            if (gi < n && gj < n && (!diag || lc < lr)) A[(size_t)gi * n + gj] = b[lr * kSpdLd + lc];
            const int ti = kSpdB * i + lc, tj = kSpdB * j + lr;  // lanes along a row of At
            if (ti < n && tj < n && (!diag || lr < lc)) At[(size_t)tj * n + ti] = b[lc * kSpdLd + lr];
        };
        if (q == 0) {
            for (int p = 0; p < nb; ++p) {
                put(blk + p * kSpdBlk, p, p, true);
                const int gi = kSpdB * p + tid;
                if (tid < kSpdB && gi < n) A[(size_t)gi * n + gi] = dv[kSpdB * p + tid];
            }
        } else {
            for (int s = 0; s < owned; ++s)
                if (s_i[s] != s_j[s]) put(blk + s * kSpdBlk, s_i[s], s_j[s], false);
        }
    }
    if (nb > 1) cl.sync();  // no CTA leaves while another may still read its shared memory
    if (q == 0 && tid == 0 && s_fail) atomicCAS(status, 0, MGENKF_ERR_NOT_SPD);
}

// acc[c] += sum of M[k n + i] v[c][k] over k = k0, k0 + step, .. < end where
// take(k), eight loads in flight ahead of the products
template <int NCOL, class Take>
__device__ __forceinline__ void spd_dot(const double *__restrict__ M, const double (&v)[NCOL][kSpdMax], int n, int i,
                                        int k0, int end, int step, Take take, double (&acc)[NCOL]) {
    constexpr int B = 8;
    double w[B], wn[B];
    auto load = [&](int k, double(&d)[B]) {
#pragma unroll
        for (int q = 0; q < B; ++q) {
            const int kq = k + q * step;
            d[q] = kq < end && take(kq) ? __ldg(M + (size_t)kq * n + i) : 0.0;
        }
    };
    load(k0, w);
    for (int k = k0; k < end; k += B * step) {
        load(k + B * step, wn);
#pragma unroll
        for (int q = 0; q < B; ++q)
            if (k + q * step < end) {
#pragma unroll
                for (int c = 0; c < NCOL; ++c) acc[c] = fma(w[q], v[c][k + q * step], acc[c]);
            }
#pragma unroll
        for (int q = 0; q < B; ++q) w[q] = wn[q];
    }
}

// x_c = W^T D^-1 W rhs_c for the columns c0 .. c0 + NCOL - 1 (of ncol; each n
// values, contiguous; x over rhs is allowed), W and D as spd_factor_body left
// them.  A thread owns a row and one of G interleaved shares of the sum over k;
// with two shares the second takes the rows' warps in reverse, so that every
// sub-partition gets the same part of the triangle.
template <int NCOL>
__device__ __forceinline__ void spd_apply_body(const double *__restrict__ A, const double *__restrict__ At, int n,
                                               const double *rhs, double *out, int ncol, __nv_bfloat16 *out16,
                                               int ld16, const int *status, int c0) {
    __shared__ double s_b[NCOL][kSpdMax], s_z[NCOL][kSpdMax], s_part[NCOL][kSpdThreads];
    if (*status) return;
    const int tid = threadIdx.x, nr = (n + 31) & ~31, G = kSpdThreads / nr, nw = nr >> 5;
    const int g = tid / nr, wv = (tid - g * nr) >> 5, wr = g & 1 ? nw - 1 - wv : wv;
    const int i = wr * 32 + (tid & 31);
    const bool act = g < G, row = act && i < n;
    for (int q = tid; q < NCOL * n; q += kSpdThreads) {
        const int c = q / n, k = q - c * n;
        s_b[c][k] = c0 + c < ncol ? rhs[(size_t)(c0 + c) * n + k] : 0.0;
    }
    __syncthreads();
    double acc[NCOL];
#pragma unroll
    for (int c = 0; c < NCOL; ++c) acc[c] = 0.0;
    if (act) {
        spd_dot<NCOL>(At, s_b, n, i, g, min(n, 32 * (wr + 1)), G, [&](int k) { return row && k < i; }, acc);
#pragma unroll
        for (int c = 0; c < NCOL; ++c) s_part[c][g * nr + i] = acc[c];
    }
    __syncthreads();
    for (int q = tid; q < NCOL * n; q += kSpdThreads) {
        const int c = q / n, k = q - c * n;
        double z = s_b[c][k];
        for (int h = 0; h < G; ++h) z += s_part[c][h * nr + k];
        s_z[c][k] = z * A[(size_t)k * n + k];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NCOL; ++c) acc[c] = 0.0;
    if (act) {
        spd_dot<NCOL>(A, s_z, n, i, 32 * wr + g, n, G, [&](int k) { return row && k > i; }, acc);
#pragma unroll
        for (int c = 0; c < NCOL; ++c) s_part[c][g * nr + i] = acc[c];
    }
    __syncthreads();
    for (int q = tid; q < NCOL * n; q += kSpdThreads) {
        const int c = q / n, k = q - c * n;
        if (c0 + c >= ncol) continue;
        double x = s_z[c][k];
        for (int h = 0; h < G; ++h) x += s_part[c][h * nr + k];
        out[(size_t)(c0 + c) * n + k] = x;
        if (out16) out16[(size_t)(c0 + c) * ld16 + k] = __double2bfloat16(x);
    }
}

}  // namespace mgk
