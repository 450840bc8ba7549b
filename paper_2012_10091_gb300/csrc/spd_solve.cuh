// spd_solve.cuh -- FP64 solve of a small SPD system with many right-hand sides
// (the gain solve, Algorithm 3 step 8), device bodies shared by the launches
// over one problem and over many.
//
// GB300 issues one FP64 instruction of a warp per SM sub-partition in 64 cycles,
// whatever its lanes do, and with no further latency: a step that depends on
// the previous one costs its FP64 instructions, and work costs its warp
// instructions divided by the sub-partitions it is spread over.  So
//   * the factorisation S = L D L^T (unit L) runs on a cluster of C CTAs.  The
//     matrix is cut into 16 x 16 blocks; CTA 0 does nothing but the serial chain
//     (the diagonal blocks), the others own the blocks of the lower triangle and
//     do the products.  Every row is eliminated pivot by pivot, in blocks too:
//     with the inverses of the diagonal blocks (or of L, in place of the
//     substitutions) the solves of few observations and of smooth ensembles
//     were 1.6 to 4.5 times further from extended precision, this is within 1.1
//     of a plain Cholesky solve (64 to 128 members, conditions up to 1e12);
//   * the solves are substitutions by blocks, a column per CTA over the whole
//     GPU: a warp takes the 16 pivots of a block through the block's rows and the
//     next block's, the others apply the block before to the rows behind.
// Measured back to back, n = 128 (129 columns): Cholesky by column panels on eight
// CTAs and one warp of substitution per column 150 + 43 us, this 70 + 23 (with the
// inverse of L instead 71 + 17); n = 64: 62 + 22 and 37 + 13 us (36 + 8).  The chain
// bounds the factorisation: about 600 cycles per pivot (five dependent FP64
// instructions, a barrier, shared-memory latency) and 7 k per panel for the blocks
// that lead to the next diagonal block.
#pragma once

#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

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
// (n = 100: 61 us with 8 and 63 with 16, 112: 63 and 62, 160: 97 and 89, 256: 245
// and 166).
constexpr int kSpdGroupCluster = 8;
constexpr int spd_cluster(int n) { return n > 112 ? 16 : 8; }

// the worker that owns block (i, j), j <= i: 1 .. C - 1.  Within a column (and a
// row) consecutive blocks have different owners.
template <int C>
__device__ __forceinline__ int spd_owner(int i, int j) {
    return 1 + (i + j) % (C - 1);
}
// block slots per CTA for nb block rows: a worker owns at most i / (C - 1) + 1
// blocks of row i; CTA 0 keeps the nb diagonal blocks of L and its two work blocks
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

// 1 / d of a pivot.  A pivot that is not positive and finite raises *fail and
// yields 1, so that the factorisation runs on.
__device__ __forceinline__ double spd_pivot(double d, int *fail) {
    // comparisons of doubles would take the FP64 pipe (64 cycles each): one test of
    // the high word on the chain, sign included
    if (!recip64_range(d) || __double2hiint(d) < 0) {
        if (!(d > 0.0) || !isfinite(d)) {
            *fail = 1;
            return 1.0;
        }
        return 1.0 / d;
    }
    return recip64_in_range(d);
}

// A diagonal block by warps 0-3 (128 threads): e[0] holds it (both triangles);
// its unit lower factor into `lpp` (below the diagonal, zeros elsewhere) and
// 1 / D into `dinv`.  Pivot k takes one barrier: warp 0 updates the next
// diagonal entry by itself and forms its reciprocal (two and three dependent
// FP64 instructions, the chain) while warps 1-3, on the other three
// sub-partitions, eliminate column k from the rows below in one of two buffers.
__device__ __forceinline__ void spd_diag(double (*e)[kSpdBlk], double *lpp, double *dinv, int *fail) {
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
            // element (r, c), c = g, g + 6, g + 12, of a row below the pivot: the
            // multiplier at c = k, the reduced matrix right of it
            const double l = cur[r * kSpdLd + k] * y;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int c = g + 6 * q;
                if (c < kSpdB) {
                    double v = cur[r * kSpdLd + c];
                    if (r > k && c >= k) v = c == k ? l : fma(-l, cur[k * kSpdLd + c], v);
                    nxt[r * kSpdLd + c] = v;
                }
            }
        }
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    for (int q = tid; q < kSpdB * kSpdB; q += 128) {
        const int r = q >> 4, c = q & 15;
        lpp[r * kSpdLd + c] = r > c ? e[0][r * kSpdLd + c] : 0.0;
    }
}

// Q = A L_pp^-T and P = Q / D of a block below the diagonal block (the thread's
// element, half a warp per row), pivot by pivot
__device__ __forceinline__ void spd_panel(const double *a, const double *lpp, const double *dinv, double *Q, double *P) {
    const int r = threadIdx.x >> 4, c = threadIdx.x & 15;
    double v = a[r * kSpdLd + c];
#pragma unroll
    for (int k = 0; k + 1 < kSpdB; ++k) {
        const double q = __shfl_sync(0xffffffffu, v, k, 16);
        const double w = fma(-q, lpp[c * kSpdLd + k], v);
        v = c > k ? w : v;
    }
    Q[r * kSpdLd + c] = v;
    P[r * kSpdLd + c] = v * dinv[c];
}

// S (n x n row-major, lower triangle read) -> A: L below the diagonal, 1 / D on
// it; At: the transpose of L above its diagonal.  A pivot that is not positive and
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
    double *blk = spd_sm;                        // worker: its blocks; CTA 0: L_pp of every panel, then e[2]
    double *pub = blk + slots * kSpdBlk;         // worker: Q, P of its blocks of the panel's column
    double *op = pub + 6 * kSpdBlk;              // two pairs of operands
    double *dv = op + 4 * kSpdBlk;               // CTA 0: 1 / D of every panel; worker: of the current one
    double(*e)[kSpdBlk] = reinterpret_cast<double(*)[kSpdBlk]>(blk + nb * kSpdBlk);
    const int lr = tid >> 4, lc = tid & 15;      // element in row order (loads, stores)
    const int ur = tid & 15, uc = tid >> 4;      // element of a product: a warp has all rows of two columns
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
        cl.sync();  // L_pp and 1 / D_p are published, every product of panel p - 1 is done
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
            double *Q = op + kSpdBlk, *P = op + 2 * kSpdBlk;
            spd_panel(op, blk + p * kSpdBlk, dv + kSpdB * p, Q, P);
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
            // L_pp and 1 / D_p here, then Q_i = A_ip L_pp^-T and P_i = Q_i / D_p = L_ip
            // of the column's blocks
            double *lpp = op;
            lpp[lr * kSpdLd + lc] = cl.map_shared_rank(blk, 0)[p * kSpdBlk + lr * kSpdLd + lc];
            if (tid < kSpdB) dv[tid] = cl.map_shared_rank(dv, 0)[kSpdB * p + tid];
            if (tid == 0 && p + 1 == nb) s_fail = *cl.map_shared_rank(&s_fail, 0);
            __syncthreads();
            for (int s = 0; s < owned; ++s)
                if (s_j[s] == p && s_i[s] > p) {
                    double *o = pub + 2 * ((s_i[s] - p - 1) / (C - 1)) * kSpdBlk;
                    spd_panel(blk + s * kSpdBlk, lpp, dv, o, o + kSpdBlk);
                }
        }
        if (p + 1 == nb) break;
        cl.sync();  // Q and P are published, CTA 0 has read A_{p+1,p}
        // address of Q_i (P_i one block on)
        auto qp = [&](int i) {
            return cl.map_shared_rank(pub, spd_owner<C>(i, p)) + 2 * ((i - p - 1) / (C - 1)) * kSpdBlk;
        };
        const int le = lr * kSpdLd + lc;
        {
            for (int s = 0; s < owned; ++s)
                if (s_j[s] == p && s_i[s] > p)
                    blk[s * kSpdBlk + le] = pub[(2 * ((s_i[s] - p - 1) / (C - 1)) + 1) * kSpdBlk + le];
            // block (i, j) -= P_i Q_j^T; the operands of the next block are fetched
            // during the products of this one
            auto active = [&](int s) {
                return s < owned && s_j[s] > p && !(s_i[s] == p + 1 && s_j[s] == p + 1);
            };
            auto next = [&](int s) {
                while (s < owned && !active(s)) ++s;
                return s;
            };
            double f0 = 0.0, f1 = 0.0;
            auto fetch = [&](int s) {
                f0 = qp(s_i[s])[kSpdBlk + le];
                f1 = qp(s_j[s])[le];
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
                double v = *b;
#pragma unroll
                for (int k = 0; k < kSpdB; ++k) v = fma(-o[ur * kSpdLd + k], o[kSpdBlk + uc * kSpdLd + k], v);
                *b = v;
                s = t;
                w ^= 1;
            }
        }
    }
    __syncthreads();
    if (!s_fail) {
        // L below the diagonal and its transpose, 1 / D on the diagonal of A
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

// Threads of a CTA that solves for one column of order n: a warp for the chain
// and a thread per row past the first (forward) or before the last (backward)
// two blocks, on warps of the other three sub-partitions.
inline int spd_apply_threads(int n) {
    const int rows = (n + kSpdB - 1) / kSpdB * kSpdB - 2 * kSpdB;
    return 128 * (rows <= 96 ? 1 : (rows + 95) / 96);
}

// a where bit k of m is set, else b, on the words' bits (16 predicates alive at
// once are more than there are)
__device__ __forceinline__ double spd_select(unsigned m, int k, double a, double b) {
    const int t = (int)(m << (31 - k)) >> 31;
    return __hiloint2double((__double2hiint(a) & t) | (__double2hiint(b) & ~t),
                            (__double2loint(a) & t) | (__double2loint(b) & ~t));
}

// x = L^-T D^-1 L^-1 rhs of one column (n contiguous values; x over rhs is
// allowed), L and D as spd_factor_body left them, 128 threads or more as
// spd_apply_threads says.  Step p, one barrier each: warp 0 takes the pivots of
// block p one by one through the rows of block p (a half of its lanes) and of the
// next one (the other half, from zero: added to the rest of their sums when the
// next step begins and the halves change places); the other warps meanwhile
// apply the pivots of the step before to the rows behind the next block.  Bound
// by the chain, a shuffle and an FMA (117 cycles) per pivot, so the elements of L
// for the next step are loaded between its steps.
__device__ __forceinline__ void spd_apply_body(const double *__restrict__ A, const double *__restrict__ At, int n,
                                               const double *rhs, double *out, __nv_bfloat16 *out16,
                                               const int *status) {
    constexpr int B = kSpdB;
    __shared__ double s_v[kSpdMax], s_z[2][B];
    if (*status) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nb = (n + B - 1) / B;
    const bool lead = warp == 0;
    // the rows of the other warps, from the first one they serve; none on warp 0's sub-partition
    const int u = (warp & 3) ? ((warp >> 2) * 3 + (warp & 3) - 1) * 32 + lane : kSpdMax;
    for (int k = tid; k < nb * B; k += blockDim.x) s_v[k] = k < n ? rhs[k] : 0.0;
    const double d = tid < n ? A[(size_t)tid * n + tid] : 0.0;  // n <= blockDim.x
    // the elements of a step, L[row][cb + k] of a row below or L[cb + k][row] of one
    // above, in one of two sets; loads without branches (a divergent one costs
    // more than it saves): past the edge they repeat the last row or column, and
    // are not used
    double la[B], lb[B];
    const double *src = nullptr;
    int kmax = 0;
    auto from = [&](const double *M, int row, int cb) {
        kmax = min(B, n - cb) - 1;
        src = M + (size_t)cb * n + min(max(row, 0), n - 1);
    };
    auto load = [&](double(&l)[B], int k) { l[k] = __ldg(src + min(k, kmax) * n); };
    auto load_all = [&](double(&l)[B]) {
#pragma unroll
        for (int k = 0; k < B; ++k) load(l, k);
    };
    // the pivots of the step before on this thread's row (zeros past the edge)
    auto apply = [&](const double(&l)[B], const double *z, double v) {
#pragma unroll
        for (int k = 0; k < B; ++k) v = fma(-l[k], z[k], v);
        return v;
    };
    const int rf = 2 * B + u;  // forward row
    from(At, lead ? lane : rf, 0);
    if (lead)
        load_all(la);
    else
        load_all(lb);
    __syncthreads();
    double v = 0.0;
    if (!lead && rf < n) v = s_v[rf];
    // step p with l, ln: the other set, for the next step; T: 16 in odd steps
    auto forward = [&](auto T_, int p, const double(&l)[B], double(&ln)[B]) {
        constexpr int T = decltype(T_)::value;
        if (lead) {
            const int i = lane ^ T;  // lanes i < 16: block p, others: the next one
            // bit k: pivot k is applied to this row
            const unsigned m = B * p + i >= n ? 0u : i < B ? (1u << i) - 1u : 0xffffu;
            v = i < B ? s_v[B * p + i] + v : 0.0;
            if (p + 1 < nb) from(At, B * p + (i < B ? i + 2 * B : i), B * (p + 1));
#pragma unroll
            for (int k = 0; k < B; ++k) {
                const double z = __shfl_sync(0xffffffffu, v, k ^ T);
                load(ln, k);
                v = spd_select(m, k, fma(-l[k], z, v), v);
            }
            if (i < B) {
                s_z[p & 1][i] = v;
                s_v[B * p + i] = v;
            }
        } else if (p > 0 && rf < n && rf >= B * (p + 1)) {
            from(At, rf, B * p);
            load_all(ln);
            v = apply(l, s_z[(p - 1) & 1], v);
            if (rf < B * (p + 2)) s_v[rf] = v;
        }
        __syncthreads();
    };
    for (int p = 0; p < nb; p += 2) {
        forward(std::integral_constant<int, 0>{}, p, la, lb);
        if (p + 1 < nb) forward(std::integral_constant<int, B>{}, p + 1, lb, la);
    }
    from(A, lead ? B * (nb - 1) + (lane < B ? lane : lane - 2 * B) : u, B * (nb - 1));
    if (lead)
        load_all(la);
    else
        load_all(lb);
    if (tid < n) s_v[tid] *= d;
    __syncthreads();
    v = !lead && u < B * (nb - 2) ? s_v[u] : 0.0;
    auto backward = [&](auto T_, int p, const double(&l)[B], double(&ln)[B]) {
        constexpr int T = decltype(T_)::value;
        if (lead) {
            const int i = lane ^ T;  // lanes i < 16: block p, others: the one before
            const unsigned m = (i < B ? 0xfffeu << i : p > 0 ? 0xffffu : 0u) & ((1u << min(B, n - B * p)) - 1u);
            v = i < B ? s_v[B * p + i] + v : 0.0;
            if (p > 0) from(A, B * p + i - 2 * B, B * (p - 1));
#pragma unroll
            for (int k = B - 1; k >= 0; --k) {
                const double x = __shfl_sync(0xffffffffu, v, k ^ T);
                load(ln, k);
                v = spd_select(m, k, fma(-l[k], x, v), v);
            }
            if (i < B) {
                s_z[p & 1][i] = v;
                if (B * p + i < n) {
                    out[B * p + i] = v;
                    if (out16) out16[B * p + i] = __double2bfloat16(v);
                }
            }
        } else if (p + 1 < nb && u < B * p) {
            from(A, u, B * p);
            load_all(ln);
            v = apply(l, s_z[(p + 1) & 1], v);
            if (u >= B * (p - 1)) s_v[u] = v;
        }
        __syncthreads();
    };
    for (int p = nb - 1; p >= 0; p -= 2) {
        backward(std::integral_constant<int, 0>{}, p, la, lb);
        if (p > 0) backward(std::integral_constant<int, B>{}, p - 1, lb, la);
    }
}

}  // namespace mgk
