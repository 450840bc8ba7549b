// analysis.cu -- kernels of the coarse-mesh EnKF analysis (Algorithm 3, state
// part: steps 2-3, 7-8) and of the multigrid correction (Algorithm 4 steps 4-5).
//
// Layout (per analysis): members [ne][nx] (member-major, state vector of one
// member contiguous), predicted observations yf [ne+1][ny] (row ne = H^C x^C*),
// anomalies Y [ne][ny], innovations Z [ne+1][ny] (row i = y^o + eps_i - yf_i,
// row ne = y^o - H^C x^C*), gain coefficients T [(ne+1)][ne] (column c of
// T = Y^T C^-1 [D | d*] contiguous).  Every covariance-type reduction, the
// Cholesky factorisation and the triangular solves run in FP64.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <type_traits>
#include <vector>

#include "analysis.h"
#include "batch_analysis.h"
#include "common.cuh"
#include "spd_solve.cuh"
#include "update_tc.h"

namespace mgk {

static inline int grid_for(size_t n, int block, int cap = 8 * kNumSMs) {
    long long g = (long long)((n + block - 1) / block);
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

// ---------------------------------------------------------------------------
// restriction Pi_C (injection), Algorithm 4 step 4
// ---------------------------------------------------------------------------
// Kernel bodies take their block index and block count as arguments, so that
// the grouped analysis of many problems (one launch per step, blocks mapped to
// problems by a table) runs the same per-element arithmetic as one handle.
template <typename T>
__device__ __forceinline__ void restrict_body(const T *__restrict__ fine, T *__restrict__ xs, int dim, int V,
                                              int nc, int r, size_t blk, size_t nblk, T *__restrict__ zero) {
    const size_t nf = (size_t)nc * r;
    const size_t cpl = dim == 1 ? (size_t)nc : (size_t)nc * nc;
    const size_t fpl = dim == 1 ? nf : nf * nf;
    const size_t total = (size_t)V * cpl;
    for (size_t i = blk * blockDim.x + threadIdx.x; i < total; i += nblk * blockDim.x) {
        const size_t v = i / cpl, k = i % cpl;
        size_t src;
        if (dim == 1) {
            src = (size_t)r * k;
        } else {
            const size_t jy = k / nc, jx = k % nc;
            src = (size_t)r * jy * nf + (size_t)r * jx;
        }
        xs[i] = fine[v * fpl + src];
        if (zero) zero[i] = T(0);  // the coarse correction, cleared before the analysis writes it
    }
}

template <typename T>
__global__ void k_restrict(const T *__restrict__ fine, T *__restrict__ xs, int dim, int V, int nc, int r) {
    launch_wait();
    restrict_body<T>(fine, xs, dim, V, nc, r, blockIdx.x, gridDim.x, nullptr);
}

template <typename T>
void launch_restrict(const T *fine, T *xstar, int dim, int V, int nc, int r, cudaStream_t s) {
    count_launches(1);
    const size_t total = (size_t)V * (dim == 1 ? (size_t)nc : (size_t)nc * nc);
    launch_kernel(k_restrict<T>, grid_for(total, 256), 256, 0, s, LaunchHow{}, fine, xstar, dim, V, nc, r);
}

// ---------------------------------------------------------------------------
// predicted observations H^C x (Algorithm 3 step 2): sparse 4- or 16-tap rows
// ---------------------------------------------------------------------------
// Thread: observation j = bx * blockDim.x + threadIdx.x, rows i = i0 .. i0 +
// rows - 1 of yf (members, then x^C* as row ne); its taps (<= 16) stay in
// registers for those rows, loaded 16 bytes at a time (the rows of the tables are
// 16 or 64 bytes: scalar loads of a warp touched 32 segments each).  One problem
// alone takes a row per thread (enough threads to hide the gathers; two rows
// with scalar loads: NS analysis of 64 members and 2048 observations 185 us, 179
// with 16-byte loads, 176 with one row); a grouped launch over many problems 8.
constexpr int kObsRows = 8, kObsRowsOne = 1;

// a 16-byte load of consecutive values (the tap rows are 4 or 16 long and start at
// the beginning of their buffers)
template <class V, class S>
__device__ __forceinline__ void load_vec(const S *p, S *out) {
    const V v = __ldg(reinterpret_cast<const V *>(p));
    memcpy(out, &v, sizeof(V));
}

// With FP32 states and the weights split into FP32 pairs (wh, wl: w = wh + wl
// up to 2^-48 |w|, mixed precision) the taps are summed in double-FP32
// arithmetic on the FP32 pipes: wh x exactly as p + e (e by FMA), wl x
// rounded, the products summed into a running FP32 sum and the FP32 sum of its
// rounding errors (error-free two-sum); otherwise in FP64.
template <typename T>
__device__ __forceinline__ void obs_apply_body(const T *__restrict__ members, const T *__restrict__ xstar,
                                               size_t nx, int ne, int ny, int taps,
                                               const int32_t *__restrict__ tap_idx,
                                               const double *__restrict__ tap_w, double *__restrict__ yf, int bx,
                                               int i0, int rows, const float *__restrict__ wh = nullptr,
                                               const float *__restrict__ wl = nullptr) {
    const int j = bx * blockDim.x + threadIdx.x;
    if (j >= ny) return;
    int32_t idx[16];
    const int i1 = min(i0 + rows, ne + 1);
    if constexpr (std::is_same<T, float>::value) {
        if (wh) {
            float w1[16], w2[16];
#pragma unroll
            for (int t = 0; t < 16; t += 4)
                if (t < taps) {
                    const size_t o = (size_t)j * taps + t;
                    load_vec<int4>(tap_idx + o, idx + t);
                    load_vec<float4>(wh + o, w1 + t);
                    load_vec<float4>(wl + o, w2 + t);
                }
            for (int i = i0; i < i1; ++i) {
                const float *x = i < ne ? members + (size_t)i * nx : xstar;
                float s = 0.f, c = 0.f;
#pragma unroll
                for (int t = 0; t < 16; ++t)
                    if (t < taps) {
                        const float xv = x[idx[t]];
                        const float p = __fmul_rn(w1[t], xv), e = __fmaf_rn(w1[t], xv, -p);
                        const float q = __fmul_rn(w2[t], xv);
                        const float u = __fadd_rn(s, p), bv = __fsub_rn(u, s);
                        c = __fadd_rn(c, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(u, bv)), __fsub_rn(p, bv)),
                                                   __fadd_rn(e, q)));
                        s = u;
                    }
                yf[(size_t)i * ny + j] = (double)s + (double)c;
            }
            return;
        }
    }
    double w[16];
#pragma unroll
    for (int t = 0; t < 16; t += 4)
        if (t < taps) {
            const size_t o = (size_t)j * taps + t;
            load_vec<int4>(tap_idx + o, idx + t);
            load_vec<double2>(tap_w + o, w + t);
            load_vec<double2>(tap_w + o + 2, w + t + 2);
        }
    for (int i = i0; i < i1; ++i) {
        const T *x = i < ne ? members + (size_t)i * nx : xstar;
        double acc = 0.0;
#pragma unroll
        for (int t = 0; t < 16; ++t)
            if (t < taps) acc = fma(w[t], (double)x[idx[t]], acc);
        yf[(size_t)i * ny + j] = acc;
    }
}

template <typename T>
__global__ void __launch_bounds__(128) k_obs_apply(const T *__restrict__ members, const T *__restrict__ xstar,
                                                   size_t nx, int ne, int ny, int taps,
                                                   const int32_t *__restrict__ tap_idx,
                                                   const double *__restrict__ tap_w, double *__restrict__ yf,
                                                   const float *__restrict__ wh, const float *__restrict__ wl) {
    launch_wait();
    obs_apply_body<T>(members, xstar, nx, ne, ny, taps, tap_idx, tap_w, yf, blockIdx.x, blockIdx.y * kObsRowsOne,
                      kObsRowsOne, wh, wl);
}

template <typename T>
void launch_obs_apply(const T *members, const T *xstar, size_t nx, int ne, int ny, int taps,
                      const int32_t *tap_idx, const double *tap_w, double *yf, cudaStream_t s, const float *wh,
                      const float *wl) {
    count_launches(1);
    dim3 grid(ceil_div(ny, 128), ceil_div(ne + 1, kObsRowsOne));
    launch_kernel(k_obs_apply<T>, grid, 128, 0, s, LaunchHow{}, members, xstar, nx, ne, ny, taps, tap_idx, tap_w, yf,
                  wh, wl);
}

// ---------------------------------------------------------------------------
// observation means and innovations (Algorithm 1 step 4; Algorithm 4 step 5)
// ---------------------------------------------------------------------------
// x = hi[o] + lo[o] up to 2^-48 |x|: hi = x rounded to FP32, lo = the
// remainder (exact in FP64) rounded to FP32.  The operands of the
// double-FP32 gain products (mixed precision).
__device__ __forceinline__ void split_df(double x, float *__restrict__ hi, float *__restrict__ lo, size_t o) {
    const float h = __double2float_rn(x);
    hi[o] = h;
    lo[o] = __double2float_rn(__dsub_rn(x, (double)h));
}

// yo_copy (if not NULL) receives y^o as read; Zh, Zl (if not NULL) the
// double-FP32 split of row ne of Z
__device__ __forceinline__ void obs_mean_body(const double *__restrict__ yf, const double *__restrict__ yo, int ne,
                                              double inv_ne, int ny, double *__restrict__ ybar,
                                              double *__restrict__ Z, int *status, int blk,
                                              double *__restrict__ yo_copy, float *__restrict__ Zh = nullptr,
                                              float *__restrict__ Zl = nullptr) {
    // 32 observations per CTA (lane), 8 slices of the members (warp); the slice
    // sums are combined in a fixed order.
    __shared__ double part[8][33];
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int j = blk * 32 + lane;
    double acc = 0.0;
    if (j < ny)
        for (int i = slice; i < ne; i += 8) acc += yf[(size_t)i * ny + j];
    part[slice][lane] = acc;
    __syncthreads();
    if (slice == 0 && j < ny) {
        double sum = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) sum += part[q][lane];
        ybar[j] = sum * inv_ne;
        const double y = yo[j];
        if (!isfinite(y)) atomicCAS(status, 0, kStNonFinite);
        if (yo_copy) yo_copy[j] = y;
        const double d = y - yf[(size_t)ne * ny + j];
        Z[(size_t)ne * ny + j] = d;
        if (Zh) split_df(d, Zh, Zl, (size_t)ne * ny + j);
    }
}

__global__ void __launch_bounds__(256) k_obs_mean(const double *__restrict__ yf, const double *__restrict__ yo,
                                                  int ne, double inv_ne, int ny, double *__restrict__ ybar,
                                                  double *__restrict__ Z, int *status, float *__restrict__ Zh,
                                                  float *__restrict__ Zl) {
    launch_wait();
    obs_mean_body(yf, yo, ne, inv_ne, ny, ybar, Z, status, blockIdx.x, nullptr, Zh, Zl);
}

void launch_obs_mean(const double *yf, const double *yo, int ne, int ny, double *ybar, double *Z,
                     int *status, cudaStream_t s, float *Zh, float *Zl) {
    count_launches(1);
    launch_kernel(k_obs_mean, ceil_div(ny, 32), 256, 0, s, LaunchHow{}, yf, yo, ne, 1.0 / ne, ny, ybar, Z, status, Zh,
                  Zl);
}

// RMS of the innovation d* = y^o - H^C x^C* (one value; fixed-order FP64 sums)
__device__ __forceinline__ void innov_rms_body(const double *__restrict__ d, int ny, double *__restrict__ out) {
    __shared__ double part[256];
    double acc = 0.0;
    for (int j = threadIdx.x; j < ny; j += 256) acc = fma(d[j], d[j], acc);
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = sqrt(part[0] / ny);
}

__global__ void __launch_bounds__(256) k_innov_rms(const double *__restrict__ d, int ny, double *__restrict__ out) {
    launch_wait();
    innov_rms_body(d, ny, out);
}

void launch_innov_rms(const double *Z, int ne, int ny, double *out, cudaStream_t s) {
    launch_kernel(k_innov_rms, 1, 256, 0, s, LaunchHow{}, Z + (size_t)ne * ny, ny, out);
    count_launches(1);
}

// perturbed observations (Eq. perturbed_y) and normalised anomalies Y (Algorithm 3 step 7)
// One thread per Philox block, the 4 consecutive elements o = 4b .. 4b + 3 of
// the Ne x Ny perturbation matrix (flat index o = i Ny + j), or (L = 1, CTAs of
// 128 threads) a warp per element of 32 blocks.  gen_eps: 0 = eps given, 1 =
// normals in FP64, 2 = Box-Muller in FP32 (the mixed path).
template <bool F32, int L = 4>
__device__ __forceinline__ void obs_perturb_body(const double *__restrict__ yf, const double *__restrict__ ybar,
                                                 const double *__restrict__ yo, double *__restrict__ eps,
                                                 int gen_eps, uint64_t seed, const uint64_t *__restrict__ cycle,
                                                 double sigma, int ne, int ny, double isq, double *__restrict__ Y,
                                                 double *__restrict__ Z, size_t blk, float *__restrict__ Yh = nullptr,
                                                 float *__restrict__ Yl = nullptr, float *__restrict__ Zh = nullptr,
                                                 float *__restrict__ Zl = nullptr) {
    const size_t total = (size_t)ne * ny;
    const size_t b = L == 1 ? blk * 32 + (threadIdx.x & 31) : blk * blockDim.x + threadIdx.x;
    const size_t o0 = L == 1 ? 4 * b + (threadIdx.x >> 5) : 4 * b;
    if (o0 >= total) return;
    double z[L];
    if (gen_eps) {
        if constexpr (L == 1)
            z[0] = philox_normal1(seed, kEpsTag, *cycle, (uint64_t)b, threadIdx.x >> 5);
        else if constexpr (F32)
            philox_normals4_f32(seed, kEpsTag, *cycle, (uint64_t)b, z);
        else
            philox_normals4(seed, kEpsTag, *cycle, (uint64_t)b, z);
    }
    int i = (int)(o0 / ny), j = (int)(o0 - (size_t)i * ny);
#pragma unroll
    for (int l = 0; l < L; ++l) {
        const size_t o = o0 + l;
        if (o < total) {
            // explicit roundings: no contraction into an FMA, whatever the
            // kernel the body is inlined into
            double e;
            if (gen_eps) {
                e = __dmul_rn(sigma, z[l]);
                eps[o] = e;
            } else {
                e = eps[o];
            }
            const double f = yf[o];
            const double yv = __dmul_rn(__dsub_rn(f, ybar[j]), isq), zv = __dsub_rn(__dadd_rn(yo[j], e), f);
            Y[o] = yv;
            Z[o] = zv;
            if (Yh) {
                split_df(yv, Yh, Yl, o);
                split_df(zv, Zh, Zl, o);
            }
        }
        if (++j == ny) {
            j = 0;
            ++i;
        }
    }
}

template <bool F32, int L>
__global__ void __launch_bounds__(128) k_obs_perturb(const double *__restrict__ yf, const double *__restrict__ ybar,
                              const double *__restrict__ yo, double *__restrict__ eps, int gen_eps, uint64_t seed,
                              const uint64_t *__restrict__ cycle, double sigma, int ne, int ny, double isq,
                              double *__restrict__ Y, double *__restrict__ Z, float *__restrict__ Yh,
                              float *__restrict__ Yl, float *__restrict__ Zh, float *__restrict__ Zl) {
    launch_wait();
    obs_perturb_body<F32, L>(yf, ybar, yo, eps, gen_eps, seed, cycle, sigma, ne, ny, isq, Y, Z, blockIdx.x, Yh, Yl,
                             Zh, Zl);
}

void launch_obs_perturb(const double *yf, const double *ybar, const double *yo, double *eps,
                        int gen_eps, uint64_t seed, const uint64_t *cycle, double sigma, int ne, int ny,
                        double *Y, double *Z, cudaStream_t s, const DfOperands &df) {
    count_launches(1);
    const size_t blocks = ((size_t)ne * ny + 3) / 4;
    // isq = 1/sqrt(Ne - 1) from the host (an FP64 division and square root per thread on the device)
    const unsigned grid = (unsigned)ceil_div(blocks, 128);
    const double isq = 1.0 / std::sqrt((double)(ne - 1));
    if (gen_eps == 2)
        launch_kernel(k_obs_perturb<true, 4>, grid, 128, 0, s, LaunchHow{}, yf, ybar, yo, eps, 1, seed, cycle, sigma, ne,
                      ny, isq, Y, Z, df.Yh, df.Yl, df.Zh, df.Zl);
    else if (gen_eps && single_normals(blocks))
        launch_kernel(k_obs_perturb<false, 1>, ceil_div(blocks, 32), 128, 0, s, LaunchHow{}, yf, ybar, yo, eps,
                      gen_eps, seed, cycle, sigma, ne, ny, isq, Y, Z, df.Yh, df.Yl, df.Zh, df.Zl);
    else
        launch_kernel(k_obs_perturb<false, 4>, grid, 128, 0, s, LaunchHow{}, yf, ybar, yo, eps, gen_eps, seed, cycle,
                      sigma, ne, ny, isq, Y, Z, df.Yh, df.Yl, df.Zh, df.Zl);
}

// Fine-to-coarse feedback: the forecast ensemble re-centred on the restricted
// fine forecast, x^(i) += x^C* - mean_i x^(i) (FP64 mean and shift).  One
// thread per point; members member-major.
template <typename T>
__global__ void __launch_bounds__(256) k_recentre(T *__restrict__ m, size_t nx, int ne, const T *__restrict__ xstar,
                                                  const int *status) {
    launch_wait();
    if (*status) return;
    const size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (p >= nx) return;
    double s = 0.0;
    for (int i = 0; i < ne; ++i) s += (double)m[(size_t)i * nx + p];
    const double shift = (double)xstar[p] - s / ne;
    for (int i = 0; i < ne; ++i) m[(size_t)i * nx + p] = (T)((double)m[(size_t)i * nx + p] + shift);
}

template <typename T>
void launch_recentre(T *members, size_t nx, int ne, const T *xstar, const int *status, cudaStream_t s) {
    count_launches(1);
    launch_kernel(k_recentre<T>, (unsigned)ceil_div(nx, 256), 256, 0, s, LaunchHow{}, members, nx, ne, xstar, status);
}
template void launch_recentre<float>(float *, size_t, int, const float *, const int *, cudaStream_t);
template void launch_recentre<double>(double *, size_t, int, const double *, const int *, cudaStream_t);

// ---------------------------------------------------------------------------
// ensemble mean and normalised anomalies X
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void ens_anom_body(const T *__restrict__ m, size_t nx, int ne, double inv_ne, double isq,
                                              double *__restrict__ X64, __nv_bfloat16 *__restrict__ X16, int ldx,
                                              const int *status, size_t blk) {
    // CTA: 32 consecutive points (lane) x the members split over the 8 warps.
    // Mean: per-warp slice sums combined in a fixed order by warp 0; then the
    // normalised anomalies: FP64 member-major rows, or BF16 point-major rows
    // assembled in shared memory so every row of ldx values is stored
    // contiguously.  GB300 runs about 2 FP64 FMAs per clock per SM, so FP32
    // states are averaged without FP64 operations (below), and 1/Ne and
    // 1/sqrt(Ne - 1) come from the host.
    extern __shared__ __align__(16) unsigned char sm_raw[];
    double *part = reinterpret_cast<double *>(sm_raw);                        // [8][32]
    double *mean = part + 8 * 32;                                             // [32]
    __nv_bfloat16 *tile = reinterpret_cast<__nv_bfloat16 *>(mean + 32);      // [32][ldx + 8]
    if (*status) return;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const size_t p0 = blk * 32;
    const size_t p = p0 + lane;
    const bool ok = p < nx;
    // FP32 states: slice sums in floats [0, 256) of `part`, x_ref and the mean
    // offset per lane in floats [256, 320)
    float *rfm = reinterpret_cast<float *>(part) + 256;
    if constexpr (std::is_same<T, float>::value) {
        // FP32 states: the mean as x_ref + dm, x_ref = member 0's value at the
        // point and dm the mean of the differences x_i - x_ref.  Members at a
        // point lie within a small spread of each other, so the differences
        // are exact (Sterbenz) and their FP32 sum carries an error of order
        // 2^-24 of the spread, not of the state.  Slice q (members q, q + 8,
        // ...) is summed in member order, the 8 slices in slice order (the
        // tensor-core update forms its anomalies with these same operations).
        const float xr = ok ? (float)m[p] : 0.f;
        float ps = 0.f;
        if (ok)
            for (int i = wp; i < ne; i += 8) ps = __fadd_rn(ps, __fsub_rn((float)m[(size_t)i * nx + p], xr));
        float *partf = reinterpret_cast<float *>(part);
        partf[wp * 32 + lane] = ps;
        __syncthreads();
        if (wp == 0) {
            float D = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) D = __fadd_rn(D, partf[q * 32 + lane]);
            const float dm = __fmul_rn(D, (float)inv_ne);
            rfm[lane] = xr;
            rfm[32 + lane] = dm;
            mean[lane] = (double)xr + (double)dm;
        }
    } else {
        double acc = 0.0;
        if (ok)
            for (int i = wp; i < ne; i += 8) acc += (double)m[(size_t)i * nx + p];
        part[wp * 32 + lane] = acc;
        __syncthreads();
        if (wp == 0) {
            double sum = 0.0;
#pragma unroll
            for (int q = 0; q < 8; ++q) sum += part[q * 32 + lane];
            mean[lane] = sum * inv_ne;
        }
    }
    __syncthreads();
    const double xb = mean[lane];
    const int ldt = ldx + 8;
    if (X64) {
        if (ok)
            for (int i = wp; i < ne; i += 8) X64[(size_t)i * nx + p] = ((double)m[(size_t)i * nx + p] - xb) * isq;
        return;
    }
    // BF16 path (FP32 states): FP32 centring on the exact differences,
    // ((x_i - x_ref) - dm) / sqrt(Ne - 1), then BF16 rounding (2^-9 of the
    // anomaly, far above the FP32 errors of the centring)
    const float isqf = (float)isq, xr = rfm[lane], dm = rfm[32 + lane];
    for (int i = wp; i < ldx; i += 8)
        tile[lane * ldt + i] = __float2bfloat16(
            (ok && i < ne) ? __fmul_rn(__fsub_rn(__fsub_rn((float)m[(size_t)i * nx + p], xr), dm), isqf) : 0.f);
    __syncthreads();
    // store: row r of the tile (point p0 + r) is ldx bf16 = ldx/8 16-byte chunks
    const int chunks = ldx / 8;
    for (int e = threadIdx.x; e < 32 * chunks; e += blockDim.x) {
        const int r = e / chunks, cidx = e % chunks;
        if (p0 + r < nx)
            reinterpret_cast<uint4 *>(X16 + (p0 + r) * ldx)[cidx] =
                reinterpret_cast<const uint4 *>(tile + r * ldt)[cidx];
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_ens_anom(const T *__restrict__ m, size_t nx, int ne, double inv_ne,
                                                  double isq, double *__restrict__ X64,
                                                  __nv_bfloat16 *__restrict__ X16, int ldx, const int *status) {
    launch_wait();
    ens_anom_body<T>(m, nx, ne, inv_ne, isq, X64, X16, ldx, status, blockIdx.x);
}

// dynamic shared memory of the anomaly kernel for BF16 rows of ldx values
static size_t ens_anom_smem(int ldx) {
    return sizeof(double) * 9 * 32 + sizeof(__nv_bfloat16) * 32 * (size_t)(ldx + 8);
}

template <typename T>
void launch_ens_anom(const T *members, size_t nx, int ne, double *X64, __nv_bfloat16 *X16,
                     const int *status, cudaStream_t s) {
    count_launches(1);
    const int ldx = (ne + 15) / 16 * 16;
    const size_t smem = ens_anom_smem(ldx);
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_ens_anom<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int ctas = ceil_div(nx, 32);
    // chained while a CTA is short (2 to 38 CTAs: 2 to 4 us gained up to 192 members, 30 to
    // 39 us lost at 400)
    launch_kernel(k_ens_anom<T>, ctas, 256, smem, s, LaunchHow{1, 1, 1, ctas <= kNumSMs / 4 && ne <= 192}, members, nx, ne,
                  1.0 / ne, 1.0 / std::sqrt((double)(ne - 1)), X64, X16, ldx, status);
}

// ---------------------------------------------------------------------------
// FP64 GEMMs of the gain (Algorithm 3 step 8)
// ---------------------------------------------------------------------------
// [out1 | out2^T] = A [B1; B2]^T / divisor (+ diag on out1's diagonal), FP64.
// One 8 x 16 output tile per CTA of 128 threads (a warp on each scheduler), one
// output per thread, k in chunks of 32 staged in shared memory; the next
// chunk's loads are issued before the current chunk's FMAs, so they are in
// flight while GB300's slow FP64 pipe works.  When B1 is A and n1 = m, out1 = A
// A^T / divisor + diag I is symmetric: 16 x 16 tiles strictly below its diagonal
// are not computed (a quarter of the FMAs of S = I + Y^T R^-1 Y [Y | D | d*]),
// their values are the mirror of the tiles above (the same products, so the
// same bits).  The K splits of a tile are a cluster: the partial sums stay in
// shared memory and are added, in the order of the splits, by the CTA that
// writes the output.  Bound by the FP64 pipes of the SM with the most CTAs:
// half the tile of before (16 x 16, two warps per scheduler) evens them out.
// S and T of 128 members, 512 observations: 36 us and 5 us for a reduction
// launch, 38 us so; 100 members, 80 observations: 12 and 9.5 us.
constexpr int kGemmThreads = 128, kGemmRows = 8;
constexpr int kGemmMaxPer = 4;  // splits per CTA of a cluster of 8
__device__ __forceinline__ double gemm_nt_tile(const double *__restrict__ A, int m, const double *__restrict__ B1,
                                               int n1, const double *__restrict__ B2, int n2, int K, int kb,
                                               int ke, int a0, int c0) {
    __shared__ double As[kGemmRows][33], Bs[16][33];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int kq = threadIdx.x & 31, rr = threadIdx.x >> 5;  // staging: column, and rows rr, rr + 4, ...
    const double *arow[2], *brow[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int a = a0 + rr + 4 * q, c = c0 + rr + 4 * q;
        if (q < 2) arow[q] = a < m ? A + (size_t)a * K : nullptr;
        brow[q] = c < n1 ? B1 + (size_t)c * K : (c < n1 + n2 ? B2 + (size_t)(c - n1) * K : nullptr);
    }
    double va[2], vb[4];
    auto fetch = [&](int k0) {
        const int k = k0 + kq;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (q < 2) va[q] = (arow[q] && k < ke) ? arow[q][k] : 0.0;
            vb[q] = (brow[q] && k < ke) ? brow[q][k] : 0.0;
        }
    };
    fetch(kb);
    double acc = 0.0;
    for (int k0 = kb; k0 < ke; k0 += 32) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (q < 2) As[rr + 4 * q][kq] = va[q];
            Bs[rr + 4 * q][kq] = vb[q];
        }
        __syncthreads();
        if (k0 + 32 < ke) fetch(k0 + 32);
        for (int k8 = 0; k8 < min(32, ke - k0); k8 += 8)  // zeros past ke
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) acc = fma(As[ty][k8 + kk], Bs[tx][k8 + kk], acc);
        __syncthreads();
    }
    return acc;
}

// output (a, c) of [out1 | out2^T] from its sum; mirror: also out1's (c, a)
__device__ __forceinline__ void gemm_put(double acc, int a, int c, int m, int n1, int n2, bool mirror, double divisor,
                                         double diag, double *__restrict__ out1, double *__restrict__ out2) {
    if (a >= m) return;
    if (c < n1) {
        out1[(size_t)a * n1 + c] = (a == c ? diag : 0.0) + acc / divisor;
        if (mirror) out1[(size_t)c * n1 + a] = acc / divisor;
    } else if (c < n1 + n2) {
        out2[(size_t)(c - n1) * m + a] = acc / divisor;
    }
}

// The sums of a tile of E outputs over the splits of its cluster (gridDim.z
// CTAs, `per` splits each): part[l][e] holds this CTA's; put(e, sum) is called
// for the outputs of this CTA, E / gridDim.z of them.
template <int E, class Put>
__device__ __forceinline__ void gemm_cluster_sum(double (*part)[E], int per, Put put) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int ctas = gridDim.z, rank = blockIdx.z;
    cl.sync();
    const int share = E / ctas, e = rank * share + threadIdx.x;
    if ((int)threadIdx.x < share) {
        double acc = 0.0;
#pragma unroll 4
        for (int z = 0; z < ctas * per; ++z) acc += cl.map_shared_rank(&part[0][0], z / per)[(z % per) * E + e];
        put(e, acc);
    }
    cl.sync();  // no CTA leaves while another may still read its partial sums
}

// tile (blockIdx.x, blockIdx.y), splits of kchunk, `per` of them in each CTA of
// the cluster along z
__global__ void __launch_bounds__(kGemmThreads)
    k_gemm_nt(const double *__restrict__ A, int m, const double *__restrict__ B1, int n1,
              const double *__restrict__ B2, int n2, int K, int per, int kchunk, double divisor, double diag,
              double *__restrict__ out1, double *__restrict__ out2, const int *status) {
    launch_wait();
    if (status && *status) return;
    __shared__ double part[kGemmMaxPer][kGemmThreads];
    const bool sym = B1 == A && n1 == m;
    const int a0 = blockIdx.y * kGemmRows, c0 = blockIdx.x * 16;
    if (sym && c0 < (a0 & ~15)) return;  // mirrored from the tile above the diagonal
    const bool mirror = sym && c0 > (a0 & ~15);
    auto put = [&](int e, double acc) {
        gemm_put(acc, a0 + (e >> 4), c0 + (e & 15), m, n1, n2, mirror, divisor, diag, out1, out2);
    };
    double acc = 0.0;
    for (int l = 0; l < per; ++l) {
        const int kb = (blockIdx.z * per + l) * kchunk;
        acc = gemm_nt_tile(A, m, B1, n1, B2, n2, K, kb, min(K, kb + kchunk), a0, c0);
        part[l][threadIdx.x] = acc;
    }
    if (gridDim.z == 1)
        put(threadIdx.x, acc);
    else
        gemm_cluster_sum(part, per, put);
}

// Partial sums over K chunks in memory, for more splits than a cluster takes.
__global__ void __launch_bounds__(kGemmThreads)
    k_gemm_nt_split(const double *__restrict__ A, int m, const double *__restrict__ B1, int n1,
                    const double *__restrict__ B2, int n2, int K, int kchunk, double *__restrict__ part,
                    const int *status) {
    launch_wait();
    if (status && *status) return;
    const int a0 = blockIdx.y * kGemmRows, c0 = blockIdx.x * 16;
    if (B1 == A && n1 == m && c0 < (a0 & ~15)) return;
    const int kb = blockIdx.z * kchunk;
    const double acc = gemm_nt_tile(A, m, B1, n1, B2, n2, K, kb, min(K, kb + kchunk), a0, c0);
    const int a = a0 + (threadIdx.x >> 4), c = c0 + (threadIdx.x & 15);
    if (a < m && c < n1 + n2) part[((size_t)blockIdx.z * m + a) * (n1 + n2) + c] = acc;
}

__device__ __forceinline__ void gemm_nt_reduce_body(const double *__restrict__ part, int nsplit, int m, int n1,
                                                    int n2, bool sym, double divisor, double diag,
                                                    double *__restrict__ out1, double *__restrict__ out2, int blk,
                                                    int nblk) {
    const int ncol = n1 + n2;
    for (int e = blk * blockDim.x + threadIdx.x; e < m * ncol; e += nblk * blockDim.x) {
        const int a = e / ncol, c = e % ncol;
        // below the diagonal tiles of a symmetric out1: the mirrored element
        const bool mirror = sym && c < n1 && (c >> 4) < (a >> 4);
        const int ra = mirror ? c : a, rc = mirror ? a : c;
        double acc = 0.0;
        for (int z = 0; z < nsplit; ++z) acc += part[((size_t)z * m + ra) * ncol + rc];
        if (c < n1)
            out1[(size_t)a * n1 + c] = (a == c ? diag : 0.0) + acc / divisor;
        else
            out2[(size_t)(c - n1) * m + a] = acc / divisor;
    }
}

__global__ void k_gemm_nt_reduce(const double *__restrict__ part, int nsplit, int m, int n1, int n2, bool sym,
                                 double divisor, double diag, double *__restrict__ out1,
                                 double *__restrict__ out2, const int *status) {
    launch_wait();
    if (status && *status) return;
    gemm_nt_reduce_body(part, nsplit, m, n1, n2, sym, divisor, diag, out1, out2, blockIdx.x, gridDim.x);
}

int gemm_nt_splits(int m, int n1, int n2, int K) {
    const int tiles = ceil_div(n1 + n2, 16) * ceil_div(m, 16);
    int splits = 1;
    while (tiles * splits * 2 <= 2 * kNumSMs && K / (splits * 2) >= 128) splits *= 2;
    return splits;
}

// ---------------------------------------------------------------------------
// The gain products of the mixed path in double-FP32 arithmetic on the FP32
// pipes (GB300 runs FP32 FMAs about 64 times faster than FP64 ones): each FP64
// operand is a pair hi + lo of FP32 values (split_df); a b = ah bh + ah bl +
// al bh (+ al bl, below 2^-48 |a b|, dropped), ah bh exactly as p + e with
// e = fma(ah, bh, -p); the products are summed into a running FP32 sum s and
// the FP32 sum c of its rounding errors (error-free two-sum) and of the small
// terms.  The result s + c carries a relative error of order 2^-44 of the sum
// of |a b|, far below the BF16 rounding of T that follows.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void df_mac(float ah, float al, float bh, float bl, float &s, float &c) {
    const float p = __fmul_rn(ah, bh);
    const float e = __fmaf_rn(ah, bh, -p);
    const float x = __fmaf_rn(ah, bl, __fmaf_rn(al, bh, e));
    const float t = __fadd_rn(s, p), bv = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, bv)), __fsub_rn(p, bv)), x));
    s = t;
}

constexpr int kDfThreads = 256;  // a 16 x 16 output tile: four groups of 64 threads, 2 x 2 outputs per thread
constexpr int kDfK = 32;         // K chunk staged in shared memory

// One output, (a0 + t / 16, c0 + t % 16) for thread t, of [Y^T R^-1 Y | Y^T R^-1
// [D | d*]] over k in [kb, ke), from the double-FP32 operands.  Each group takes
// a quarter of every K chunk, so that eight warps and not two hide the latency
// of the error-free sums (64 members, 2048 observations: 24 us and a reduction
// of 8, 17 us with the cluster's sums); the groups' sums are added in FP64.
__device__ __forceinline__ double gemm_df_tile(const DfOperands &df, int ne, int K, int kb, int ke, int a0, int c0) {
    __shared__ float sAh[16][kDfK + 1], sAl[16][kDfK + 1], sBh[16][kDfK + 1], sBl[16][kDfK + 1];
    __shared__ double red[4][256];
    const int m = ne, n1 = ne, n2 = ne + 1;
    const int tid = threadIdx.x, grp = tid >> 6, tx = tid & 7, ty = (tid >> 3) & 7;
    // staging: row tid / 16 of the A and B tiles, k = (tid mod 16) * 2 and the next of the chunk
    const int sr = tid >> 4, sk = (tid & 15) * 2;
    const int ar = a0 + sr, cr = c0 + sr;
    const float *ah = ar < m ? df.Yh + (size_t)ar * K : nullptr, *al = ar < m ? df.Yl + (size_t)ar * K : nullptr;
    const float *bh = cr < n1 ? df.Yh + (size_t)cr * K : (cr < n1 + n2 ? df.Zh + (size_t)(cr - n1) * K : nullptr);
    const float *bl = cr < n1 ? df.Yl + (size_t)cr * K : (cr < n1 + n2 ? df.Zl + (size_t)(cr - n1) * K : nullptr);
    float va[2][2], vb[2][2];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int k = k0 + sk + j;
            const bool ok = k < ke;
            va[0][j] = (ah && ok) ? ah[k] : 0.f;
            va[1][j] = (al && ok) ? al[k] : 0.f;
            vb[0][j] = (bh && ok) ? bh[k] : 0.f;
            vb[1][j] = (bl && ok) ? bl[k] : 0.f;
        }
    };
    float s[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, c[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
    fetch(kb);
    for (int k0 = kb; k0 < ke; k0 += kDfK) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            sAh[sr][sk + j] = va[0][j];
            sAl[sr][sk + j] = va[1][j];
            sBh[sr][sk + j] = vb[0][j];
            sBl[sr][sk + j] = vb[1][j];
        }
        __syncthreads();
        if (k0 + kDfK < ke) fetch(k0 + kDfK);  // in flight during the chunk's products
#pragma unroll 4
        for (int kk = grp * (kDfK / 4); kk < (grp + 1) * (kDfK / 4); ++kk) {
            float xh[2], xl[2], yh[2], yl[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                xh[i] = sAh[2 * ty + i][kk];
                xl[i] = sAl[2 * ty + i][kk];
                yh[i] = sBh[2 * tx + i][kk];
                yl[i] = sBl[2 * tx + i][kk];
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) df_mac(xh[i], xl[i], yh[j], yl[j], s[i][j], c[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
            red[grp][(2 * ty + i) * 16 + 2 * tx + j] = (double)s[i][j] + (double)c[i][j];
    __syncthreads();
    const double acc = ((red[0][tid] + red[1][tid]) + red[2][tid]) + red[3][tid];
    __syncthreads();  // red may be written again
    return acc;
}

__global__ void __launch_bounds__(kDfThreads) k_gemm_df(DfOperands df, int ne, int K, int per, int kchunk,
                                                        double divisor, double diag, double *__restrict__ out1,
                                                        double *__restrict__ out2, double *__restrict__ parts,
                                                        const int *status) {
    launch_wait();
    if (*status) return;
    __shared__ double part[kGemmMaxPer][kDfThreads];
    const int a0 = blockIdx.y * 16, c0 = blockIdx.x * 16, m = ne, n1 = ne, n2 = ne + 1;
    if (c0 < a0) return;  // mirrored from the tile above the diagonal
    auto put = [&](int e, double acc) {
        gemm_put(acc, a0 + (e >> 4), c0 + (e & 15), m, n1, n2, c0 > a0, divisor, diag, out1, out2);
    };
    double acc = 0.0;
    for (int l = 0; l < per; ++l) {
        const int kb = (blockIdx.z * per + l) * kchunk;
        acc = gemm_df_tile(df, ne, K, kb, min(K, kb + kchunk), a0, c0);
        part[l][threadIdx.x] = acc;
    }
    if (parts) {  // more splits than a cluster takes: partial sums in memory
        const int a = a0 + (threadIdx.x >> 4), c = c0 + (threadIdx.x & 15);
        if (a < m && c < n1 + n2) parts[((size_t)blockIdx.z * m + a) * (n1 + n2) + c] = acc;
    } else if (gridDim.z == 1) {
        put(threadIdx.x, acc);
    } else {
        gemm_cluster_sum(part, per, put);
    }
}

// cluster of the K splits (a power of two): CTAs and splits per CTA, or 0 CTAs
// if there are more than a portable cluster takes
struct GemmCluster {
    int ctas, per;
};
static GemmCluster gemm_cluster(int splits) {
    const int ctas = std::min(splits, 8), per = splits / ctas;
    return per <= kGemmMaxPer ? GemmCluster{ctas, per} : GemmCluster{0, 1};
}
void launch_gemm_df(const DfOperands &df, int ne, int ny, double s2, double *S, double *Bt, const int *status,
                    cudaStream_t s, double *part) {
    const int splits = part ? gemm_nt_splits(ne, ne, ne + 1, ny) : 1;
    const int kchunk = ceil_div(ceil_div(ny, splits), 32) * 32;
    const GemmCluster g = gemm_cluster(splits);
    const dim3 grid(ceil_div(2 * ne + 1, 16), ceil_div(ne, 16), g.ctas ? g.ctas : splits);
    count_launches(g.ctas ? 1 : 2);
    // chained unless its CTAs are long and about as many as the SMs (gained or lost:
    // up to 80 CTAs 2 us gained, 144 of 128 products of K 1 gained, 168 to 288 of 128
    // 3 lost, 220 of 512 17 lost, 210 of 2048 76 lost, 528 CTAs of any length 1 to 3
    // gained; NS analysis of 64 members and 2048 observations 178 us chained, 172)
    const unsigned ctas = grid.x * grid.y * grid.z, length = g.per * kchunk;
    const bool chained = ctas <= kNumSMs / 2 || ctas > 2u * kNumSMs || length <= (ctas <= kNumSMs ? 128u : 64u);
    launch_kernel(k_gemm_df, grid, kDfThreads, 0, s, LaunchHow{1, 1, (unsigned)std::max(g.ctas, 1), chained}, df, ne, ny,
                  g.per, kchunk, s2, 1.0, S, Bt, g.ctas ? (double *)nullptr : part, status);
    if (!g.ctas)
        launch_kernel(k_gemm_nt_reduce, grid_for((size_t)ne * (2 * ne + 1), 256), 256, 0, s, LaunchHow{}, part,
                      splits, ne, ne, ne + 1, true, s2, 1.0, S, Bt, status);
}

void launch_gemm_nt_f64(const double *A, int m, const double *B1, int n1, const double *B2, int n2,
                        int K, double scale_div, double diag, double *out1, double *out2,
                        const int *status, cudaStream_t s, double *part) {
    const int splits = part ? gemm_nt_splits(m, n1, n2, K) : 1;
    const int kchunk = ceil_div(ceil_div(K, splits), 32) * 32;
    const GemmCluster g = gemm_cluster(splits);
    const dim3 grid(ceil_div(n1 + n2, 16), ceil_div(m, kGemmRows), g.ctas ? g.ctas : splits);
    count_launches(g.ctas ? 1 : 2);
    if (g.ctas) {
        // S and T follow short kernels (up to 288 CTAs 2 to 3 us gained); the direct form's
        // T (n1 = 0) follows the solves, which hold most SMs while its CTAs are placed on
        // the others (60 CTAs 2 to 4 us gained, 144 of 60 to 250 products 10 to 43 lost)
        const bool chained = grid.x * grid.y * grid.z <= (n1 == 0 ? 64u : 2u * kNumSMs);
        launch_kernel(k_gemm_nt, grid, kGemmThreads, 0, s, LaunchHow{1, 1, (unsigned)g.ctas, chained}, A, m, B1, n1,
                      B2, n2, K, g.per, kchunk, scale_div, diag, out1, out2, status);
        return;
    }
    launch_kernel(k_gemm_nt_split, grid, kGemmThreads, 0, s, LaunchHow{}, A, m, B1, n1, B2, n2, K, kchunk, part,
                  status);
    launch_kernel(k_gemm_nt_reduce, grid_for((size_t)m * (n1 + n2), 256), 256, 0, s, LaunchHow{}, part, splits, m, n1,
                  n2, B1 == A && n1 == m, scale_div, diag, out1, out2, status);
}

__global__ void k_gemm_tn(const double *__restrict__ Y, int ne, int ny, double diag,
                          double *__restrict__ C, const int *status) {
    launch_wait();
    if (*status) return;
    __shared__ double As[32][17];
    __shared__ double Bs[32][17];
    const int j0 = blockIdx.y * 16, l0 = blockIdx.x * 16;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double acc = 0.0;
    for (int k0 = 0; k0 < ne; k0 += 32) {
        for (int e = threadIdx.x; e < 32 * 16; e += 256) {
            const int kk = e >> 4, r = e & 15, k = k0 + kk;
            As[kk][r] = (k < ne && j0 + r < ny) ? Y[(size_t)k * ny + j0 + r] : 0.0;
            Bs[kk][r] = (k < ne && l0 + r < ny) ? Y[(size_t)k * ny + l0 + r] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 32; ++kk) acc = fma(As[kk][ty], Bs[kk][tx], acc);
        __syncthreads();
    }
    const int j = j0 + ty, l = l0 + tx;
    if (j < ny && l < ny) C[(size_t)j * ny + l] = acc + (j == l ? diag : 0.0);
}

void launch_gemm_tn_f64(const double *Y, int ne, int ny, double diag, double *C, const int *status,
                        cudaStream_t s) {
    count_launches(1);
    dim3 grid(ceil_div(ny, 16), ceil_div(ny, 16));
    launch_kernel(k_gemm_tn, grid, 256, 0, s, LaunchHow{}, Y, ne, ny, diag, C, status);
}

// ---------------------------------------------------------------------------
// SPD solves: up to order 256 spd_solve.cuh, above (direct form) a Cholesky
// factorisation in global memory by one CTA and a substitution per column
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_cholesky(double *M, double *Lt, int n, int *status) {
    // Right-looking Cholesky by one CTA.  Column k: pivot l = sqrt(M_kk) and its
    // reciprocal (one division per column), scale the column below it, then the
    // rank-1 update of the trailing lower triangle.
    __shared__ double s_inv;
    if (*status) return;
    const int tid = threadIdx.x, nth = blockDim.x;
    const int tx = tid & 31, ty = tid >> 5, nty = nth >> 5;
    for (int k = 0; k < n; ++k) {
        const double d = M[(size_t)k * n + k];
        if (!(d > 0.0) || !isfinite(d)) {  // uniform: every thread read the same pivot
            if (tid == 0) atomicCAS(status, 0, kStNotSpd);
            return;
        }
        __syncthreads();  // every thread has read the pivot before it is overwritten
        if (tid == 0) {
            const double l = sqrt(d);
            M[(size_t)k * n + k] = l;
            s_inv = 1.0 / l;
        }
        __syncthreads();
        const double inv = s_inv;
        for (int i = k + 1 + tid; i < n; i += nth) M[(size_t)i * n + k] *= inv;
        __syncthreads();
        for (int i = k + 1 + ty; i < n; i += nty) {
            const double lik = M[(size_t)i * n + k];
            for (int j = k + 1 + tx; j <= i; j += 32)
                M[(size_t)i * n + j] = fma(-lik, M[(size_t)j * n + k], M[(size_t)i * n + j]);
        }
        __syncthreads();
    }
    for (int e = tid; e < n * n; e += nth) {
        const int i = e / n, j = e % n;
        const double val = j <= i ? M[(size_t)i * n + j] : 0.0;
        M[e] = val;
        Lt[(size_t)j * n + i] = val;
    }
}

template <int C>
__global__ void __launch_bounds__(kSpdThreads) k_spd_factor(double *A, double *At, int n, int *status) {
    launch_wait();
    spd_factor_body<C>(A, At, n, status);
}

template <int C>
static void spd_factor_launch(double *A, double *At, int n, int *status, cudaStream_t s) {
    static OncePerDevice attr;
    attr.run([](int) {
        cudaError_t e = cudaFuncSetAttribute(k_spd_factor<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)spd_factor_smem(kSpdMax, C));
        if (e == cudaSuccess && C > 8)
            e = cudaFuncSetAttribute(k_spd_factor<C>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        return e;
    });
    launch_kernel(k_spd_factor<C>, C, kSpdThreads, spd_factor_smem(n, C), s, LaunchHow{C}, A, At, n, status);
}

// NT: 256, or 384 for orders above 224, where the registers are limited so that
// two CTAs share an SM (there are more columns than SMs; n = 256: 86 us with one, 59)
template <int NT>
__global__ void __launch_bounds__(NT, NT > 256 ? 2 : 1)
    k_spd_apply(const double *__restrict__ A, const double *__restrict__ At, int n, const double *rhs, double *out,
                __nv_bfloat16 *out16, int ld16, const int *status) {
    launch_wait();
    const size_t c = blockIdx.x;
    spd_apply_body(A, At, n, rhs + c * n, out + c * n, out16 ? out16 + c * ld16 : nullptr, status);
}

void launch_spd_factor(double *A, double *At, int n, int *status, cudaStream_t s) {
    count_launches(1);
    if (n <= kSpdMax) {
        if (spd_cluster(n) == 16)
            spd_factor_launch<16>(A, At, n, status, s);
        else
            spd_factor_launch<8>(A, At, n, status, s);
    } else {
        k_cholesky<<<1, 256, 0, s>>>(A, At, n, status);
    }
}

template <int MAXR>
__global__ void __launch_bounds__(32) k_chol_solve(const double *__restrict__ L,
                                                   const double *__restrict__ Lt, int n,
                                                   const double *rhs, double *out, int ncol,
                                                   __nv_bfloat16 *out16, int ld16,
                                                   const int *status) {
    if (*status) return;
    const int c = blockIdx.x;
    const int lane = threadIdx.x;
    if (c >= ncol) return;
    double b[MAXR];
#pragma unroll
    for (int m = 0; m < MAXR; ++m) {
        const int i = lane + 32 * m;
        b[m] = i < n ? rhs[(size_t)c * n + i] : 0.0;
    }
    // forward substitution L z = b (column-oriented: after z_j, b_i -= L_ij z_j)
#pragma unroll
    for (int s = 0; s < MAXR; ++s) {
        if (s * 32 >= n) break;
        for (int l = 0; l < 32; ++l) {
            const int j = s * 32 + l;
            if (j >= n) break;
            if (lane == l) b[s] = b[s] / L[(size_t)j * n + j];
            const double zj = __shfl_sync(0xffffffffu, b[s], l);
#pragma unroll
            for (int m = s; m < MAXR; ++m) {
                const int i = lane + 32 * m;
                if (i > j && i < n) b[m] = fma(-Lt[(size_t)j * n + i], zj, b[m]);
            }
        }
    }
    // back substitution L^T x = z (after x_j, z_i -= L_ji x_j for i < j)
#pragma unroll
    for (int s = MAXR - 1; s >= 0; --s) {
        if (s * 32 >= n) continue;
        for (int l = 31; l >= 0; --l) {
            const int j = s * 32 + l;
            if (j >= n) continue;
            if (lane == l) b[s] = b[s] / L[(size_t)j * n + j];
            const double xj = __shfl_sync(0xffffffffu, b[s], l);
#pragma unroll
            for (int m = 0; m <= s; ++m) {
                const int i = lane + 32 * m;
                if (i < j) b[m] = fma(-L[(size_t)j * n + i], xj, b[m]);
            }
        }
    }
#pragma unroll
    for (int m = 0; m < MAXR; ++m) {
        const int i = lane + 32 * m;
        if (i < n) {
            out[(size_t)c * n + i] = b[m];
            if (out16) out16[(size_t)c * ld16 + i] = __double2bfloat16(b[m]);
        }
    }
}

void launch_spd_solve(const double *A, const double *At, int n, const double *rhs, double *out, int ncol,
                      __nv_bfloat16 *out16, int ld16, const int *status, cudaStream_t s) {
    count_launches(1);
    if (n <= kSpdMax)
        launch_kernel(spd_apply_threads(n) > 256 ? k_spd_apply<384> : k_spd_apply<256>, ncol, spd_apply_threads(n), 0,
                      s, LaunchHow{}, A, At, n, rhs, out, out16, ld16, status);
    else if (n <= 512)
        k_chol_solve<16><<<ncol, 32, 0, s>>>(A, At, n, rhs, out, ncol, out16, ld16, status);
    else
        k_chol_solve<64><<<ncol, 32, 0, s>>>(A, At, n, rhs, out, ncol, out16, ld16, status);
}

// ---------------------------------------------------------------------------
// member update x^a,(i) = x^f,(i) + X T_i and coarse correction dC = X T_ne
// (Eq. ensemble_update with K = X T; Algorithm 4 step 5)
// ---------------------------------------------------------------------------
// A warp takes 32 points and Q columns (the columns of T in shared memory, read
// by broadcast; X eight members ahead in registers), a CTA one warp per
// scheduler.  Bound by the FP64 pipes, 64 cycles of a scheduler per warp
// instruction whatever its lanes hold, so Q is the number of columns whose CTAs
// fill the SMs most evenly (update_cols): a fixed 8 columns in CTAs of 8 warps
// left half the SMs idle in the last round and multiplied 31 columns of padding
// at ne + 1 = 129.  4096 points x 128 members: 199 -> 122 us (Q = 7); 200 x 100:
// 68 -> 16 us; 64 x 32: 27 -> 6.5 us (Q = 1).
constexpr int kUpdateWarps = 4, kUpdateMaxCols = 8;
template <typename T, int Q>
__global__ void __launch_bounds__(32 * kUpdateWarps) k_update_f64(T *__restrict__ members, T *__restrict__ dC,
                                                                  const double *__restrict__ X,
                                                                  const double *__restrict__ Tm, size_t nx, int ne,
                                                                  const int *status) {
    launch_wait();
    extern __shared__ double2 Ts2[];  // [Q columns][ne rounded up to 8]
    if (*status) return;
    double *Ts = reinterpret_cast<double *>(Ts2);
    const int c0 = blockIdx.y * Q, pitch = (ne + 7) & ~7;
#pragma unroll
    for (int q = 0; q < Q; ++q)
        for (int a = threadIdx.x; a < pitch; a += blockDim.x)
            Ts[q * pitch + a] = a < ne && c0 + q <= ne ? Tm[(size_t)(c0 + q) * ne + a] : 0.0;
    const size_t p = blockIdx.x * (size_t)(32 * kUpdateWarps) + threadIdx.x;
    const bool in = p < nx;
    double x[8], acc[Q];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = in && i < ne ? X[(size_t)i * nx + p] : 0.0;
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[q] = 0.0;
    __syncthreads();
    if (blockIdx.x * (size_t)(32 * kUpdateWarps) + (threadIdx.x & ~31) >= nx) return;  // no point of this warp
    for (int a = 0; a < pitch; a += 8) {
        double xn[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) xn[i] = in && a + 8 + i < ne ? X[(size_t)(a + 8 + i) * nx + p] : 0.0;
#pragma unroll
        for (int i = 0; i < 8; i += 2)
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const double2 t = Ts2[(q * pitch + a + i) >> 1];
                acc[q] = fma(x[i], t.x, acc[q]);
                acc[q] = fma(x[i + 1], t.y, acc[q]);
            }
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = xn[i];
    }
    if (!in) return;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int c = c0 + q;
        if (c < ne)
            members[(size_t)c * nx + p] = (T)((double)members[(size_t)c * nx + p] + acc[q]);
        else if (c == ne)
            dC[p] = (T)acc[q];
    }
}

// columns per warp: the fewest rounds of CTAs times the work of one (its
// columns, and about 16 instructions to start and end); of equal ones the most
static int update_cols(size_t nx, int ne) {
    const long long pb = (long long)((nx + 32 * kUpdateWarps - 1) / (32 * kUpdateWarps));
    int best = 1;
    long long cost = 0;
    for (int q = 1; q <= kUpdateMaxCols; ++q) {
        const long long ctas = pb * ceil_div(ne + 1, q);
        const long long c = (ctas + kNumSMs - 1) / kNumSMs * ((long long)q * ne + 16);
        if (q == 1 || c <= cost) {
            cost = c;
            best = q;
        }
    }
    return best;
}

template <typename T, int Q>
static void update_launch(int cols, T *members, T *dC, const double *X, const double *Tm, size_t nx, int ne,
                          const int *status, cudaStream_t s) {
    if constexpr (Q > 1)
        if (cols < Q) return update_launch<T, Q - 1>(cols, members, dC, X, Tm, nx, ne, status, s);
    const dim3 grid(ceil_div(nx, 32 * kUpdateWarps), ceil_div(ne + 1, Q));
    const size_t smem = sizeof(double) * Q * (size_t)((ne + 7) & ~7);  // <= 32 KB for ne <= 512
    // chained while a thread has few FMAs, ne of each column: it follows the solves, which
    // hold most SMs while its CTAs are placed on the others (66 to 144 CTAs of up to
    // 104 FMAs: 2 to 4 us gained; 152 of 896: 157 lost, 126 of 512: 117 lost)
    const bool chained = grid.x * grid.y <= 2u * kNumSMs && Q * ((ne + 7) & ~7) <= 112;
    launch_kernel(k_update_f64<T, Q>, grid, 32 * kUpdateWarps, smem, s, LaunchHow{1, 1, 1, chained}, members, dC, X,
                  Tm, nx, ne, status);
}

template <typename T>
void launch_update_f64(T *members, T *dC, const double *X, const double *Tm, size_t nx, int ne,
                       const int *status, cudaStream_t s) {
    count_launches(1);
    update_launch<T, kUpdateMaxCols>(update_cols(nx, ne), members, dC, X, Tm, nx, ne, status, s);
}

// BF16 anomaly product with FP32 accumulation (CUDA-core version): X^T tile of
// 64 points and T tile of 32 columns staged in shared memory.
__global__ void __launch_bounds__(256) k_update_bf16(float *__restrict__ members,
                                                     float *__restrict__ dC,
                                                     const __nv_bfloat16 *__restrict__ Xt,
                                                     const __nv_bfloat16 *__restrict__ Tt, int ldx,
                                                     size_t nx, int ne, const int *status) {
    extern __shared__ __nv_bfloat16 sm16[];
    if (*status) return;
    const int lds = ldx + 2;
    __nv_bfloat16 *Xs = sm16;             // [64][lds]
    __nv_bfloat16 *Tsm = sm16 + 64 * lds; // [32][lds]
    const size_t p0 = blockIdx.x * (size_t)64;
    const int c0 = blockIdx.y * 32;
    for (int e = threadIdx.x; e < 64 * ldx; e += blockDim.x) {
        const int r = e / ldx, a = e % ldx;
        Xs[r * lds + a] = p0 + r < nx ? Xt[(p0 + r) * ldx + a] : __float2bfloat16(0.f);
    }
    for (int e = threadIdx.x; e < 32 * ldx; e += blockDim.x) {
        const int r = e / ldx, a = e % ldx;
        Tsm[r * lds + a] = c0 + r <= ne ? Tt[(size_t)(c0 + r) * ldx + a] : __float2bfloat16(0.f);
    }
    __syncthreads();
    const int pl = threadIdx.x & 63, cg = threadIdx.x >> 6;
    const size_t p = p0 + pl;
    if (p >= nx) return;
    float acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = 0.f;
    for (int a = 0; a < ne; ++a) {
        const float x = __bfloat162float(Xs[pl * lds + a]);
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] = fmaf(x, __bfloat162float(Tsm[(cg * 8 + q) * lds + a]), acc[q]);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int c = c0 + cg * 8 + q;
        if (c < ne)
            members[(size_t)c * nx + p] += acc[q];
        else if (c == ne)
            dC[p] = acc[q];
    }
}

void launch_update_bf16(float *members, float *dC, const __nv_bfloat16 *Xt, const __nv_bfloat16 *Tt,
                        int ldx, size_t nx, int ne, const int *status, cudaStream_t s) {
    count_launches(1);
    dim3 grid(ceil_div(nx, 64), ceil_div(ne + 1, 32));
    const size_t smem = sizeof(__nv_bfloat16) * (size_t)(64 + 32) * (ldx + 2);  // <= 99 KB
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_update_bf16, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_update_bf16<<<grid, 256, smem, s>>>(members, dC, Xt, Tt, ldx, nx, ne, status);
}

// ---------------------------------------------------------------------------
// prolongation of the coarse correction, Algorithm 4 step 5 second line
// ---------------------------------------------------------------------------
// a b + c rounded once, in the precision of T
template <typename T>
__device__ __forceinline__ T fma_t(T a, T b, T c) {
    if constexpr (std::is_same<T, float>::value)
        return fmaf(a, b, c);
    else
        return fma(a, b, c);
}

// periodic index of a 4-point stencil tap: c in [-1, nc + 2)
__device__ __forceinline__ int wrap_tap(int c, int nc) {
    if (c < 0) c += nc;
    while (c >= nc) c -= nc;
    return c;
}

// fine (+)= Pi_F(dC): the 4-point Lagrange interpolant at fine offset m of
// coarse interval J (nodes J - 1 .. J + 2).  2-D is the tensor product,
// evaluated separably: four 4-tap sums along x, then one 4-tap sum along y.
// 2-D launch: x over the points of a fine row, y over the rows of all
// variables, so the only divisions are by r and the periodic wraps are
// compares.
// 2-D: fine column fx of the r fine rows of coarse interval Jy of variable v
// (vj = v nc + Jy).  The four sums along x (coarse rows Jy - 1 .. Jy + 2) are
// the same for the r rows and are formed once; each row is then its 4-tap sum
// along y.  The fine values of up to 4 rows are loaded before any of them is written.
// wt: the weights converted to T ([m][t], in shared memory).
template <typename T>
__device__ __forceinline__ void prolong2d_interval(T *__restrict__ fine, const T *__restrict__ dC, int nc, int r,
                                                   const T (*wt)[4], int fx, int vj) {
    const int nf = nc * r;
    const int v = vj / nc, Jy = vj - v * nc;
    const int Jx = fx / r, mx = fx - Jx * r;
    int cx[4];
    T wx[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        cx[t] = wrap_tap(Jx - 1 + t, nc);
        wx[t] = wt[mx][t];
    }
    const T *d = dC + (size_t)v * nc * nc;
    T sx[4];
#pragma unroll
    for (int ty = 0; ty < 4; ++ty) {
        const T *dr = d + (size_t)wrap_tap(Jy - 1 + ty, nc) * nc;
        T a = T(0);
#pragma unroll
        for (int tx = 0; tx < 4; ++tx) a = fma_t(wx[tx], dr[cx[tx]], a);
        sx[ty] = a;
    }
    T *f = fine + (size_t)v * nf * nf + (size_t)Jy * r * nf + fx;
    for (int m0 = 0; m0 < r; m0 += 4) {
        T old[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (m0 + k < r) old[k] = f[(size_t)(m0 + k) * nf];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (m0 + k < r) {
                T acc = T(0);
#pragma unroll
                for (int ty = 0; ty < 4; ++ty) acc = fma_t(wt[m0 + k][ty], sx[ty], acc);
                f[(size_t)(m0 + k) * nf] = old[k] + acc;
            }
    }
}

// the Lagrange weights of offsets 0 .. r - 1 converted to T, into shared memory
template <typename T>
__device__ __forceinline__ void prolong_stage_weights(const ProlongWeights &w, int r, T (*wt)[4]) {
    for (int e = threadIdx.x; e < 4 * r; e += blockDim.x) wt[e >> 2][e & 3] = (T)w.w[e >> 2][e & 3];
    __syncthreads();
}

template <typename T>
__global__ void k_prolong_add(T *__restrict__ fine, const T *__restrict__ dC, int dim, int V, int nc,
                              int r, ProlongWeights w, const int *status) {
    launch_wait();
    if (*status) return;
    const int nf = nc * r;
    if (dim == 1) {
        const size_t total = (size_t)V * nf;
        for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
             idx += (size_t)gridDim.x * blockDim.x) {
            const int v = (int)(idx / nf), k = (int)(idx - (size_t)v * nf);
            const T *d = dC + (size_t)v * nc;
            const int J = k / r, m = k - J * r;
            T acc = T(0);
#pragma unroll
            for (int t = 0; t < 4; ++t) acc += (T)w.w[m][t] * d[wrap_tap(J - 1 + t, nc)];
            fine[idx] += acc;
        }
        return;
    }
    __shared__ T wt[kMaxRatio][4];
    prolong_stage_weights<T>(w, r, wt);
    const int fx = blockIdx.x * blockDim.x + threadIdx.x;
    if (fx >= nf) return;
    for (int vj = blockIdx.y; vj < V * nc; vj += gridDim.y) prolong2d_interval<T>(fine, dC, nc, r, wt, fx, vj);
}

template <typename T>
void launch_prolong_add(T *fine, const T *dC, int dim, int V, int nc, int r,
                        const ProlongWeights &w, const int *status, cudaStream_t s) {
    count_launches(1);
    const int nf = nc * r;
    if (dim == 1) {
        launch_kernel(k_prolong_add<T>, grid_for((size_t)V * nf, 256), 256, 0, s, LaunchHow{}, fine, dC, dim, V, nc,
                      r, w, status);
    } else {
        const dim3 grid(ceil_div(nf, 128), std::min(V * nc, 65535));
        launch_kernel(k_prolong_add<T>, grid, 128, 0, s, LaunchHow{}, fine, dC, dim, V, nc, r, w, status);
    }
}

// ---------------------------------------------------------------------------
// relative RMSE, Eq. L2norm_u (deterministic two-pass reduction)
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_rmse_partial(const T *__restrict__ x, const double *__restrict__ truth, int V,
                               size_t npts, double *__restrict__ partials) {
    __shared__ double red[2][32];
    for (int v = 0; v < V; ++v) {
        double num = 0.0, den = 0.0;
        for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < npts;
             k += (size_t)gridDim.x * blockDim.x) {
            const double t = truth[v * npts + k];
            const double d = (double)x[v * npts + k] - t;
            num = fma(d, d, num);
            den = fma(t, t, den);
        }
        for (int o = 16; o > 0; o >>= 1) {
            num += __shfl_down_sync(0xffffffffu, num, o);
            den += __shfl_down_sync(0xffffffffu, den, o);
        }
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (lane == 0) {
            red[0][w] = num;
            red[1][w] = den;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double a = 0.0, b = 0.0;
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q) {
                a += red[0][q];
                b += red[1][q];
            }
            partials[((size_t)blockIdx.x * V + v) * 2 + 0] = a;
            partials[((size_t)blockIdx.x * V + v) * 2 + 1] = b;
        }
        __syncthreads();
    }
}

__global__ void k_rmse_final(const double *__restrict__ partials, int nblocks, int V,
                             double *__restrict__ out) {
    const int v = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (v >= V) return;
    double a = 0.0, b = 0.0;
    for (int q = lane; q < nblocks; q += 32) {
        a += partials[((size_t)q * V + v) * 2 + 0];
        b += partials[((size_t)q * V + v) * 2 + 1];
    }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if (lane == 0) out[v] = sqrt(a / b);
}

template <typename T>
void launch_rmse(const T *x, const double *truth, int V, size_t npts, double *partials, int nblocks,
                 double *out, cudaStream_t s) {
    count_launches(2);
    k_rmse_partial<T><<<nblocks, 256, 0, s>>>(x, truth, V, npts, partials);
    k_rmse_final<<<1, 32 * V, 0, s>>>(partials, nblocks, V, out);
}

// ---------------------------------------------------------------------------
// conversions and normals
// ---------------------------------------------------------------------------
// FP64 <-> FP32 on the integer pipes: a conversion instruction takes the FP64 pipe
// (64 cycles of a scheduler per warp), which bound these kernels, not HBM: 64
// members of 128^2 x 4 values 12 us each way, 10 and 8.5 us so (50 MB).
// Numbers that stay normal, and zeros, are formed from their bits by the
// definition of the formats (to FP32: round to nearest, ties to even; the carry
// out of 2^128 is infinity); all others take the instruction.
__device__ __forceinline__ float convert_value(double x, float) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x), a = hi & 0x7fffffffu;
    if (a - 0x38100000u < 0x0fe00000u) {  // exponent field 1 .. 254 in FP32
        const uint32_t q = __funnelshift_l(lo, a - 0x38000000u, 3);
        const uint32_t r = q + (((lo & 0x1fffffffu) + 0x0fffffffu + (q & 1u)) >> 29);
        return __uint_as_float(r | (hi & 0x80000000u));
    }
    if ((a | lo) == 0) return __uint_as_float(hi);
    return (float)x;
}
__device__ __forceinline__ double convert_value(float x, double) {
    const uint32_t u = __float_as_uint(x), a = u & 0x7fffffffu;
    if (a - 0x00800000u < 0x7f000000u)  // normal
        return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(u << 29));
    if (a == 0) return __hiloint2double((int)u, 0);
    return (double)x;
}
__device__ __forceinline__ double convert_value(double x, double) { return x; }

// eight values in flight per thread
template <typename Tin, typename Tout>
__global__ void __launch_bounds__(256) k_convert(const Tin *__restrict__ in, Tout *__restrict__ out, size_t n) {
    launch_wait();
    constexpr int U = 8;
    const size_t nt = (size_t)gridDim.x * blockDim.x;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += U * nt) {
        Tin x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = i + u * nt < n ? in[i + u * nt] : Tin(0);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u * nt < n) out[i + u * nt] = convert_value(x[u], Tout());
    }
}

template <typename Tin, typename Tout>
void launch_convert(const Tin *in, Tout *out, size_t n, cudaStream_t s) {
    if (n == 0) return;
    count_launches(1);
    launch_kernel(k_convert<Tin, Tout>, grid_for(n, 256), 256, 0, s, LaunchHow{}, in, out, n);
}

// the analysis counter that keys the perturbation stream lives on the device,
// so a captured cycle advances it on every replay
__global__ void k_bump_counter(uint64_t *c) {
    launch_wait();
    *c += 1;
}

void launch_bump_counter(uint64_t *c, cudaStream_t s) {
    count_launches(1);
    launch_kernel(k_bump_counter, 1, 1, 0, s, LaunchHow{}, c);
}

__global__ void k_tt_bf16(const double *__restrict__ Tm, __nv_bfloat16 *__restrict__ Tt, int ne,
                          int ld, const int *status) {
    launch_wait();
    if (*status) return;
    const int total = (ne + 1) * ne;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int c = e / ne, a = e % ne;
        Tt[(size_t)c * ld + a] = __double2bfloat16(Tm[e]);
    }
}

void launch_tt_bf16(const double *Tm, __nv_bfloat16 *Tt, int ne, int ld, const int *status,
                    cudaStream_t s) {
    count_launches(1);
    launch_kernel(k_tt_bf16, grid_for((size_t)(ne + 1) * ne, 256), 256, 0, s, LaunchHow{}, Tm, Tt, ne, ld, status);
}

// one thread per Philox block (4 normals)
__global__ void k_normals(uint64_t seed, uint64_t tag, uint64_t ctr0, int64_t count,
                          double *__restrict__ out) {
    launch_wait();
    const int64_t nblk = (count + 3) / 4;
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < nblk; b += (int64_t)gridDim.x * blockDim.x) {
        double z[4];
        philox_normals4(seed, tag, ctr0, (uint64_t)b, z);
#pragma unroll
        for (int l = 0; l < 4; ++l)
            if (4 * b + l < count) out[4 * b + l] = z[l];
    }
}

// the same with a warp per element of 32 Philox blocks (CTAs of 128 threads)
__global__ void __launch_bounds__(128) k_normals1(uint64_t seed, uint64_t tag, uint64_t ctr0, int64_t count,
                                                  double *__restrict__ out) {
    launch_wait();
    const int64_t b = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31), o = 4 * b + (threadIdx.x >> 5);
    if (o < count) out[o] = philox_normal1(seed, tag, ctr0, (uint64_t)b, threadIdx.x >> 5);
}

void launch_normals(uint64_t seed, uint64_t tag, uint64_t ctr0, int64_t count, double *out,
                    cudaStream_t s) {
    if (count <= 0) return;
    count_launches(1);
    const size_t blocks = (size_t)(count + 3) / 4;
    if (single_normals(blocks)) {
        launch_kernel(k_normals1, ceil_div(blocks, 32), 128, 0, s, LaunchHow{}, seed, tag, ctr0, count, out);
        return;
    }
    launch_kernel(k_normals, grid_for((size_t)((count + 3) / 4), 256), 256, 0, s, LaunchHow{}, seed, tag, ctr0, count,
                  out);
}

// ---------------------------------------------------------------------------
// grouped analysis of many problems: one launch per step, block b working on
// block map[b].y of problem map[b].x with the single-problem kernel body
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) kg_restrict(const GroupProb *__restrict__ P, const int2 *__restrict__ map) {
    const int2 e = map[blockIdx.x];
    const GroupProb &g = P[e.x];
    restrict_body<float>(g.fine, g.xstar, 2, 4, g.nc, g.r, e.y, ceil_div(g.nx, 256), g.dC);
}

__global__ void __launch_bounds__(128) kg_obs_apply(const GroupProb *__restrict__ P, const int2 *__restrict__ map) {
    const int2 e = map[blockIdx.x];
    const GroupProb &g = P[e.x];
    const int gx = ceil_div(g.ny, 128);
    obs_apply_body<float>(g.members, g.xstar, g.nx, g.ne, g.ny, g.taps, g.tap_idx, g.tap_w, g.yf, e.y % gx,
                          (e.y / gx) * kObsRows, kObsRows, g.tap_wh, g.tap_wl);
}

__global__ void __launch_bounds__(256) kg_obs_mean(const GroupProb *__restrict__ P, const int2 *__restrict__ map) {
    const int2 e = map[blockIdx.x];
    const GroupProb &g = P[e.x];
    obs_mean_body(g.yf, g.yo_in, g.ne, g.inv_ne, g.ny, g.ybar, g.Z, g.status, e.y, g.yo, g.df.Zh, g.df.Zl);
}

__global__ void __launch_bounds__(128) kg_obs_perturb(const GroupProb *__restrict__ P, const int2 *__restrict__ map) {
    const int2 e = map[blockIdx.x];
    const GroupProb &g = P[e.x];
    obs_perturb_body<true>(g.yf, g.ybar, g.yo, g.eps, 1, g.seed, g.cycle, g.sigma, g.ne, g.ny, g.isq, g.Y, g.Z, e.y,
                           g.df.Yh, g.df.Yl, g.df.Zh, g.df.Zl);
}

__global__ void __launch_bounds__(256) kg_innov_rms(const GroupProb *__restrict__ P, const int2 *__restrict__ map) {
    const GroupProb &g = P[map[blockIdx.x].x];
    innov_rms_body(g.Z + (size_t)g.ne * g.ny, g.ny, g.innov);
}

// block e.y = (z ty + by) tx + bx over the tiles of [S | Y^T R^-1 [D | d*]]
// and the K chunks z (tiles strictly below the diagonal of S are not listed)
__global__ void __launch_bounds__(kDfThreads) kg_gemm(const GroupProb *__restrict__ P, const int2 *__restrict__ map) {
    const int2 e = map[blockIdx.x];
    const GroupProb &g = P[e.x];
    if (*g.status) return;
    const int ne = g.ne, tx = ceil_div(2 * ne + 1, 16), ty = ceil_div(ne, 16);
    const int bx = e.y % tx, by = (e.y / tx) % ty, bz = e.y / (tx * ty);
    const int a0 = by * 16, c0 = bx * 16, n1 = ne, n2 = ne + 1;
    if (c0 < a0) return;  // mirrored from the tile above the diagonal (by the reduction when split)
    const int kb = g.splits > 1 ? bz * g.kchunk : 0, ke = g.splits > 1 ? min(g.ny, kb + g.kchunk) : g.ny;
    const double acc = gemm_df_tile(g.df, ne, g.ny, kb, ke, a0, c0);
    const int a = a0 + (threadIdx.x >> 4), c = c0 + (threadIdx.x & 15);
    if (g.splits == 1)
        gemm_put(acc, a, c, ne, n1, n2, c0 > a0, g.s2, 1.0, g.S, g.Bt);
    else if (a < ne && c < n1 + n2)
        g.part[((size_t)bz * ne + a) * (n1 + n2) + c] = acc;
}

__global__ void __launch_bounds__(256) kg_gemm_reduce(const GroupProb *__restrict__ P, const int2 *__restrict__ map) {
    const int2 e = map[blockIdx.x];
    const GroupProb &g = P[e.x];
    if (*g.status) return;
    gemm_nt_reduce_body(g.part, g.splits, g.ne, g.ne, g.ne + 1, true, g.s2, 1.0, g.S, g.Bt, e.y,
                        ceil_div((size_t)g.ne * (2 * g.ne + 1), 256));
}

// cluster c = blocks 8 c .. 8 c + 7, all of one problem (map entry per cluster)
__global__ void __cluster_dims__(kSpdGroupCluster, 1, 1) __launch_bounds__(kSpdThreads)
    kg_spd_factor(const GroupProb *__restrict__ P, const int2 *__restrict__ map) {
    const GroupProb &g = P[map[blockIdx.x / kSpdGroupCluster].x];
    spd_factor_body<kSpdGroupCluster>(g.S, g.Lt, g.ne, g.status);
}

__global__ void __launch_bounds__(256)  // n <= 160 (group_supported)
    kg_spd_apply(const GroupProb *__restrict__ P, const int2 *__restrict__ map) {
    const int2 e = map[blockIdx.x];
    const GroupProb &g = P[e.x];
    double *x = g.Bt + (size_t)e.y * g.ne;
    spd_apply_body(g.S, g.Lt, g.ne, x, x, g.Tt + (size_t)e.y * g.ldx, g.status);
}

// prolongation of the coarse intervals vj = kProlongIntervals e.y .. + 7 of
// one problem, all fine columns; the problem's scalars and weights are read
// once per block (the table entry is shared by all of the problem's blocks);
// block 0 of each problem advances its analysis counter
constexpr int kProlongIntervals = 8;

__global__ void __launch_bounds__(256) kg_prolong(const GroupProb *__restrict__ P, const int2 *__restrict__ map) {
    __shared__ float wt[kMaxRatio][4];
    __shared__ float *s_fine;
    __shared__ const float *s_dc;
    __shared__ int s_nc, s_r, s_skip;
    const int2 e = map[blockIdx.x];
    if (threadIdx.x == 0) {
        const GroupProb &g = P[e.x];
        if (e.y == 0) *g.cycle += 1;
        s_skip = *g.status;
        s_fine = g.fine;
        s_dc = g.dC;
        s_nc = g.nc;
        s_r = g.r;
    }
    __syncthreads();
    if (s_skip) return;
    const int nc = s_nc, r = s_r, nf = nc * r;
    prolong_stage_weights<float>(P[e.x].pw, r, wt);
    const int vj0 = e.y * kProlongIntervals, vj1 = min(vj0 + kProlongIntervals, 4 * nc);
    for (int fx = threadIdx.x; fx < nf; fx += blockDim.x)
        for (int vj = vj0; vj < vj1; ++vj) prolong2d_interval<float>(s_fine, s_dc, nc, r, wt, fx, vj);
}

bool group_supported(int ne, int ny) {
    // the BF16 rows of the anomalies and T fit the update's shared memory
    return ne >= 2 && ne <= 160 && ny >= 1;
}

void group_plan_free(GroupPlan *plan) {
    if (plan->d_probs) cudaFree(plan->d_probs);
    if (plan->d_maps) cudaFree(plan->d_maps);
    *plan = GroupPlan();
}

bool group_plan_build(GroupPlan *plan, const std::vector<GroupProb> &probs, const std::vector<CUtensorMap> &maps,
                      cudaStream_t s) {
    group_plan_free(plan);
    const int np = (int)probs.size();
    if (np < 1 || maps.size() != 2 * probs.size()) return false;
    std::vector<int2> m[kGsSteps];
    int maxne = 0;
    for (int j = 0; j < np; ++j) {
        const GroupProb &g = probs[j];
        if (!group_supported(g.ne, g.ny) || g.ldx % 16 || g.ldx < g.ne) return false;
        maxne = std::max(maxne, g.ne);
        auto add = [&](int step, long long nb) {
            for (long long b = 0; b < nb; ++b) m[step].push_back(make_int2(j, (int)b));
        };
        add(kGsRestrict, ceil_div(g.nx, 256));
        add(kGsObsApply, (long long)ceil_div(g.ny, 128) * ceil_div(g.ne + 1, kObsRows));
        add(kGsObsMean, ceil_div(g.ny, 32));
        add(kGsPerturb, ceil_div(((long long)g.ne * g.ny + 3) / 4, 128));
        add(kGsInnov, 1);
        {
            const int tx = ceil_div(2 * g.ne + 1, 16), ty = ceil_div(g.ne, 16);
            for (int z = 0; z < g.splits; ++z)
                for (int by = 0; by < ty; ++by)
                    for (int bx = by; bx < tx; ++bx) m[kGsGemm].push_back(make_int2(j, (z * ty + by) * tx + bx));
        }
        if (g.splits > 1) add(kGsReduce, ceil_div((long long)g.ne * (2 * g.ne + 1), 256));
        add(kGsFactor, 1);
        add(kGsSolve, g.ne + 1);
        add(kGsProlong, ceil_div(4 * g.nc, kProlongIntervals));
    }
    // launch shapes (the largest problem's shared memory)
    plan->factor_smem = spd_factor_smem(maxne, kSpdGroupCluster);
    plan->solve_threads = spd_apply_threads(maxne);
    // update: problems grouped by the CTAs per SM their shared memory and TMEM
    // columns allow, one launch per group of at most kUpdateLaunchMax
    {
        auto per_sm = [](size_t smem) { return (int)((size_t)227 * 1024 / smem); };
        std::vector<int> order(np);
        for (int j = 0; j < np; ++j) order[j] = j;
        auto need = [&](int j) {
            const GroupProb &g = probs[j];
            const size_t two = update_tc_smem(g.kblocks, g.ntile, g.ne, 2);
            return update_tc_launch_smem(two <= 200 * 1024 ? two : update_tc_smem(g.kblocks, g.ntile, g.ne, 1),
                                         g.tmem_cols);
        };
        for (int j = 0; j < np; ++j)
            if (need(j) > 200 * 1024) return false;
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return per_sm(need(a)) > per_sm(need(b)); });
        for (size_t k = 0; k < order.size();) {
            GroupPlan::UpdateLaunch L;
            const int cls = per_sm(need(order[k]));
            L.map_begin = (int)m[kGsUpdate].size();
            while (k < order.size() && per_sm(need(order[k])) == cls && (int)L.probs.size() < kUpdateLaunchMax) {
                const int j = order[k++];
                const int q = (int)L.probs.size();
                L.probs.push_back(j);
                for (int t = 0; t < ceil_div(probs[j].nx, 128); ++t) m[kGsUpdate].push_back(make_int2(q, t));
            }
            L.map_end = (int)m[kGsUpdate].size();
            plan->upd.push_back(L);
        }
    }
    plan->upd_maps = maps;
    plan->upd_probs.resize(np);
    for (int j = 0; j < np; ++j) {
        const GroupProb &g = probs[j];
        UpdateProb &u = plan->upd_probs[j];
        u.members = g.members;
        u.dC = g.dC;
        u.status = g.status;
        u.nx = g.nx;
        u.ne = g.ne;
        u.kblocks = g.kblocks;
        u.ntile = g.ntile;
        u.wait_limit = g.wait_limit;
        u.inv_ne = g.inv_ne;
        u.isq = g.isq;
    }
    // one allocation for the table and every map
    size_t total = 0;
    for (int k = 0; k < kGsSteps; ++k) {
        plan->map_off[k] = (int)total;
        plan->nblocks[k] = (int)m[k].size();
        total += m[k].size();
    }
    std::vector<int2> all;
    all.reserve(total);
    for (int k = 0; k < kGsSteps; ++k) all.insert(all.end(), m[k].begin(), m[k].end());
    if (cudaMalloc(&plan->d_probs, np * sizeof(GroupProb)) != cudaSuccess ||
        cudaMalloc(&plan->d_maps, std::max<size_t>(total, 1) * sizeof(int2)) != cudaSuccess) {
        cudaGetLastError();
        group_plan_free(plan);
        return false;
    }
    plan->nprob = np;
    if (cudaMemcpyAsync(plan->d_probs, probs.data(), np * sizeof(GroupProb), cudaMemcpyHostToDevice, s) !=
            cudaSuccess ||
        cudaMemcpyAsync(plan->d_maps, all.data(), total * sizeof(int2), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        group_plan_free(plan);
        return false;
    }
    return true;
}

cudaError_t group_analyse(const GroupPlan &plan, cudaStream_t s) {
    static OncePerDevice attr;
    const cudaError_t ae = attr.run([](int) {
        return cudaFuncSetAttribute(kg_spd_factor, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)spd_factor_smem(kSpdMax, kSpdGroupCluster));
    });
    if (ae != cudaSuccess) return ae;
    const GroupProb *P = plan.d_probs;
    auto M = [&](int k) { return plan.d_maps + plan.map_off[k]; };
    auto n = [&](int k) { return plan.nblocks[k]; };
    int launches = 0;
    auto step = [&](int k) {
        if (n(k)) ++launches;
        return n(k) > 0;
    };
    if (step(kGsRestrict)) kg_restrict<<<n(kGsRestrict), 256, 0, s>>>(P, M(kGsRestrict));
    if (step(kGsObsApply)) kg_obs_apply<<<n(kGsObsApply), 128, 0, s>>>(P, M(kGsObsApply));
    if (step(kGsObsMean)) kg_obs_mean<<<n(kGsObsMean), 256, 0, s>>>(P, M(kGsObsMean));
    if (step(kGsPerturb)) kg_obs_perturb<<<n(kGsPerturb), 128, 0, s>>>(P, M(kGsPerturb));
    if (step(kGsInnov)) kg_innov_rms<<<n(kGsInnov), 256, 0, s>>>(P, M(kGsInnov));
    if (step(kGsGemm)) kg_gemm<<<n(kGsGemm), kDfThreads, 0, s>>>(P, M(kGsGemm));
    if (step(kGsReduce)) kg_gemm_reduce<<<n(kGsReduce), 256, 0, s>>>(P, M(kGsReduce));
    if (step(kGsFactor))
        kg_spd_factor<<<n(kGsFactor) * kSpdGroupCluster, kSpdThreads, plan.factor_smem, s>>>(P, M(kGsFactor));
    if (step(kGsSolve)) kg_spd_apply<<<n(kGsSolve), plan.solve_threads, 0, s>>>(P, M(kGsSolve));
    count_launches(launches);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_update_tc_group(plan, s);
    if (e != cudaSuccess) return e;
    if (n(kGsProlong)) {
        count_launches(1);
        kg_prolong<<<n(kGsProlong), 256, 0, s>>>(P, M(kGsProlong));
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// explicit instantiations
// ---------------------------------------------------------------------------
#define MGK_INST(T)                                                                              \
    template void launch_restrict<T>(const T *, T *, int, int, int, int, cudaStream_t);          \
    template void launch_obs_apply<T>(const T *, const T *, size_t, int, int, int, const int32_t *, \
                                      const double *, double *, cudaStream_t, const float *,     \
                                      const float *);                                            \
    template void launch_ens_anom<T>(const T *, size_t, int, double *, __nv_bfloat16 *,          \
                                     const int *, cudaStream_t);                                 \
    template void launch_update_f64<T>(T *, T *, const double *, const double *, size_t, int,    \
                                       const int *, cudaStream_t);                               \
    template void launch_prolong_add<T>(T *, const T *, int, int, int, int,                      \
                                        const ProlongWeights &, const int *, cudaStream_t);      \
    template void launch_rmse<T>(const T *, const double *, int, size_t, double *, int, double *, \
                                 cudaStream_t);
MGK_INST(float)
MGK_INST(double)
#undef MGK_INST
template void launch_convert<double, float>(const double *, float *, size_t, cudaStream_t);
template void launch_convert<float, double>(const float *, double *, size_t, cudaStream_t);
template void launch_convert<double, double>(const double *, double *, size_t, cudaStream_t);

}  // namespace mgk
