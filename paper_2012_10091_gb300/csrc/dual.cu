// dual.cu -- multigrid Dual EnKF with parameter estimation on the Burgers
// inlet model (Sec. 4: Eqs. burgers and inlet-1D-Burgers; Algorithm 3 with its
// parameter rows, run inside Algorithm 4), FP64.
//
// Model: nodes x_j = j dx; node 0 holds the inlet u0 (1 + theta1 sin(omega t +
// theta2)), the outlet node is extrapolated linearly, the interior follows the
// flux-form central scheme; SSP-RK3 in Shu-Osher form with the inlet set at
// each stage's time.  A CTA or a cluster advances one grid held in shared memory.
//
// One cycle (mgenkf_dual_cycle):
//   fine forecast with the analysed parameter mean of the previous cycle;
//   parameter forecast theta^f = theta^a + tau (random walk, Philox normals);
//   member forecast with theta^f; perturbed observations; parameter update
//   theta^a = theta^f + Theta T, T = (I + Y^T R^-1 Y)^-1 Y^T R^-1 D (ensemble
//   space, exact R = sigma^2 I); member forecast again from the previous
//   analysis with theta^a; state update x^a = x^f + X T with the same
//   perturbations; fine correction x^F += Pi_F(X T_ne) with d* = y^o - H^C x^C*.
// Projections are open-grid 4-point Lagrange interpolants (one-sided at the
// ends); H^C is the Pi_F row at each observed fine node.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/mgenkf.h"
#include "analysis.h"
#include "common.cuh"

namespace mgk {

constexpr uint64_t kThetaTag = 0x54485441ULL;  // "THTA": parameter random walk
constexpr int kDualMaxPts = 1024;               // points per grid

// SSP-RK3 steps of nprob inlet-Burgers grids of n points, each on a cluster of
// CTAs (gridDim.x / nprob of them; one CTA where CLUSTER is false, a thread per
// node of the grid).  CTA r of a cluster owns nodes [r per, (r + 1) per) and
// carries 3 nodes of its neighbours on each side, one thread per node: stage 1 is evaluated two nodes into them,
// stage 2 one node, so that the CTAs exchange values once per step (3 nodes
// written to each neighbour's shared memory, double-buffered: a neighbour may
// still be in the step before) and a stage ends in a barrier of the CTA.
//
// Bound by the FP64 pipes: a warp instruction takes 64 cycles of its scheduler,
// so the arithmetic is kept to 20 per step: with a = dt / (4 dx), c = 4 nu / dx,
// s = v_{j-1} + v_{j+1},
//   k = c (s - 2 v_j) + (v_{j-1} - v_{j+1}) s,  dt L = a k,
//   u1 = x + a k0,  u2 = x + a/4 (k0 + k1),  x' = x + a/6 (k0 + k1 + 4 k2),
// the Shu-Osher form rearranged around x (against extended precision after 3000
// steps: 1e-15, with the weights 1/3 and 2/3 on x and u2, whose rounding errors
// add up, 1e-13).
// The inlet values of 32 steps are formed together by 64 threads (a sine takes
// some 50 dependent FP64 instructions); the outlet is extrapolated by the one
// thread that reads it.  30 steps: 100 grids of 200 nodes 176 -> 60 us, one of
// 800 (a cluster of 8, where one SM did all of it) 441 -> 48 us.
constexpr int kInletSteps = 32;  // steps of inlet values formed together
constexpr int kInletHalo = 3;    // nodes of each neighbour that a CTA of a cluster carries
__device__ __forceinline__ void inlet_push(double *local, int rank, double v) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(local), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(r), "d"(v) : "memory");
}

template <bool CLUSTER>
__global__ void __launch_bounds__(1024) k_burgers_inlet(double *__restrict__ u, int n, int ctas, int per, double a,
                                                        double c, double dt, int nsteps, double t0,
                                                        const double *__restrict__ theta, double u0, double omega) {
    launch_wait();
    extern __shared__ double sh[];
    __shared__ double inlet[2 * kInletSteps];
    constexpr int H = CLUSTER ? kInletHalo : 0;
    const int pitch = per + 2 * H;
    double *X = sh, *B = sh + 2 * pitch, *C = sh + 3 * pitch;  // x (two buffers), u1, u2
    const int prob = CLUSTER ? blockIdx.x / ctas : blockIdx.x, rank = CLUSTER ? blockIdx.x - prob * ctas : 0;
    // nodes [lo, hi) are this CTA's; slot j holds node lo - H + j
    const int lo = rank * per, hi = min(n, lo + per);
    const int j = threadIdx.x, k = lo - H + j;
    double *g = u + (size_t)prob * n;
    const double th1 = theta[2 * prob], th2 = theta[2 * prob + 1];
    const bool held = j < pitch && k >= 0 && k < min(n, hi + H);
    const bool own = held && k >= lo && k < hi;
    const bool first = held && k == 0, last = held && k == n - 1, before_last = held && k == n - 2;
    // nodes with both neighbours in this CTA
    const bool in = held && k > 0 && k < n - 1 && j > 0 && k < hi + 2;
    if (held) {
        X[j] = g[k];
        B[j] = C[j] = X[pitch + j] = 0.0;
    }
    const double a4 = 0.25 * a, a6 = a / 6.0;
    auto rate = [&](double vm, double v, double vp) {
        const double sum = vm + vp;
        return fma(c, fma(-2.0, v, sum), (vm - vp) * sum);
    };
    if (CLUSTER) {
        // every CTA of the cluster runs and its buffers are set
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
    for (int s = 0; s < nsteps; ++s) {
        if (s % kInletSteps == 0 && lo == 0) {
            if (j < 2 * min(kInletSteps, nsteps - s)) {
                const double t = t0 + (s + (j >> 1)) * dt;
                inlet[j] = u0 * (1.0 + th1 * sin(omega * (j & 1 ? t + 0.5 * dt : t + dt) + th2));
            }
        }
        if (!CLUSTER || s % kInletSteps == 0) __syncthreads();
        const double bc = inlet[2 * (s % kInletSteps)], bch = inlet[2 * (s % kInletSteps) + 1];
        const double *xc = X + (s & 1) * pitch;
        double *an = X + ((s & 1) ^ 1) * pitch;
        double x = 0.0, y = 0.0, kk = 0.0;
        if (in) {
            x = xc[j];
            const double vm = xc[j - 1], vp = before_last && s > 0 ? 2.0 * x - vm : xc[j + 1];
            kk = rate(vm, x, vp);
            y = fma(a, kk, x);
            B[j] = y;
        }
        if (first) B[j] = bc;
        __syncthreads();
        double z = 0.0;
        if (in) {
            const double vm = B[j - 1], vp = before_last ? 2.0 * y - vm : B[j + 1];
            kk += rate(vm, y, vp);
            z = fma(a4, kk, x);
            C[j] = z;
        }
        if (first) C[j] = bch;
        __syncthreads();
        double w = first ? bc : 0.0;
        if (in) {
            const double vm = C[j - 1], vp = before_last ? 2.0 * z - vm : C[j + 1];
            w = fma(a6, fma(4.0, rate(vm, z, vp), kk), x);
        }
        if (own) {
            an[j] = w;
            if (CLUSTER) {
                // slot of node k in a neighbour: k - (its lo - H)
                if (j < 2 * H && rank > 0) inlet_push(an + j + per, rank - 1, w);
                if (j >= per && rank + 1 < ctas) inlet_push(an + j - per, rank + 1, w);
            }
        }
        if (CLUSTER) {
            asm volatile("barrier.cluster.arrive.release;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        }
    }
    if (!CLUSTER) __syncthreads();
    const double *xc = X + (nsteps & 1) * pitch;
    if (own) g[k] = last && nsteps > 0 ? 2.0 * xc[j - 1] - xc[j - 2] : xc[j];
}

// theta^f = theta^a + sqrt(q) tau
__global__ void k_theta_walk(const double *__restrict__ theta, const double *__restrict__ tau, double sq, int count,
                             double *__restrict__ theta_f) {
    launch_wait();
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < count) theta_f[e] = theta[e] + sq * tau[e];
}

// theta^a_i = theta^f_i + sum_a Theta[p][a] T[a][i], Theta the normalised
// parameter anomalies (T column i at Tm[i ne ..]), and the mean of theta^a.  A
// cluster of kThetaCtas: each takes ne / kThetaCtas members, a warp per member
// over the lanes, and the first sums the CTAs' means (one CTA with a thread per
// member and parameter, chains of 3 ne FP64 instructions: 37 us for 100
// members, 17 us so).
constexpr int kThetaCtas = 8, kThetaWarps = 8;
__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__global__ void __cluster_dims__(kThetaCtas, 1, 1) __launch_bounds__(32 * kThetaWarps)
    k_theta_update(const double *__restrict__ theta_f, const double *__restrict__ Tm, int ne,
                   double inv_ne, double isq, double *__restrict__ theta_a, double *__restrict__ theta_mean,
                   const int *status) {
    launch_wait();
    __shared__ double part[kThetaCtas][2], mine[kThetaWarps][2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rank = blockIdx.x;
    const bool ok = *status == 0;
    double s0 = 0.0, s1 = 0.0;
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    if (ok) {
        double m0 = 0.0, m1 = 0.0;
        for (int a = lane; a < ne; a += 32) {
            m0 += theta_f[2 * a];
            m1 += theta_f[2 * a + 1];
        }
        m0 = warp_sum(m0) * inv_ne;
        m1 = warp_sum(m1) * inv_ne;
        for (int i = rank * kThetaWarps + warp; i < ne; i += kThetaCtas * kThetaWarps) {
            double a0 = 0.0, a1 = 0.0;
            for (int a = lane; a < ne; a += 32) {
                const double t = Tm[(size_t)i * ne + a];
                a0 = fma(theta_f[2 * a] - m0, t, a0);
                a1 = fma(theta_f[2 * a + 1] - m1, t, a1);
            }
            a0 = fma(warp_sum(a0), isq, theta_f[2 * i]);
            a1 = fma(warp_sum(a1), isq, theta_f[2 * i + 1]);
            if (lane == 0) {
                theta_a[2 * i] = a0;
                theta_a[2 * i + 1] = a1;
            }
            s0 += a0;
            s1 += a1;
        }
        if (lane == 0) {
            mine[warp][0] = s0;
            mine[warp][1] = s1;
        }
        __syncthreads();
    }
    // every CTA of the cluster runs (its shared memory may be written)
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    if (ok && threadIdx.x < 2) {
        double m = 0.0;
        for (int w = 0; w < kThetaWarps; ++w) m += mine[w][threadIdx.x];
        inlet_push(&part[rank][threadIdx.x], 0, m);
    }
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    if (ok && rank == 0 && threadIdx.x < 2) {
        double m = 0.0;
        for (int r = 0; r < kThetaCtas; ++r) m += part[r][threadIdx.x];
        theta_mean[threadIdx.x] = m * inv_ne;
    }
}

// fine += Pi_F(dC) on the open grid: 4 taps from j0[k]
__global__ void k_prolong_open(double *__restrict__ fine, const double *__restrict__ dC, int nf,
                               const int32_t *__restrict__ j0, const double *__restrict__ w, const int *status) {
    launch_wait();
    if (*status) return;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nf) return;
    const double *wk = w + 4 * (size_t)k;
    const double *d = dC + j0[k];
    fine[k] += wk[0] * d[0] + wk[1] * d[1] + wk[2] * d[2] + wk[3] * d[3];
}

}  // namespace mgk

using namespace mgk;

struct mgenkf_dual {
    mgenkf_dual_config cfg;
    int nf = 0, nc = 0, ne = 0, ny = 0;
    double t = 0.0;
    uint64_t cycle = 0;
    cudaStream_t stream = nullptr;
    cudaStream_t aux = nullptr;  // the fine forecast runs beside the members' forecasts and first analysis
    cudaEvent_t ev[2] = {nullptr, nullptr};
    double *xstar_a = nullptr;   // x^C* stand-in of the parameter analysis (its d* column is not used)
    double *fine = nullptr, *members = nullptr, *prev = nullptr, *theta = nullptr, *theta_f = nullptr;
    double *theta_mean = nullptr, *tau = nullptr, *xstar = nullptr, *dC = nullptr;
    double *yf = nullptr, *yo = nullptr, *ybar = nullptr, *eps = nullptr, *Y = nullptr, *Z = nullptr;
    double *X = nullptr, *S = nullptr, *Lt = nullptr, *Bt = nullptr, *part = nullptr;
    double *tap_w = nullptr, *pro_w = nullptr;
    int32_t *tap_idx = nullptr, *pro_j0 = nullptr;
    uint64_t *cycle_d = nullptr;
    int *status = nullptr;
    std::string err;
};

namespace {

// cubic Lagrange weights through nodes j0 .. j0 + 3 at position s (coarse index units)
void lagrange4(int j0, double s, double w[4]) {
    for (int a = 0; a < 4; ++a) {
        double v = 1.0;
        for (int b = 0; b < 4; ++b)
            if (b != a) v *= (s - (j0 + b)) / (double)(a - b);
        w[a] = v;
    }
}

int open_j0(int k, int r, int nc) {
    int j0 = k / r - 1;
    if (j0 > nc - 4) j0 = nc - 4;
    if (j0 < 0) j0 = 0;
    return j0;
}

void free_dual(mgenkf_dual *d) {
    void *p[] = {d->fine, d->members, d->prev, d->theta, d->theta_f, d->theta_mean, d->tau, d->xstar, d->dC,
                 d->yf, d->yo, d->ybar, d->eps, d->Y, d->Z, d->X, d->S, d->Lt, d->Bt, d->part, d->tap_w,
                 d->pro_w, d->tap_idx, d->pro_j0, d->cycle_d, d->status};
    for (void *q : p)
        if (q) cudaFree(q);
    if (d->xstar_a) cudaFree(d->xstar_a);
    for (cudaEvent_t e : d->ev)
        if (e) cudaEventDestroy(e);
    if (d->aux) cudaStreamDestroy(d->aux);
}

// CTAs per grid: the fewest that leave one warp to each scheduler, while the
// grids do not exceed the SMs (then each gets one)
int inlet_ctas(int nprob, int n) {
    int c = 1;
    while (c < 8 && ceil_div(n, c) + 2 * kInletHalo > 128 && nprob * 2 * c <= kNumSMs) c *= 2;
    return c;
}

cudaError_t forecast(mgenkf_dual *d, double *grids, int nprob, int n, const double *theta, int nsteps,
                     cudaStream_t s = nullptr) {
    count_launches(1);
    const int ctas = inlet_ctas(nprob, n), per = ceil_div(n, ctas);
    const double dx = d->cfg.length / n, dt = d->cfg.dt;
    const double a = dt / (4.0 * dx), c = 4.0 * d->cfg.nu / dx;
    // a thread per node held (1024 for the largest grid, which one CTA holds alone);
    // 64 threads form the inlet values
    const int held = per + (ctas > 1 ? 2 * kInletHalo : 0);
    const int threads = std::max(64, ceil_div(held, 32) * 32);
    const cudaError_t e = launch_kernel(ctas > 1 ? k_burgers_inlet<true> : k_burgers_inlet<false>, nprob * ctas,
                                        threads, 4 * held * sizeof(double), s ? s : d->stream,
                                        LaunchHow{(unsigned)ctas}, grids, n, ctas, per, a, c, dt, nsteps, d->t, theta,
                                        d->cfg.u0, d->cfg.omega);
    if (e != cudaSuccess) cudaGetLastError();  // reported by the caller, not left pending
    return e;
}

// perturbations (generated once per cycle), anomalies and T = S^-1 B (ensemble space)
void gain_solve(mgenkf_dual *d, int gen_eps, const double *xstar) {
    const cudaStream_t s = d->stream;
    const int ne = d->ne, ny = d->ny;
    launch_obs_apply<double>(d->members, xstar, d->nc, ne, ny, 4, d->tap_idx, d->tap_w, d->yf, s);
    launch_obs_mean(d->yf, d->yo, ne, ny, d->ybar, d->Z, d->status, s);
    launch_obs_perturb(d->yf, d->ybar, d->yo, d->eps, gen_eps, d->cfg.seed, d->cycle_d, d->cfg.obs_sigma, ne,
                       ny, d->Y, d->Z, s);
    const double s2 = d->cfg.obs_sigma * d->cfg.obs_sigma;
    launch_gemm_nt_f64(d->Y, ne, d->Y, ne, d->Z, ne + 1, ny, s2, 1.0, d->S, d->Bt, d->status, s, d->part);
    launch_spd_factor(d->S, d->Lt, ne, d->status, s);
    launch_spd_solve(d->S, d->Lt, ne, d->Bt, d->Bt, ne + 1, nullptr, 0, d->status, s);
}

}  // namespace

#define D_FAIL(code, msg) \
    do {                  \
        d->err = (msg);   \
        return (code);    \
    } while (0)
#define D_CUDA(x)                                                                          \
    do {                                                                                   \
        cudaError_t e_ = (x);                                                              \
        if (e_ != cudaSuccess) D_FAIL(MGENKF_ERR_CUDA, std::string(cudaGetErrorString(e_))); \
    } while (0)

extern "C" mgenkf_status mgenkf_dual_create(const mgenkf_dual_config *cfg, const int32_t *obs_index,
                                            void *cuda_stream, mgenkf_dual_t *out) {
    if (!cfg || !obs_index || !out) return MGENKF_ERR_INVALID_ARG;
    *out = nullptr;
    const mgenkf_dual_config &c = *cfg;
    if (c.ratio < 1 || c.ratio > 16 || c.n_fine % c.ratio != 0 || c.n_fine > kDualMaxPts ||
        c.n_fine / c.ratio < 8 || c.n_members < 2 || c.n_members > 256 || c.n_obs < 1 ||
        !(c.dt > 0.0) || !(c.length > 0.0) || !(c.nu >= 0.0) || !(c.obs_sigma > 0.0) || !(c.theta_q >= 0.0)) {
        mgk_set_error("mgenkf_dual_create: sizes or parameters out of range");
        return MGENKF_ERR_INVALID_ARG;
    }
    for (int j = 0; j < c.n_obs; ++j)
        if (obs_index[j] < 0 || obs_index[j] >= c.n_fine) {
            mgk_set_error("mgenkf_dual_create: observation index outside the fine grid");
            return MGENKF_ERR_INVALID_ARG;
        }
    mgenkf_dual *d = new mgenkf_dual();
    d->cfg = c;
    d->nf = c.n_fine;
    d->nc = c.n_fine / c.ratio;
    d->ne = c.n_members;
    d->ny = c.n_obs;
    d->stream = (cudaStream_t)cuda_stream;
    const size_t ne = d->ne, ny = d->ny, nc = d->nc, nf = d->nf;
    struct A {
        void **p;
        size_t bytes;
    } al[] = {
        {(void **)&d->fine, nf * 8}, {(void **)&d->members, ne * nc * 8}, {(void **)&d->prev, ne * nc * 8},
        {(void **)&d->theta, 2 * ne * 8}, {(void **)&d->theta_f, 2 * ne * 8}, {(void **)&d->theta_mean, 2 * 8},
        {(void **)&d->tau, 2 * ne * 8 + 32}, {(void **)&d->xstar, nc * 8}, {(void **)&d->dC, nc * 8},
        {(void **)&d->yf, (ne + 1) * ny * 8}, {(void **)&d->yo, ny * 8}, {(void **)&d->ybar, ny * 8},
        {(void **)&d->eps, ne * ny * 8}, {(void **)&d->Y, ne * ny * 8}, {(void **)&d->Z, (ne + 1) * ny * 8},
        {(void **)&d->X, ne * nc * 8}, {(void **)&d->S, ne * ne * 8}, {(void **)&d->Lt, ne * ne * 8},
        {(void **)&d->Bt, (ne + 1) * ne * 8},
        {(void **)&d->part, (size_t)gemm_nt_splits((int)ne, (int)ne, (int)ne + 1, (int)ny) * ne * (2 * ne + 1) * 8},
        {(void **)&d->tap_w, ny * 4 * 8}, {(void **)&d->pro_w, nf * 4 * 8}, {(void **)&d->tap_idx, ny * 4 * 4},
        {(void **)&d->pro_j0, nf * 4}, {(void **)&d->cycle_d, 8}, {(void **)&d->status, 4},
        {(void **)&d->xstar_a, nc * 8},
    };
    for (auto &a : al) {
        if (cudaMalloc(a.p, a.bytes) != cudaSuccess) {
            cudaGetLastError();
            free_dual(d);
            delete d;
            mgk_set_error("mgenkf_dual_create: device allocation failed");
            return MGENKF_ERR_OOM;
        }
    }
    // open-grid H^C taps (absolute coarse indices) and Pi_F rows
    std::vector<int32_t> ti(ny * 4), pj(nf);
    std::vector<double> tw(ny * 4), pw(nf * 4);
    for (size_t k = 0; k < nf; ++k) {
        const int j0 = open_j0((int)k, c.ratio, d->nc);
        pj[k] = j0;
        lagrange4(j0, (double)k / c.ratio, &pw[4 * k]);
    }
    for (size_t j = 0; j < ny; ++j) {
        const int k = obs_index[j];
        for (int t = 0; t < 4; ++t) {
            ti[4 * j + t] = pj[k] + t;
            tw[4 * j + t] = pw[4 * (size_t)k + t];
        }
    }
    if (cudaStreamCreateWithFlags(&d->aux, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&d->ev[0], cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&d->ev[1], cudaEventDisableTiming) != cudaSuccess ||
        cudaMemsetAsync(d->xstar_a, 0, nc * 8, d->stream) != cudaSuccess) {
        cudaGetLastError();
        free_dual(d);
        delete d;
        mgk_set_error("mgenkf_dual_create: stream or event creation failed");
        return MGENKF_ERR_CUDA;
    }
    const uint64_t zero = 0;
    const int zs = 0;
    bool ok = cudaMemcpyAsync(d->tap_idx, ti.data(), ti.size() * 4, cudaMemcpyHostToDevice, d->stream) == cudaSuccess &&
              cudaMemcpyAsync(d->tap_w, tw.data(), tw.size() * 8, cudaMemcpyHostToDevice, d->stream) == cudaSuccess &&
              cudaMemcpyAsync(d->pro_j0, pj.data(), pj.size() * 4, cudaMemcpyHostToDevice, d->stream) == cudaSuccess &&
              cudaMemcpyAsync(d->pro_w, pw.data(), pw.size() * 8, cudaMemcpyHostToDevice, d->stream) == cudaSuccess &&
              cudaMemcpyAsync(d->cycle_d, &zero, 8, cudaMemcpyHostToDevice, d->stream) == cudaSuccess &&
              cudaMemcpyAsync(d->status, &zs, 4, cudaMemcpyHostToDevice, d->stream) == cudaSuccess &&
              cudaStreamSynchronize(d->stream) == cudaSuccess;
    if (!ok) {
        free_dual(d);
        delete d;
        mgk_set_error("mgenkf_dual_create: CUDA error during set-up");
        return MGENKF_ERR_CUDA;
    }
    *out = d;
    return MGENKF_OK;
}

extern "C" mgenkf_status mgenkf_dual_set_state(mgenkf_dual_t d, const double *fine, const double *members,
                                               const double *theta, const double *theta_fine, double t0) {
    if (!d || !fine || !members || !theta || !theta_fine) return MGENKF_ERR_INVALID_ARG;
    d->err.clear();
    D_CUDA(cudaMemcpyAsync(d->fine, fine, d->nf * 8, cudaMemcpyDefault, d->stream));
    D_CUDA(cudaMemcpyAsync(d->members, members, (size_t)d->ne * d->nc * 8, cudaMemcpyDefault, d->stream));
    D_CUDA(cudaMemcpyAsync(d->theta, theta, 2 * (size_t)d->ne * 8, cudaMemcpyDefault, d->stream));
    D_CUDA(cudaMemcpyAsync(d->theta_mean, theta_fine, 2 * 8, cudaMemcpyDefault, d->stream));
    D_CUDA(cudaStreamSynchronize(d->stream));
    d->t = t0;
    return MGENKF_OK;
}

extern "C" mgenkf_status mgenkf_dual_free_run(mgenkf_dual_t d, int32_t nsteps) {
    if (!d || nsteps < 0) return MGENKF_ERR_INVALID_ARG;
    d->err.clear();
    if (nsteps == 0) return MGENKF_OK;
    D_CUDA(forecast(d, d->fine, 1, d->nf, d->theta_mean, nsteps));
    D_CUDA(forecast(d, d->members, d->ne, d->nc, d->theta, nsteps));
    D_CUDA(cudaGetLastError());
    d->t += nsteps * d->cfg.dt;
    return MGENKF_OK;
}

extern "C" mgenkf_status mgenkf_dual_cycle(mgenkf_dual_t d, int32_t nsteps, const double *y_obs) {
    if (!d || nsteps < 1 || !y_obs) return MGENKF_ERR_INVALID_ARG;
    d->err.clear();
    const cudaStream_t s = d->stream;
    const int ne = d->ne, nc = d->nc;
    D_CUDA(cudaMemcpyAsync(d->yo, y_obs, d->ny * sizeof(double), cudaMemcpyDefault, s));
    // Algorithm 4 step 2: the fine run with the analysed parameter mean, on the
    // auxiliary stream beside the members' forecasts and the parameter analysis
    // (theta_mean is rewritten only after the join below)
    D_CUDA(cudaEventRecord(d->ev[0], s));
    D_CUDA(cudaStreamWaitEvent(d->aux, d->ev[0], 0));
    const cudaError_t fine = forecast(d, d->fine, 1, d->nf, d->theta_mean, nsteps, d->aux);
    launch_restrict<double>(d->fine, d->xstar, 1, 1, nc, d->cfg.ratio, d->aux);
    D_CUDA(cudaEventRecord(d->ev[1], d->aux));
    // Algorithm 3 step 2: parameter random walk, members forecast with theta^f
    D_CUDA(cudaMemcpyAsync(d->prev, d->members, (size_t)ne * nc * 8, cudaMemcpyDeviceToDevice, s));
    launch_normals(d->cfg.seed, kThetaTag, d->cycle, 2 * (int64_t)ne, d->tau, s);
    count_launches(1);
    launch_kernel(k_theta_walk, ceil_div(2 * ne, 256), 256, 0, s, LaunchHow{},
                  d->theta, d->tau, std::sqrt(d->cfg.theta_q), 2 * ne, d->theta_f);
    const cudaError_t members = forecast(d, d->members, ne, nc, d->theta_f, nsteps);
    // steps 3-5: perturbed observations, parameter update theta^a = theta^f + Theta T
    if (members == cudaSuccess) gain_solve(d, 1, d->xstar_a);
    D_CUDA(cudaStreamWaitEvent(s, d->ev[1], 0));  // join: the fine forecast has read theta_mean
    D_CUDA(fine);                                 // no analysis of grids that have not moved
    D_CUDA(members);
    count_launches(1);
    launch_kernel(k_theta_update, kThetaCtas, 32 * kThetaWarps, 0, s, LaunchHow{},
                  d->theta_f, d->Bt, ne, 1.0 / ne, 1.0 / std::sqrt(ne - 1.0), d->theta, d->theta_mean, d->status);
    // steps 6-8: members forecast again from the previous analysis with theta^a, state update
    D_CUDA(cudaMemcpyAsync(d->members, d->prev, (size_t)ne * nc * 8, cudaMemcpyDeviceToDevice, s));
    D_CUDA(forecast(d, d->members, ne, nc, d->theta, nsteps));
    gain_solve(d, 0, d->xstar);  // the same perturbations
    launch_ens_anom<double>(d->members, nc, ne, d->X, nullptr, d->status, s);
    D_CUDA(cudaMemsetAsync(d->dC, 0, nc * sizeof(double), s));
    launch_update_f64<double>(d->members, d->dC, d->X, d->Bt, nc, ne, d->status, s);
    // Algorithm 4 step 5: x^F += Pi_F(x^C' - x^C*)
    count_launches(1);
    launch_kernel(k_prolong_open, ceil_div(d->nf, 256), 256, 0, s, LaunchHow{}, d->fine, d->dC, d->nf, d->pro_j0,
                  d->pro_w, d->status);
    launch_bump_counter(d->cycle_d, s);
    D_CUDA(cudaGetLastError());
    d->t += nsteps * d->cfg.dt;
    d->cycle += 1;
    return MGENKF_OK;
}

extern "C" mgenkf_status mgenkf_dual_get_state(mgenkf_dual_t d, double *fine, double *members, double *theta,
                                               double *theta_fine) {
    if (!d) return MGENKF_ERR_INVALID_ARG;
    d->err.clear();
    D_CUDA(cudaStreamSynchronize(d->stream));
    int st = 0;
    D_CUDA(cudaMemcpy(&st, d->status, sizeof(int), cudaMemcpyDeviceToHost));
    if (fine) D_CUDA(cudaMemcpy(fine, d->fine, d->nf * 8, cudaMemcpyDefault));
    if (members) D_CUDA(cudaMemcpy(members, d->members, (size_t)d->ne * d->nc * 8, cudaMemcpyDefault));
    if (theta) D_CUDA(cudaMemcpy(theta, d->theta, 2 * (size_t)d->ne * 8, cudaMemcpyDefault));
    if (theta_fine) D_CUDA(cudaMemcpy(theta_fine, d->theta_mean, 2 * 8, cudaMemcpyDefault));
    if (st) D_FAIL((mgenkf_status)st, "a device-side check failed (non-positive pivot or non-finite observation)");
    return MGENKF_OK;
}

extern "C" const char *mgenkf_dual_last_error(mgenkf_dual_t d) { return d ? d->err.c_str() : ""; }

extern "C" mgenkf_status mgenkf_dual_destroy(mgenkf_dual_t d) {
    if (!d) return MGENKF_OK;
    cudaStreamSynchronize(d->stream);
    free_dual(d);
    delete d;
    return MGENKF_OK;
}
