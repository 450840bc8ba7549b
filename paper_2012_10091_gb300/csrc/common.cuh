// common.cuh -- shared device/host helpers of the MGEnKF GPU library.
#pragma once

#include <utility>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <string>

#include "../../include/mgenkf.h"

namespace mgk {

// ---------------------------------------------------------------------------
// Host: run a set-up step once per device.  Kernel attributes (the dynamic
// shared-memory limit) and occupancy figures belong to one device context, so
// a flag shared by all devices would skip the step on the second device.  The
// step runs with the device current; it is retried on the next call if it
// failed.  Thread-safe.
// ---------------------------------------------------------------------------
constexpr int kMaxDevices = 128;
class OncePerDevice {
  public:
    // index of the current device in [0, kMaxDevices), or -1 on error
    static int current() {
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
        return dev;
    }
    template <class F>
    cudaError_t run(F &&f) {
        const int dev = current();
        if (dev < 0) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lock(mu_);
        if (done_[dev]) return cudaSuccess;
        const cudaError_t e = f(dev);
        if (e == cudaSuccess) done_[dev] = true;
        return e;
    }

  private:
    std::mutex mu_;
    bool done_[kMaxDevices] = {};
};

// ---------------------------------------------------------------------------
// launch helpers
// ---------------------------------------------------------------------------
constexpr int kNumSMs = 152;  // GB300: 2 dies x 76 SMs (grids are sized from the device query)

__host__ __device__ inline int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }

// Dynamic shared memory that lets `ctas` CTAs (1 to 3), and no more, share an
// SM (228 KB, 1 KB of it per CTA), or `need` where that is more or no limit is
// asked for.  A launch that becomes ready while another one drains (programmatic
// serialisation above all) is placed on whatever SMs have room at that moment:
// without a limit some SMs take several of its CTAs and others none.
inline size_t residency_smem(size_t need, int ctas) {
    const size_t limit = ctas >= 1 && ctas <= 3 ? (size_t)228 * 1024 / (ctas + 1) - 512 : 0;
    return need > limit ? need : limit;
}

// Launches that follow one another on a stream with programmatic serialisation
// ("chained"): the CTAs of the next launch are placed, and its launch latency
// passes, while the previous one runs.  Every kernel launched so starts with
// launch_wait(): from there on the launches before it have completed and their
// writes are visible, and the next one may be placed.  For the chains of small
// kernels of an analysis (the smallest cycle, 14 launches: 122 us, 98 us chained; three
// layers of the learned correction 26.6 and 20.4 us).
// A launch of long CTAs, about as many as SMs, is better placed on an empty GPU:
// chained, its CTAs take the SMs that have most room while the previous kernel
// runs, several on one where others get none (4096 points, 128 members:
// anomalies 17 us slower, the update 55; 2048 points: the update 190).  Such
// launches say so by their size (the rules stand at the launches).
struct LaunchHow {
    unsigned x = 1, y = 1, z = 1;  // cluster
    bool chained = true;
};
__device__ __forceinline__ void launch_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... P, class... Args>
inline cudaError_t launch_kernel(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                 const LaunchHow &how, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    cfg.numAttrs = 0;
    if (how.chained) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (how.x * how.y * how.z > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = how.x;
        attr[cfg.numAttrs].val.clusterDim.y = how.y;
        attr[cfg.numAttrs++].val.clusterDim.z = how.z;
    }
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// 1 / x for |x| in [2^-995, 2^993): with e = 1 - x y of an approximate reciprocal y
// (relative error 2^-23), y (1 + e + e^2) = (1 - e^3) / x (third-order Newton /
// Householder iteration): 2^-69 beside the rounding of the last step, so the
// quotient correctly rounded but where it lies within 2^-16 of a unit of a tie.
// Three FP64 instructions (64 cycles of a scheduler each), a division about eight.
__device__ __forceinline__ bool recip64_range(double x) {
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) - 0x01c00000u < 0x7c400000u;
}
__device__ __forceinline__ double recip64_in_range(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
// the same for every x (zeros, subnormals, infinities, NaN: the division)
__device__ __forceinline__ double recip64(double x) { return recip64_range(x) ? recip64_in_range(x) : 1.0 / x; }

// device status word values (a subset of mgenkf_status)
constexpr int kStatusOk = 0;

// ---------------------------------------------------------------------------
// Philox4x64-10 (Salmon, Moraes, Dror, Shaw, SC'11) and Box-Muller normals.
// ---------------------------------------------------------------------------
struct U64x4 {
    uint64_t v[4];
};

__device__ __forceinline__ U64x4 philox4x64_10(uint64_t c0, uint64_t c1, uint64_t c2, uint64_t c3,
                                               uint64_t k0, uint64_t k1) {
    const uint64_t M0 = 0xD2E7470EE14C6C93ULL, M1 = 0xCA5A826395121157ULL;
    const uint64_t W0 = 0x9E3779B97F4A7C15ULL, W1 = 0xBB67AE8584CAA73BULL;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t lo0 = M0 * c0, hi0 = __umul64hi(M0, c0);
        const uint64_t lo1 = M1 * c2, hi1 = __umul64hi(M1, c2);
        const uint64_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
        k0 += W0;
        k1 += W1;
    }
    U64x4 o;
    o.v[0] = c0;
    o.v[1] = c1;
    o.v[2] = c2;
    o.v[3] = c3;
    return o;
}

// Normals n = 4 blk .. 4 blk + 3 of the stream (seed, tag, ctr0): Philox block
// (ctr0, blk, 0, 0) with key (seed, tag); lanes (0, 1) and (2, 3) give one
// Box-Muller pair each, u = ((x >> 11) + 1) 2^-53, z = sqrt(-2 ln u1) (cos, sin)(2 pi u2).
__device__ __forceinline__ void philox_normals4(uint64_t seed, uint64_t tag, uint64_t ctr0, uint64_t blk,
                                                double (&z)[4]) {
    const U64x4 x = philox4x64_10(ctr0, blk, 0, 0, seed, tag);
    const double inv53 = 1.0 / 9007199254740992.0;
#pragma unroll
    for (int pair = 0; pair < 2; ++pair) {
        const double u1 = (double)((x.v[2 * pair] >> 11) + 1) * inv53;
        const double u2 = (double)((x.v[2 * pair + 1] >> 11) + 1) * inv53;
        const double rad = sqrt(-2.0 * log(u1));
        const double th = 6.283185307179586 * u2;
        z[2 * pair] = rad * cos(th);
        z[2 * pair + 1] = rad * sin(th);
    }
}

// one of those four, l (where a warp has one l, it runs one trigonometric function)
__device__ __forceinline__ double philox_normal1(uint64_t seed, uint64_t tag, uint64_t ctr0, uint64_t blk, int l) {
    const U64x4 x = philox4x64_10(ctr0, blk, 0, 0, seed, tag);
    const double inv53 = 1.0 / 9007199254740992.0;
    const uint64_t a = l < 2 ? x.v[0] : x.v[2], b = l < 2 ? x.v[1] : x.v[3];
    const double u1 = (double)((a >> 11) + 1) * inv53;
    const double u2 = (double)((b >> 11) + 1) * inv53;
    const double rad = sqrt(-2.0 * log(u1));
    const double th = 6.283185307179586 * u2;
    return l & 1 ? rad * sin(th) : rad * cos(th);
}

// Normals per thread: the four of a Philox block, or one each on the four warps of
// a CTA of 128 threads while that gives at most two CTAs per SM (`blocks` Philox
// blocks).  A normal is a chain of some 100 FP64 instructions of 64 cycles and
// four share part of it: 512 normals 11 us by fours, 7 us one each; 65536 take
// 11 us by fours and would take more one each.
inline bool single_normals(size_t blocks) { return blocks <= (size_t)2 * kNumSMs * 32; }

// The same four normals with the Box-Muller transform evaluated in FP32 on
// the same Philox words (each uniform rounded to FP32 first): within about
// 1e-6 of the FP64 values, without GB300's slow FP64 logarithm and sines.
__device__ __forceinline__ void philox_normals4_f32(uint64_t seed, uint64_t tag, uint64_t ctr0, uint64_t blk,
                                                    double (&z)[4]) {
    const U64x4 x = philox4x64_10(ctr0, blk, 0, 0, seed, tag);
#pragma unroll
    for (int pair = 0; pair < 2; ++pair) {
        const float u1 = __ull2float_rn((x.v[2 * pair] >> 11) + 1) * 0x1p-53f;
        const float u2 = __ull2float_rn((x.v[2 * pair + 1] >> 11) + 1) * 0x1p-53f;
        const float rad = sqrtf(-2.0f * logf(u1));
        float sn, cs;
        sincosf(6.2831853071795865f * u2, &sn, &cs);
        z[2 * pair] = (double)(rad * cs);
        z[2 * pair + 1] = (double)(rad * sn);
    }
}

constexpr uint64_t kEpsTag = 0x45505300ULL;  // "EPS\0": perturbation stream of the analysis

// ---------------------------------------------------------------------------
// small type helpers
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ double to_f64(T x) {
    return (double)x;
}

}  // namespace mgk

namespace mgk {
// number of kernel launches issued by the library (process-wide counter)
void count_launches(int n);
}  // namespace mgk

// error text of the stateless entry points (per host thread)
void mgk_set_error(const std::string &msg);
