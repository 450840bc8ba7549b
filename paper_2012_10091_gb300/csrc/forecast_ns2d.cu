// forecast_ns2d.cu -- batched SSP-RK3 forecast of the 2-D compressible
// Navier-Stokes equations (Eqs. Mass, Momentum, Energy) on periodic grids.
//
// State: 4 planes (rho, rho u, rho v, E) of n x n points, x fastest.  With
// u = (rho u)/rho, v = (rho v)/rho, p = (gamma-1)(E - rho |u|^2 / 2), T = p/rho:
//   dq/dt = -(F_{i+1} - F_{i-1}) / (2h) - (G_{j+1} - G_{j-1}) / (2h)
//           + (Fv_{i+1/2} - Fv_{i-1/2}) / h + (Gv_{j+1/2} - Gv_{j-1/2}) / h
// with nodal inviscid fluxes F = (rho u, rho u u + p, rho u v, (E + p) u),
// G = (rho v, rho v u, rho v v + p, (E + p) v) and face viscous/heat fluxes
// Fv = (0, t_xx, t_xy, t_xx u_f + t_xy v_f + kappa T_x) (normal derivatives
// compact across the face, tangential ones the average of the two central
// differences, face velocities the average of the two nodes), likewise Gv;
// t_xx = mu (4/3 u_x - 2/3 v_y), t_xy = mu (u_y + v_x), kappa = mu gamma /
// ((gamma - 1) Pr).  Every flux telescopes, so the four totals are conserved.
//
// GPU design, FP32 (the mixed path): one launch per time step over every grid
// of the cycle (Ne members and the fine run, or every grid of a batch), the
// three RK stages fused.  A persistent CTA walks tiles of TX x 2H points.  For
// each tile it copies the step-start state of the tile and a 3-point halo
// (periodic wrap) into shared memory, then evaluates stage 1 on the tile grown
// by 2 points, stage 2 on the tile grown by 1 and stage 3 on the tile, each
// stage reading the previous one from shared memory (the halo points are
// recomputed by the neighbouring tiles): per point and step the state is read
// once and written once.  Stages: s1 = u0 + k(u0), s2 = u0 + ((s1 - u0) +
// k(s1))/4, u' = u0 + 2/3 ((s2 - u0) + k(s2)), k = dt L (Shu-Osher form
// rearranged).  The step writes a second state buffer (a neighbouring tile may
// still read the old state's halo), so the steps alternate between the state
// and one scratch buffer; an odd step count ends with a copy back.
//
// Every thread works on pairs of points folded into float2: shared element
// (r, c) holds rows r and r + H of the tile's halo block, so every
// shared-memory access is 64 bits wide and every arithmetic instruction is a
// packed FFMA2 / FADD2 / FMUL2 on both points.
//
// FP64 states use one launch per stage, a row march with every flux formed once
// (ns2d_march64); s1 and s2 live in two scratch buffers.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <algorithm>
#include <vector>
#include <type_traits>

#include "common.cuh"
#include "forecast_ns2d.h"

namespace mgk {

constexpr int kNsTx = 32;
constexpr int kNsTileRows = 32;  // rows of a tile of the fused FP32 step (32 x 32 points)

// ---------------------------------------------------------------------------
// FP64: one launch per RK stage, a march down the rows
//
// GB300 issues an FP64 instruction of a warp per SM sub-partition in 64 cycles,
// whatever its lanes do (76 with all four sub-partitions busy), so the stage
// costs its FP64 instructions times the warps on the busiest sub-partition;
// shared memory, integer work and barriers are nearly free beside them.  The
// march therefore forms every quantity once: primitives and nodal fluxes at
// their node (the reciprocal of rho by a third-order iteration), the x-face
// fluxes by the thread west of the face, the y-face fluxes once per row, and
// hands them on through shared memory or registers; 80 FP64 instructions per
// point and stage, against about 180 for 32 x 8 tiles that formed the fluxes at
// every neighbour, four faces per node, a division per node and a 1.33-fold
// halo of nodes.
//
// Four warps per CTA, one point of a row per thread.  A unit is a strip of
// columns (the whole periodic width up to 128 points per side, else equal
// strips of at most 128) by `rows` rows of one grid; narrow grids put several
// units side by side in a CTA, so that all four sub-partitions work.  A strip's
// two halo columns (and the face west of its first column) are formed for all
// of its rows at once before the march, a lane per node: an instruction for two
// lanes per row would cost as much as one for 32.  Step k of the march takes in
// row k - 1 of the unit and finishes row k - 2, two barriers per step.
//
// Measured (10 steps): one 512^2 grid 2.74 -> 1.49 ms, 32 members of 64^2 and a
// 256^2 fine run 2.38 -> 1.34 ms; 80 instructions at 608 G/s would be 1.03, 0.78 ms.
// ---------------------------------------------------------------------------
constexpr int kN64Threads = 128;

struct Ns64Args {
    NsGroup<double> g[2];  // tx: strips per grid, ty: runs of rows
    int ctas0, rows;       // CTAs of group 0, rows per unit
    double gm1, k2;        // gamma - 1, 2 kappa / mu
    double c1[2], c2[2];   // -dt / (2h), dt mu / h^2 of each group
};

// what a node contributes: u, v, T' = k2 T, rho u, rho v and the nodal fluxes
// F = (rho u, F1, F2, F3), G = (rho v, F2, G2, G3)
struct Node64 {
    double U, V, T, mx, my, F1, F2, F3, G2, G3;
};
__device__ __forceinline__ Node64 node64(double rho, double mx, double my, double E, double gm1, double k2) {
    Node64 q;
    const double ri = recip64(rho);
    q.mx = mx;
    q.my = my;
    q.U = mx * ri;
    q.V = my * ri;
    const double p = fma(-0.5 * gm1, fma(mx, q.U, my * q.V), gm1 * E);
    q.T = p * (k2 * ri);
    const double H = E + p;
    q.F1 = fma(mx, q.U, p);
    q.F2 = mx * q.V;
    q.F3 = H * q.U;
    q.G2 = fma(my, q.V, p);
    q.G3 = H * q.V;
    return q;
}

// viscous and heat flux of the face between a and b in units of mu / h (normal
// stress, shear stress, twice the work and heat): dn, dt differences across the
// face of the normal and tangential velocity, sn, st their sums, tn (tt) the sum
// over a and b of the tangential difference of the normal (tangential) velocity
struct Face64 {
    double n, t, e;
};
__device__ __forceinline__ Face64 face64(double dn, double dt, double sn, double st, double tn, double tt, double dT) {
    Face64 f;
    f.n = fma(4.0 / 3.0, dn, (-1.0 / 6.0) * tt);
    f.t = fma(0.25, tn, dt);
    f.e = fma(f.n, sn, fma(f.t, st, dT));
    return f;
}

// doubles of shared memory: two rows of seven published values, the y
// differences of u, v, the x faces, and the halo columns of a strip
__host__ __device__ constexpr int n64_smem_doubles(int rows) { return 19 * kN64Threads + (rows + 2) * 22; }

template <int STAGE>
__global__ void __launch_bounds__(kN64Threads) ns2d_march64(Ns64Args A) {
    extern __shared__ double n64_sm[];
    constexpr int NT = kN64Threads;
    const int tid = threadIdx.x;
    const int gi = (int)blockIdx.x >= A.ctas0 ? 1 : 0;
    const NsGroup<double> G = gi ? A.g[1] : A.g[0];
    const double c1 = gi ? A.c1[1] : A.c1[0], c2 = gi ? A.c2[1] : A.c2[0];
    const int n = G.n, TX = (n + G.tx - 1) / G.tx, pitch = (TX + 31) & ~31, upc = NT / pitch;
    // with halo columns (strips: one unit per CTA) every thread has the CTA's unit,
    // also those past its columns or its pitch: they all fill in halo nodes
    const bool halo = G.tx > 1;
    const int sub = halo ? 0 : tid / pitch, i = tid - sub * pitch;
    const long long unit = (long long)((int)blockIdx.x - (gi ? A.ctas0 : 0)) * upc + sub;
    const int per_grid = G.tx * G.ty;
    const int prob = (int)(unit / per_grid), rem = (int)(unit - (long long)prob * per_grid);
    const int strip = rem / G.ty, seg = rem - strip * G.ty;
    const int x0 = strip * TX, w = min(TX, n - x0), y0 = seg * A.rows, rows = min(A.rows, n - y0);
    const bool mine = sub < upc && prob < G.nprob, act = mine && i < w;  // has a unit, has a column of it
    const size_t plane = (size_t)n * n, off = (size_t)(mine ? prob : 0) * 4 * plane;
    const double *u0 = G.u0 + off;
    const double *in = STAGE == 0 ? u0 : (STAGE == 1 ? G.s1 : G.s2) + off;
    double *out = (STAGE == 0 ? G.s1 : STAGE == 1 ? G.s2 : G.u0) + off;
    const double gm1 = A.gm1, k2 = A.k2;
    auto wrap = [n](int g) { return g < 0 ? g + n : g >= n ? g - n : g; };

    double *P = n64_sm;             // [row parity][U V T mx F1 F2 F3][thread]
    double *D = P + 14 * NT;        // [u, v differences in y][thread]
    double *F = D + 2 * NT;         // [face east of the thread][thread]
    double *HP = F + 3 * NT;        // [row][west, east column][7]
    double *HC = HP + (A.rows + 2) * 14;  // [row][U V T] of the first column
    double *HD = HC + (A.rows + 2) * 3;   // [row][2] y differences of the east column
    double *HF = HD + (A.rows + 2) * 2;   // [row][3] the face west of the first column
    const bool he = halo && i == w - 1, hw = halo && i == 0;
    const int te = i == w - 1 ? tid - (w - 1) : tid + 1, tw = i == 0 ? tid + w - 1 : tid - 1;
    // the previous launch has completed; the next one may be placed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (halo) {  // uniform over the CTA
        for (int e = tid; e < 3 * (rows + 2); e += NT) {
            const int k = e / 3, c = e - 3 * k;
            const size_t o = (size_t)wrap(y0 - 1 + k) * n + wrap(c == 0 ? x0 - 1 : c == 1 ? x0 : x0 + w);
            const Node64 q = node64(in[o], in[plane + o], in[2 * plane + o], in[3 * plane + o], gm1, k2);
            if (c == 1) {
                HC[3 * k] = q.U;
                HC[3 * k + 1] = q.V;
                HC[3 * k + 2] = q.T;
            } else {
                const double v[7] = {q.U, q.V, q.T, q.mx, q.F1, q.F2, q.F3};
                double *h = HP + 14 * k + (c ? 7 : 0);
#pragma unroll
                for (int f = 0; f < 7; ++f) h[f] = v[f];
            }
        }
        __syncthreads();
        for (int e = tid; e < rows; e += NT) {
            const int k = e + 1;
            const double *a = HP + 14 * k, *b = HC + 3 * k;
            const double uy = (a[14] - a[-14]) + (b[3] - b[-3]), vy = (a[15] - a[-13]) + (b[4] - b[-2]);
            const Face64 f = face64(b[0] - a[0], b[1] - a[1], a[0] + b[0], a[1] + b[1], uy, vy, b[2] - a[2]);
            HF[3 * k] = f.n;
            HF[3 * k + 1] = f.t;
            HF[3 * k + 2] = f.e;
            HD[2 * k] = a[14 + 7] - a[-14 + 7];
            HD[2 * k + 1] = a[15 + 7] - a[-13 + 7];
        }
        // read after the first barrier of the march
    }

    double q[4] = {1.0, 0.0, 0.0, 0.0}, qc[4] = {0.0, 0.0, 0.0, 0.0};
    const size_t col = (size_t)(act ? x0 + i : 0);
    auto load = [&](int k) {
        const size_t o = (size_t)wrap(y0 - 1 + k) * n + col;
#pragma unroll
        for (int f = 0; f < 4; ++f) q[f] = in[f * plane + o];
    };
    if (act) load(0);
    Node64 m1{}, cc{}, p1{};
    double uxc = 0.0, vxc = 0.0;
    Face64 yf{};
    for (int k = 0; k < A.rows + 2; ++k) {
        const bool have = act && k < rows + 2, fin = have && k >= 2;
        double *Pk = P + (k & 1) * 7 * NT, *Pc = P + ((k + 1) & 1) * 7 * NT;
        double qn[4] = {0.0, 0.0, 0.0, 0.0}, base[4] = {0.0, 0.0, 0.0, 0.0};
        if (have) {
            m1 = cc;
            cc = p1;
            p1 = node64(q[0], q[1], q[2], q[3], gm1, k2);
            Pk[tid] = p1.U;
            Pk[NT + tid] = p1.V;
            Pk[2 * NT + tid] = p1.T;
            Pk[3 * NT + tid] = p1.mx;
            Pk[4 * NT + tid] = p1.F1;
            Pk[5 * NT + tid] = p1.F2;
            Pk[6 * NT + tid] = p1.F3;
        }
        double uy = 0.0, vy = 0.0;
        const size_t oc = (size_t)wrap(y0 - 2 + k) * n + col;
        if (fin) {
            uy = p1.U - m1.U;
            vy = p1.V - m1.V;
            D[tid] = uy;
            D[NT + tid] = vy;
            if (STAGE > 0)
#pragma unroll
                for (int f = 0; f < 4; ++f) base[f] = u0[f * plane + oc];
        }
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            qn[f] = qc[f];  // the row to finish in this step
            qc[f] = q[f];
        }
        if (act && k + 1 < rows + 2) load(k + 1);
        __syncthreads();
        double uxk = 0.0, vxk = 0.0;
        Face64 top{}, fe{};
        double r[4] = {0.0, 0.0, 0.0, 0.0};
        if (have) {
            const double *hk = HP + 14 * k;
            uxk = (he ? hk[7] : Pk[te]) - (hw ? hk[0] : Pk[tw]);
            vxk = (he ? hk[8] : Pk[NT + te]) - (hw ? hk[1] : Pk[NT + tw]);
            if (k >= 1)
                top = face64(p1.V - cc.V, p1.U - cc.U, cc.V + p1.V, cc.U + p1.U, vxk + vxc, uxk + uxc, p1.T - cc.T);
        }
        if (fin) {
            const double *hc = HP + 14 * (k - 1);
            const double Ue = he ? hc[7] : Pc[te], Ve = he ? hc[8] : Pc[NT + te], Te = he ? hc[9] : Pc[2 * NT + te];
            const double uye = he ? HD[2 * (k - 1)] : D[te], vye = he ? HD[2 * (k - 1) + 1] : D[NT + te];
            fe = face64(Ue - cc.U, Ve - cc.V, cc.U + Ue, cc.V + Ve, uy + uye, vy + vye, Te - cc.T);
            F[tid] = fe.n;
            F[NT + tid] = fe.t;
            F[2 * NT + tid] = fe.e;
            double dx[4];
#pragma unroll
            for (int f = 0; f < 4; ++f)
                dx[f] = (he ? hc[10 + f] : Pc[(3 + f) * NT + te]) - (hw ? hc[3 + f] : Pc[(3 + f) * NT + tw]);
            r[0] = dx[0] + (p1.my - m1.my);
            r[1] = dx[1] + (p1.F2 - m1.F2);
            r[2] = dx[2] + (p1.G2 - m1.G2);
            r[3] = dx[3] + (p1.G3 - m1.G3);
        }
        __syncthreads();
        if (fin) {
            const double *hf = HF + 3 * (k - 1);
            const double wn = hw ? hf[0] : F[tw], wt = hw ? hf[1] : F[NT + tw], we = hw ? hf[2] : F[2 * NT + tw];
            const double v[4] = {0.0, (fe.n - wn) + (top.t - yf.t), (fe.t - wt) + (top.n - yf.n),
                                 (fe.e - we) + (top.e - yf.e)};
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                const double cv = f == 3 ? 0.5 * c2 : c2;
                double res;
                if (STAGE == 0) {
                    res = qn[f] + (f == 0 ? c1 * r[0] : fma(cv, v[f], c1 * r[f]));
                } else {
                    double t = fma(c1, r[f], qn[f] - base[f]);
                    if (f > 0) t = fma(cv, v[f], t);
                    res = fma(STAGE == 1 ? 0.25 : 2.0 / 3.0, t, base[f]);
                }
                out[f * plane + oc] = res;
            }
        }
        uxc = uxk;
        vxc = vxk;
        yf = top;
    }
}

// ---------------------------------------------------------------------------
// FP32: folded pairs of points in float2, packed arithmetic, fused RK stages
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
// a - b with one rounding (packed subtraction; no constant operand)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    unsigned long long ra, rb, rd;
    memcpy(&ra, &a, 8);
    memcpy(&rb, &b, 8);
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
    float2 d;
    memcpy(&d, &rd, 8);
    return d;
}
// a b.  A product that goes into one sum only becomes a fused multiply-add of it
// in the assembler, one with two uses does not; volatile keeps the compiler from
// sharing a product between two rows of the march, so that each kernel rounds
// every flux alike and the kernels agree bit for bit.
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    unsigned long long ra, rb, rd;
    memcpy(&ra, &a, 8);
    memcpy(&rb, &b, 8);
    asm volatile("mul.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
    float2 d;
    memcpy(&d, &rd, 8);
    return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// approximate reciprocal in one instruction (__fdividef(1, x) spends six more on
// |x| above 2^126, where both give 0)
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ int wrap_index(int g, int n) {
    if (g < 0) g += n;
    if (g >= n) {
        g -= n;
        if (g >= n) g %= n;  // only grids narrower than a tile
    }
    return g;
}

// 4-byte asynchronous global -> shared copy
__device__ __forceinline__ void cp_async4(float *smem, const float *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(gmem) : "memory");
}
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}
// 16-byte asynchronous global -> shared copy (L2 only: each chunk is read once per tile)
__device__ __forceinline__ void cp_async16(void *smem, const float *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// ---------------------------------------------------------------------------
// The FP32 step on 2-D tiles (the per-handle path: the members and the fine
// run in one persistent launch).  A CTA walks tiles of TX x 2H points; for each
// it copies the step-start state of the tile and a 3-point halo into shared
// memory, evaluates stage 1 on the tile grown by 2 points, stage 2 on the
// tile grown by 1 and stage 3 on the tile, each stage reading the previous
// one from shared memory.  Shared element (r, c) holds rows r and r + H of the
// halo block (one float2).
// ---------------------------------------------------------------------------
// where the tiles of a launch come from: a device table of groups (batched
// path) or the two groups of one handle.  next() moves gi forward to the
// group holding `tile`; a CTA visits its tiles in increasing order.
struct PairTiles {
    NsGroup<float> g[2];  // g[1].tile_begin = tiles of g[0]
    __device__ __forceinline__ void next(int tile, int &gi) const { gi = tile < g[1].tile_begin ? 0 : 1; }
    // no runtime index into the parameter array
    __device__ __forceinline__ NsGroup<float> group(int gi) const { return gi ? g[1] : g[0]; }
};

// what every thread needs of one tile, prepared by thread 0 two tiles ahead
struct TileDesc {
    const float *in;  // step-start state (4 planes of the grid)
    float *out;       // state after the step
    int n, x0, y0, pad;
    float inv_h, inv_2h, dt, pad2;
};

// Steps alternate between the grid's state (u0) and its scratch buffer (s1):
// parity 0 reads u0 and writes s1, parity 1 the reverse.
template <int TX, int H, class Tiles>
__device__ __forceinline__ void make_desc(const Tiles &src, int tile, int &gi, int parity, TileDesc *d) {
    src.next(tile, gi);
    const NsGroup<float> G = src.group(gi);
    const int local = tile - G.tile_begin;
    const int tiles_per_prob = G.tx * G.ty;
    const int prob = local / tiles_per_prob;
    const int tt = local - prob * tiles_per_prob;
    const int ty = tt / G.tx;
    const int n = G.n;
    const size_t off = (size_t)prob * 4 * n * n;
    float *u0 = G.u0 + off, *other = G.s1 + off;
    d->in = parity ? other : u0;
    d->out = parity ? u0 : other;
    d->n = n;
    d->x0 = (tt - ty * G.tx) * TX;
    d->y0 = ty * (2 * H);
    d->inv_h = G.inv_h;
    d->inv_2h = G.inv_2h;
    d->dt = G.dt;
}

// dq/dt of the folded pair at shared index c (9-point stencil); `cons` holds
// the conserved planes (rho, rho u, rho v, E), `prim` u, v, p, T, each HALO
// elements long
template <int HX, int HALO>
__device__ __forceinline__ void x2_rhs(const float2 *cons, const float2 *prim, int c, float inv_h, float inv_2h,
                                       float mu, float kap, float2 (&L)[4]) {
    const int e_ = c + 1, w_ = c - 1, n_ = c + HX, s_ = c - HX;
    const float2 *Q1 = cons + HALO, *Q2 = cons + 2 * HALO, *Q3 = cons + 3 * HALO;
    const float2 *U = prim, *V = prim + HALO, *P = prim + 2 * HALO, *TT = prim + 3 * HALO;
    const float2 mi2h = f2(-inv_2h);
    float2 r[4];
    {   // inviscid part: central differences of the nodal fluxes
        const float2 mxe = Q1[e_], mxw = Q1[w_], myn = Q2[n_], mys = Q2[s_];
        const float2 Ue = U[e_], Uw = U[w_], Vn = V[n_], Vs = V[s_];
        const float2 Pe = P[e_], Pw = P[w_], Pn = P[n_], Ps = P[s_];
        const float2 Fe1 = fma2(mxe, Ue, Pe), Fw1 = fma2(mxw, Uw, Pw);
        const float2 Fe2 = mul2(mxe, V[e_]), Fw2 = mul2(mxw, V[w_]);
        const float2 Fe3 = mul2(add2(Q3[e_], Pe), Ue), Fw3 = mul2(add2(Q3[w_], Pw), Uw);
        const float2 Gn1 = mul2(myn, U[n_]), Gs1 = mul2(mys, U[s_]);
        const float2 Gn2 = fma2(myn, Vn, Pn), Gs2 = fma2(mys, Vs, Ps);
        const float2 Gn3 = mul2(add2(Q3[n_], Pn), Vn), Gs3 = mul2(add2(Q3[s_], Ps), Vs);
        r[0] = mul2(add2(sub2(mxe, mxw), sub2(myn, mys)), mi2h);
        r[1] = mul2(add2(sub2(Fe1, Fw1), sub2(Gn1, Gs1)), mi2h);
        r[2] = mul2(add2(sub2(Fe2, Fw2), sub2(Gn2, Gs2)), mi2h);
        r[3] = mul2(add2(sub2(Fe3, Fw3), sub2(Gn3, Gs3)), mi2h);
    }
    // viscous and heat fluxes on the four faces of the node.  The 1/h and
    // 1/(4h) of the derivatives sit in the stress coefficients, and the 1/2 of
    // the face velocities (and a factor 2 on the heat flux) in the final
    // 1/(2h) of the energy equation: the face fluxes of the discretisation,
    // with fewer multiplications.
    const float2 c43 = f2(4.f / 3.f), m16 = f2(-1.f / 6.f), q4 = f2(0.25f);
    const float2 k2 = f2(mu > 0.f ? 2.f * kap / mu : 0.f), mh2 = f2(mu * inv_h * inv_h), hmh2 = f2(0.5f * mu * inv_h * inv_h);
    float2 fx[2][3], fy[2][3];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        {   // x-face between columns a and b = a + 1
            const int a = side ? c : w_, b = side ? e_ : c;
            const float2 Ua = U[a], Ub = U[b], Va = V[a], Vb = V[b];
            const float2 dU = sub2(Ub, Ua), dV = sub2(Vb, Va);
            const float2 tU = add2(sub2(U[a + HX], U[a - HX]), sub2(U[b + HX], U[b - HX]));
            const float2 tV = add2(sub2(V[a + HX], V[a - HX]), sub2(V[b + HX], V[b - HX]));
            const float2 txx = fma2(c43, dU, mul2(m16, tV)), txy = fma2(q4, tU, dV);
            fx[side][0] = txx;
            fx[side][1] = txy;
            // 2 x (work + heat): txx (Ua + Ub) + txy (Va + Vb) + 2 kappa dT / h
            fx[side][2] = fma2(txx, add2(Ua, Ub), fma2(txy, add2(Va, Vb), mul2(k2, sub2(TT[b], TT[a]))));
        }
        {   // y-face between rows a and b = a + 1
            const int a = side ? c : s_, b = side ? n_ : c;
            const float2 Ua = U[a], Ub = U[b], Va = V[a], Vb = V[b];
            const float2 dU = sub2(Ub, Ua), dV = sub2(Vb, Va);
            const float2 tU = add2(sub2(U[a + 1], U[a - 1]), sub2(U[b + 1], U[b - 1]));
            const float2 tV = add2(sub2(V[a + 1], V[a - 1]), sub2(V[b + 1], V[b - 1]));
            const float2 tyy = fma2(c43, dV, mul2(m16, tU)), txy = fma2(q4, tV, dU);
            fy[side][0] = txy;
            fy[side][1] = tyy;
            fy[side][2] = fma2(txy, add2(Ua, Ub), fma2(tyy, add2(Va, Vb), mul2(k2, sub2(TT[b], TT[a]))));
        }
    }
    L[0] = r[0];
#pragma unroll
    for (int k = 1; k < 3; ++k)
        L[k] = fma2(add2(sub2(fx[1][k - 1], fx[0][k - 1]), sub2(fy[1][k - 1], fy[0][k - 1])), mh2, r[k]);
    L[3] = fma2(add2(sub2(fx[1][2], fx[0][2]), sub2(fy[1][2], fy[0][2])), hmh2, r[3]);
}

// primitives u, v, p, T of a folded pair of conserved values (one approximate
// reciprocal of rho per point)
template <int HALO>
__device__ __forceinline__ void put_prims(float2 *prim, int f, float2 rho, float2 mx, float2 my, float2 E, float gm1) {
    const float2 rinv = make_float2(rcp_approx(rho.x), rcp_approx(rho.y));
    const float2 u = mul2(mx, rinv), v = mul2(my, rinv);
    const float2 ke = mul2(mul2(f2(0.5f), rho), fma2(u, u, mul2(v, v)));
    const float2 p = mul2(f2(gm1), sub2(E, ke));
    prim[f] = u;
    prim[HALO + f] = v;
    prim[2 * HALO + f] = p;
    prim[3 * HALO + f] = mul2(p, rinv);
}

// Shared memory of the fused step for tiles of TX x 2H points (TX x H folded
// pairs) with a 3-point halo.
template <int TX, int H>
struct StepSmem {
    static constexpr int NT = 256;                 // threads per CTA
    static constexpr int FX = TX + 6, FR = H + 6;  // folded block: columns x0-3 .., rows r and r + H of rows y0-3 ..
    static constexpr int NF = FX * FR;             // folded elements per array
    // raw block of the step-start state: rows y0 - 3 .. y0 + 2H + 2, columns
    // x0 - 4 .. x0 + TX + 3 (16-byte aligned), 4 planes, row-major
    static constexpr int RW = TX + 8, RR = 2 * H + 6, RAW = 4 * RR * RW;  // floats
    static constexpr int CHUNKS = 4 * RR * (RW / 4);                      // 16-byte copies per tile
    static constexpr int COPIES = (CHUNKS + NT - 1) / NT;                 // per thread
    // u0 (4 arrays), the current stage (4), its primitives (4), raw block, 4 descriptors
    static constexpr size_t bytes() { return sizeof(float2) * 12 * NF + sizeof(float) * RAW + 4 * sizeof(TileDesc); }
    static_assert((TX * H) % NT == 0, "the last stage gives every thread the same number of pairs");
};

// Issue the 16-byte copies of one tile's raw block.  Copy c of a thread is
// (plane, row, chunk); x0 - 4 and n are multiples of 4, so a chunk never
// straddles the periodic wrap.
template <int TX, int H>
__device__ __forceinline__ void step_issue(const TileDesc &d, float *raw) {
    using S = StepSmem<TX, H>;
    const int n = d.n, plane = n * n;  // 4 planes of one grid stay below 2^31 elements
#pragma unroll
    for (int q = 0; q < S::COPIES; ++q) {
        const int c = threadIdx.x + q * S::NT;
        if (c < S::CHUNKS) {
            // plane k, raw row r, first column x of the chunk (divisions by constants)
            const int row = c / (S::RW / 4), k = row / S::RR, r = row - k * S::RR, x = 4 * (c - row * (S::RW / 4));
            const float *src = d.in + k * plane + wrap_index(d.y0 - 3 + r, n) * n + wrap_index(d.x0 - 4 + x, n);
            cp_async16(raw + row * S::RW + x, src);
        }
    }
}

// Fold the raw block (folded element (r, c) holds raw rows r and r + H at raw
// column c + 1) into u0 and form its primitives.
template <int TX, int H>
__device__ __forceinline__ void step_fold(const float *raw, float2 *Q0, float2 *PR, float gm1) {
    using S = StepSmem<TX, H>;
    constexpr int NF = S::NF, PL = S::RR * S::RW;
    for (int e = threadIdx.x; e < NF; e += S::NT) {
        const int r = e / S::FX, c = e - r * S::FX;
        const float *pa = raw + r * S::RW + c + 1, *pb = pa + H * S::RW;
        const float2 rho = make_float2(pa[0], pb[0]);
        const float2 mx = make_float2(pa[PL], pb[PL]);
        const float2 my = make_float2(pa[2 * PL], pb[2 * PL]);
        const float2 E = make_float2(pa[3 * PL], pb[3 * PL]);
        Q0[e] = rho;
        Q0[NF + e] = mx;
        Q0[2 * NF + e] = my;
        Q0[3 * NF + e] = E;
        put_prims<NF>(PR, e, rho, mx, my, E, gm1);
    }
}

// Stage K (1 or 2) on the folded block shrunk by K on every side: reads the
// previous stage (u0 for K = 1) and its primitives, and after a barrier
// replaces them with this stage's values (the results wait in registers).
template <int TX, int H, int K>
__device__ __forceinline__ void step_stage(const float2 *Q0, float2 *QS, float2 *PR, const TileDesc &d, float gm1,
                                           float mu, float kap) {
    using S = StepSmem<TX, H>;
    constexpr int W = S::FX - 2 * K, R = S::FR - 2 * K, N = W * R, E = (N + S::NT - 1) / S::NT, NF = S::NF;
    const float2 *cons = K == 1 ? Q0 : QS;
    const float2 dt = f2(d.dt);
    float2 res[E][4];
    int fo[E];
#pragma unroll
    for (int q = 0; q < E; ++q) {
        const int e = threadIdx.x + q * S::NT;
        fo[q] = -1;
        if (e < N) {
            const int r = e / W, c = e - r * W;
            const int f = (r + K) * S::FX + c + K;
            fo[q] = f;
            float2 L[4];
            x2_rhs<S::FX, NF>(cons, PR, f, d.inv_h, d.inv_2h, mu, kap, L);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 base = Q0[k * NF + f];
                res[q][k] = K == 1 ? fma2(dt, L[k], base) : fma2(f2(0.25f), fma2(dt, L[k], sub2(QS[k * NF + f], base)), base);
            }
        }
    }
    __syncthreads();  // every read of the previous stage is done
#pragma unroll
    for (int q = 0; q < E; ++q) {
        const int f = fo[q];
        if (f >= 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k) QS[k * NF + f] = res[q][k];
            put_prims<NF>(PR, f, res[q][0], res[q][1], res[q][2], res[q][3], gm1);
        }
    }
    __syncthreads();  // this stage is complete
}

// Stage 3 on the tile itself, straight to the output state.
template <int TX, int H>
__device__ __forceinline__ void step_last(const float2 *Q0, const float2 *QS, const float2 *PR, const TileDesc &d,
                                          float mu, float kap) {
    using S = StepSmem<TX, H>;
    constexpr int E = TX * H / S::NT, NF = S::NF;
    const float2 dt = f2(d.dt);
    const int n = d.n, plane = n * n;
#pragma unroll
    for (int q = 0; q < E; ++q) {
        const int e = threadIdx.x + q * S::NT;
        const int r = e / TX, c = e - r * TX;
        const int f = (r + 3) * S::FX + c + 3;
        const int x = d.x0 + c, ya = d.y0 + r, yb = ya + H;
        if (x >= n || ya >= n) continue;
        float2 L[4];
        x2_rhs<S::FX, NF>(QS, PR, f, d.inv_h, d.inv_2h, mu, kap, L);
        float *oa = d.out + ya * n + x, *ob = oa + H * n;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 base = Q0[k * NF + f];
            const float2 res = fma2(f2(2.f / 3.f), fma2(dt, L[k], sub2(QS[k * NF + f], base)), base);
            oa[k * plane] = res.x;
            if (yb < n) ob[k * plane] = res.y;
        }
    }
}

// One SSP-RK3 step of every tile of a launch.  Persistent: each CTA walks
// tiles blockIdx.x, + gridDim.x, ...; the raw block of the next tile is
// copied while the three stages of the current one run; thread 0 describes
// tiles two ahead (4 descriptor slots).
template <int TX, int H, int MINB, class Tiles>
__global__ void __launch_bounds__(256, MINB)
    ns2d_rk3_step(Tiles src, int total_tiles, int parity, float gm1, float mu, float kap) {
    using S = StepSmem<TX, H>;
    constexpr int NF = S::NF;
    extern __shared__ float4 step_smem4[];
    float2 *Q0 = reinterpret_cast<float2 *>(step_smem4);
    float2 *QS = Q0 + 4 * NF;
    float2 *PR = QS + 4 * NF;
    float *raw = reinterpret_cast<float *>(PR + 4 * NF);
    TileDesc *desc = reinterpret_cast<TileDesc *>(raw + S::RAW);
    const int G = gridDim.x;
    // Steps follow one another with programmatic serialisation (see
    // step_launch): the next step may be scheduled from here on, and its CTAs
    // take the SMs as this launch's CTAs leave; each CTA describes its first
    // tiles (static tables only) before it waits for the previous launch to
    // complete and its writes to be visible.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int tile = blockIdx.x;
    if (tile >= total_tiles) return;
    int gi = 0;  // thread 0: group of the last tile it described
    if (threadIdx.x == 0)
        for (int q = 0; q < 2; ++q)
            if (tile + q * G < total_tiles) make_desc<TX, H>(src, tile + q * G, gi, parity, &desc[q]);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    step_issue<TX, H>(desc[0], raw);
    cp_async_commit();
    for (int it = 0; tile < total_tiles; ++it, tile += G) {
        cp_async_wait0();  // this tile's raw block has landed
        __syncthreads();   // ... for every thread; the previous tile is done everywhere
        step_fold<TX, H>(raw, Q0, PR, gm1);
        __syncthreads();   // the raw block is free, u0 and its primitives are ready
        if (tile + G < total_tiles) step_issue<TX, H>(desc[(it + 1) & 3], raw);
        cp_async_commit();
        if (threadIdx.x == 0 && tile + 2 * G < total_tiles)
            make_desc<TX, H>(src, tile + 2 * G, gi, parity, &desc[(it + 2) & 3]);
        const TileDesc &d = desc[it & 3];
        step_stage<TX, H, 1>(Q0, QS, PR, d, gm1, mu, kap);
        step_stage<TX, H, 2>(Q0, QS, PR, d, gm1, mu, kap);
        step_last<TX, H>(Q0, QS, PR, d, mu, kap);
    }
}

// ---------------------------------------------------------------------------
// The FP32 step as a column march.  A unit (one CTA) is two row segments of
// grids of one size, each a band of columns; thread t owns column c0 + t of
// both, as the two halves of a float2, so that the neighbours of a pair are
// pairs too (with two columns of one row in a pair the values at the fold had
// to be swapped: 45 of 840 instructions a step).  With one band the T =
// blockDim.x threads span the whole periodic width; with several each band
// carries a 3-column halo on both sides, recomputed by its neighbours.  The
// CTA marches down the rows of its segments: in step j it takes row j of the
// step-start state (3 rows above the segment first; copied asynchronously three
// steps ahead), evaluates stage 1 one row behind, stage 2 three rows behind and
// stage 3 five rows behind, and stores the new state's row.  Each stage keeps
// the three rows of its input around the row it evaluates in registers (its own
// column); only the east and west neighbours come from shared memory, through
// ring buffers of the last rows each stage published (one barrier per step).
// The face between two rows is evaluated once and carried to the next row.
// Bound by the latency of a step (one or two warps per scheduler, 40% of the
// issue slots).  512^2 / 128^2 x 64 handle, 10 steps: 514 us with pairs of
// columns, ring rows of a pitch known at run time and rows moved through the
// register windows (840 instructions a step), 372 us as below (450); 24
// problems of 64^2 .. 768^2: 8.13 and 6.2 ms with their analysis.
// ---------------------------------------------------------------------------
// one row of a stage input at the thread's column pair
struct Rec {
    float2 rho, mx, my, E, U, V, P, T;
};

// primitives u, v, p, T of a pair of conserved values (one approximate
// reciprocal of rho per point)
__device__ __forceinline__ Rec make_rec(float2 rho, float2 mx, float2 my, float2 E, float gm1) {
    Rec r;
    r.rho = rho;
    r.mx = mx;
    r.my = my;
    r.E = E;
    const float2 rinv = make_float2(rcp_approx(rho.x), rcp_approx(rho.y));
    r.U = mul2(mx, rinv);
    r.V = mul2(my, rinv);
    const float2 ke = mul2(mul2(f2(0.5f), rho), fma2(r.U, r.U, mul2(r.V, r.V)));
    r.P = mul2(f2(gm1), sub2(E, ke));
    r.T = mul2(r.P, rinv);
    return r;
}

// Viscous and heat fluxes of one face, in units of mu/h (pure-number stress
// coefficients; the 1/2 of the face velocities and a factor 2 on the heat
// flux are in the final 1/(2h) of the energy equation).  tU, tV: sums of the
// two central tangential differences of u and v across the face.
struct Face {
    float2 f0, f1, f2;
};
// x-face between columns a and b = a + 1: (t_xx, t_xy, 2 x (work + heat))
__device__ __forceinline__ Face face_x(float2 Ua, float2 Ub, float2 Va, float2 Vb, float2 tU, float2 tV, float2 Ta,
                                       float2 Tb, float2 k2) {
    const float2 dU = sub2(Ub, Ua), dV = sub2(Vb, Va);
    const float2 txx = fma2(f2(4.f / 3.f), dU, mul2(f2(-1.f / 6.f), tV)), txy = fma2(f2(0.25f), tU, dV);
    Face F;
    F.f0 = txx;
    F.f1 = txy;
    F.f2 = fma2(txx, add2(Ua, Ub), fma2(txy, add2(Va, Vb), mul2(k2, sub2(Tb, Ta))));
    return F;
}
// y-face between rows a and b = a + 1: (t_xy, t_yy, 2 x (work + heat))
__device__ __forceinline__ Face face_y(float2 Ua, float2 Ub, float2 Va, float2 Vb, float2 tU, float2 tV, float2 Ta,
                                       float2 Tb, float2 k2) {
    const float2 dU = sub2(Ub, Ua), dV = sub2(Vb, Va);
    const float2 tyy = fma2(f2(4.f / 3.f), dV, mul2(f2(-1.f / 6.f), tU)), txy = fma2(f2(0.25f), tV, dU);
    Face F;
    F.f0 = txy;
    F.f1 = tyy;
    F.f2 = fma2(txy, add2(Ua, Ub), fma2(tyy, add2(Va, Vb), mul2(k2, sub2(Tb, Ta))));
    return F;
}

// Shared ring rows of the march: P pairs each (P >= T, a compile-time pitch, so
// that every access is a register and an immediate), thread t's pair at slot t.
// Three steps share a block of rows (slot i = j mod 3 within the block of step
// j), and the blocks of a ring are taken in turn:
//   u, v (v = 0, 1) of stage input k (k = 0 u0, 1 s1, 2 s2): two blocks of 18
//     rows, row 6k + 3v + i
//   rho u, E, p, T (f = 0..3) of stage input k: one block, row 12k + 3f + i
//     (read one step after they are published)
//   rho, rho u, rho v, E (q) of u0, own column only: three blocks of 12 rows,
//     row 3q + i, filled asynchronously three steps ahead and kept for five
constexpr int kMarchUV = 18, kMarchFlux = 2 * kMarchUV, kMarchU0 = kMarchFlux + 36, kMarchU0Block = 12;
constexpr int kMarchRows = kMarchU0 + 3 * kMarchU0Block;
constexpr int kMarchPitch[] = {32, 64, 96, 128, 192, 256};
constexpr size_t march_smem_bytes(int pitch) { return sizeof(float2) * kMarchRows * (size_t)pitch; }
constexpr int kMarchMaxThreads = 256;
constexpr int kMarchBandMax = kMarchMaxThreads - 6;  // output columns of a band
constexpr int kMarchNarrowBand = 122;  // output columns of a narrow band: 128 threads per CTA

// a thread's places in the ring rows: its own slot, the east and the west
// neighbour's (cyclic over the T columns)
struct Ring {
    float2 *own;
    const float2 *e, *w;
};

// Stage input K, evaluated in step j (I = j mod 3) at the centre row c of the
// window (m1, c, p1 published in steps j - 2, j - 1, j).  yf: in, the face
// between m1 and c (carried from the previous step); out, the face between c
// and p1.  FULL = false computes only that face (the step before a stage's
// first row).  cur / prev: this step's block of ring rows and the other one.
template <int P, int I, int K, bool FULL>
__device__ __forceinline__ void march_rhs(const Ring &cur, const Ring &prev, const Ring &one, const Rec &m1,
                                          const Rec &c, const Rec &p1, float inv_h, float inv_2h, float mu, float kap,
                                          Face &yf, float2 (&L)[4]) {
    // u (v = 0) and v (v = 1) of the east / west neighbour, d rows above p1
    auto east = [&](int v, int d) {
        return I >= d ? cur.e[(6 * K + 3 * v + I - d) * P] : prev.e[(6 * K + 3 * v + I - d + 3) * P];
    };
    auto west = [&](int v, int d) {
        return I >= d ? cur.w[(6 * K + 3 * v + I - d) * P] : prev.w[(6 * K + 3 * v + I - d + 3) * P];
    };
    const float2 k2 = f2(mu > 0.f ? 2.f * kap / mu : 0.f);
    const float2 Uec = east(0, 1), Uwc = west(0, 1), Vec = east(1, 1), Vwc = west(1, 1);
    const float2 Uep = east(0, 0), Uwp = west(0, 0), Vep = east(1, 0), Vwp = west(1, 0);
    // face between c and p1
    const Face top = face_y(c.U, p1.U, c.V, p1.V, add2(sub2(Uec, Uwc), sub2(Uep, Uwp)),
                            add2(sub2(Vec, Vwc), sub2(Vep, Vwp)), c.T, p1.T, k2);
    if (FULL) {
        const float2 Uem = east(0, 2), Uwm = west(0, 2), Vem = east(1, 2), Vwm = west(1, 2);
        constexpr int F = (kMarchFlux + 12 * K + (I + 2) % 3) * P, S = 3 * P;
        const float2 mxe = one.e[F], mxw = one.w[F], Ee = one.e[F + S], Ew = one.w[F + S];
        const float2 Pe = one.e[F + 2 * S], Pw = one.w[F + 2 * S], Te = one.e[F + 3 * S], Tw = one.w[F + 3 * S];
        // inviscid part: central differences of the nodal fluxes
        const float2 mi2h = f2(-inv_2h);
        const float2 myn = p1.my, mys = m1.my;
        const float2 Fe1 = fma2(mxe, Uec, Pe), Fw1 = fma2(mxw, Uwc, Pw);
        const float2 Fe2 = mul2(mxe, Vec), Fw2 = mul2(mxw, Vwc);
        const float2 Fe3 = mul2(add2(Ee, Pe), Uec), Fw3 = mul2(add2(Ew, Pw), Uwc);
        const float2 Gn1 = mul2(myn, p1.U), Gs1 = mul2(mys, m1.U);
        const float2 Gn2 = fma2(myn, p1.V, p1.P), Gs2 = fma2(mys, m1.V, m1.P);
        const float2 Gn3 = mul2(add2(p1.E, p1.P), p1.V), Gs3 = mul2(add2(m1.E, m1.P), m1.V);
        const float2 r0 = mul2(add2(sub2(mxe, mxw), sub2(myn, mys)), mi2h);
        const float2 r1 = mul2(add2(sub2(Fe1, Fw1), sub2(Gn1, Gs1)), mi2h);
        const float2 r2 = mul2(add2(sub2(Fe2, Fw2), sub2(Gn2, Gs2)), mi2h);
        const float2 r3 = mul2(add2(sub2(Fe3, Fw3), sub2(Gn3, Gs3)), mi2h);
        // x-faces of the centre row
        const Face fw = face_x(Uwc, c.U, Vwc, c.V, add2(sub2(Uwp, Uwm), sub2(p1.U, m1.U)),
                               add2(sub2(Vwp, Vwm), sub2(p1.V, m1.V)), Tw, c.T, k2);
        const Face fe = face_x(c.U, Uec, c.V, Vec, add2(sub2(p1.U, m1.U), sub2(Uep, Uem)),
                               add2(sub2(p1.V, m1.V), sub2(Vep, Vem)), c.T, Te, k2);
        const float2 mh2 = f2(mu * inv_h * inv_h), hmh2 = f2(0.5f * mu * inv_h * inv_h);
        L[0] = r0;
        L[1] = fma2(add2(sub2(fe.f0, fw.f0), sub2(top.f0, yf.f0)), mh2, r1);
        L[2] = fma2(add2(sub2(fe.f1, fw.f1), sub2(top.f1, yf.f1)), mh2, r2);
        L[3] = fma2(add2(sub2(fe.f2, fw.f2), sub2(top.f2, yf.f2)), hmh2, r3);
    }
    yf = top;
}

// row segment of one grid: half of a unit (columns from c0, which may be
// negative; rows from y0; columns t in [ilo, ihi) and `rows` rows are stored)
struct MarchHalf {
    const float *in;  // step-start state of the grid (4 planes)
    float *out;       // state after the step
    int c0, y0, rows, ilo, ihi;
};
// one unit of a march launch: two row segments of grids of one size
struct MarchUnit {
    MarchHalf h[2];
    int n, rows;  // points per side; rows of the longer half
    float inv_h, inv_2h, dt;
};

// bands and row segments of one n x n grid (host and device agree)
// bands of at most kMarchBandMax columns (the whole width up to 256), or
// with `narrow` of at most kMarchNarrowBand (the whole width up to 128)
__host__ __device__ __forceinline__ int march_bands(int n, bool narrow = false) {
    if (narrow) return n <= 128 ? 1 : (n + kMarchNarrowBand - 1) / kMarchNarrowBand;
    return n <= kMarchMaxThreads ? 1 : (n + kMarchBandMax - 1) / kMarchBandMax;
}
__host__ __device__ __forceinline__ int march_band_width(int n, int bands) { return (n + bands - 1) / bands; }
__host__ __device__ __forceinline__ int march_threads(int n, bool narrow = false) {
    const int b = march_bands(n, narrow);
    return b == 1 ? n : march_band_width(n, b) + 6;
}

// segment `id` of a group (grids, bands and row segments in that order)
__device__ __forceinline__ MarchHalf march_half(const NsGroup<float> &G, int id, int parity) {
    const int per_grid = G.tx * G.ty;
    const int prob = id / per_grid;
    const int rem = id - prob * per_grid;
    const int band = rem / G.ty, seg = rem - band * G.ty;
    const int n = G.n;
    const size_t off = (size_t)prob * 4 * n * n;
    float *u0 = G.u0 + off, *other = G.s1 + off;
    MarchHalf u;
    u.in = parity ? other : u0;
    u.out = parity ? u0 : other;
    const int S = (n + G.ty - 1) / G.ty;
    u.y0 = seg * S;
    u.rows = min(S, n - u.y0);
    if (G.tx == 1) {
        u.c0 = 0;
        u.ilo = 0;
        u.ihi = n;
    } else {
        const int bw = march_band_width(n, G.tx), bx0 = band * bw;
        u.c0 = bx0 - 3;
        u.ilo = 3;
        u.ihi = 3 + min(bw, n - bx0);
    }
    return u;
}

// unit `local` of a group: segments 2 local and 2 local + 1 (the last of an
// odd count goes alone: its partner repeats it and stores nothing)
__device__ __forceinline__ MarchUnit march_unit(const NsGroup<float> &G, int local, int parity) {
    const int count = G.nprob * G.tx * G.ty;
    MarchUnit u;
    u.h[0] = march_half(G, 2 * local, parity);
    u.h[1] = u.h[0];
    if (2 * local + 1 < count)
        u.h[1] = march_half(G, 2 * local + 1, parity);
    else
        u.h[1].rows = 0;
    u.n = G.n;
    u.rows = max(u.h[0].rows, u.h[1].rows);
    u.inv_h = G.inv_h;
    u.inv_2h = G.inv_2h;
    u.dt = G.dt;
    return u;
}

// where the units of a launch come from: a device table of groups of one grid
// size, or one group passed by value (groups == NULL)
struct MarchUnits {
    const NsGroup<float> *groups;
    int ngroups;
    NsGroup<float> one;
    __device__ __forceinline__ MarchUnit unit(int u, int parity) const {
        if (!groups) return march_unit(one, u, parity);
        int gi = 0;
        while (gi + 1 < ngroups && groups[gi + 1].tile_begin <= u) ++gi;
        const NsGroup<float> G = groups[gi];
        return march_unit(G, u - G.tile_begin, parity);
    }
    __device__ __forceinline__ NsGroup<float> group(int gi) const { return groups ? groups[gi] : one; }
};

template <int V>
using Int = std::integral_constant<int, V>;

// One SSP-RK3 step of one unit per CTA (blockDim.x = march_threads(n) of the
// launch's grid size).  Step j of the march: rows of u0 arrive in steps
// 0 .. rows + 5 (rows y0 - 3 .. y0 + rows + 2 of each half); stage 1 evaluates
// row y0 - 4 + j in steps 2 .. rows + 5, stage 2 row y0 - 6 + j in steps
// 5 .. rows + 6, stage 3 row y0 - 8 + j in steps 8 .. rows + 7; a stage's
// output row is published one step after it is computed.  The steps go in
// blocks of three, so that the rows of the register windows change their names
// instead of moving (one at a time, a quarter of the instructions were moves).
template <int P>
__global__ void __launch_bounds__(P, 1) ns2d_rk3_march(MarchUnits src, int parity, float gm1, float mu, float kap) {
    extern __shared__ float4 march_smem4[];
    float2 *X = reinterpret_cast<float2 *>(march_smem4);
    const int T = blockDim.x, t = threadIdx.x;
    const MarchUnit u = src.unit(blockIdx.x, parity);
    const int n = u.n, plane = n * n;  // 4 planes of one grid stay below 2^31 elements
    const int R = u.rows;
    const Ring one{X + t, X + (t + 1 == T ? 0 : t + 1), X + (t == 0 ? T - 1 : t - 1)};
    Ring cur = one, prev{one.own + kMarchUV * P, one.e + kMarchUV * P, one.w + kMarchUV * P};
    // u0's blocks: this step's, the previous and the next one (also the one before the previous)
    float2 *q0 = one.own + kMarchU0 * P, *qnext = q0 + kMarchU0Block * P, *qprev = qnext + kMarchU0Block * P;
    const int xa = wrap_index(u.h[0].c0 + t, n), xb = wrap_index(u.h[1].c0 + t, n);
    // elements of the next row to load and of the next row to store, per half
    int ia = wrap_index(u.h[0].y0 - 3, n) * n + xa, ib = wrap_index(u.h[1].y0 - 3, n) * n + xb;
    int oa = u.h[0].y0 * n + xa, ob = u.h[1].y0 * n + xb;
    // last step in which this thread stores
    const int enda = t >= u.h[0].ilo && t < u.h[0].ihi ? u.h[0].rows + 8 : 0;
    const int endb = t >= u.h[1].ilo && t < u.h[1].ihi ? u.h[1].rows + 8 : 0;
    // Steps follow one another with programmatic serialisation (march_launch):
    // each CTA has decoded its unit (static tables only); the previous launch has
    // completed and its writes are visible from here on, and only then may the
    // next one be placed: placed earlier, its CTAs take the SMs that drain first
    // and leave others idle (512^2 / 128^2 handle, 10 steps: 514 against 479 us).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // issue the copies of the next row of u0 into a row of a block
    auto load_row = [&](float2 *row) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            cp_async4(&row[3 * q * P].x, u.h[0].in + q * plane + ia);
            cp_async4(&row[3 * q * P].y, u.h[1].in + q * plane + ib);
        }
        ia += n;
        ib += n;
        if (ia >= plane) ia -= plane;
        if (ib >= plane) ib -= plane;
    };
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        load_row(q0 + i * P);
        cp_async_commit();
    }
    const float2 dt = f2(u.dt);
    // rows of u0, s1, s2 by their step (mod 3): A[j % 3] arrived in step j,
    // B[j % 3] and C[j % 3] were computed in it
    Rec A[3] = {}, B[3] = {}, C[3] = {};
    Face yf1{}, yf2{}, yf3{};  // carried faces

    // step j (I = j mod 3); STEADY: all stages run
    auto step = [&](auto I_, auto STEADY_, int j) {
        constexpr int I = decltype(I_)::value, I1 = (I + 1) % 3, I2 = (I + 2) % 3;
        constexpr bool STEADY = decltype(STEADY_)::value;
        auto publish = [&](auto K_, const Rec &r) {
            constexpr int K = decltype(K_)::value, F = (kMarchFlux + 12 * K + I) * P, S = 3 * P;
            cur.own[(6 * K + I) * P] = r.U;
            cur.own[(6 * K + 3 + I) * P] = r.V;
            one.own[F] = r.mx;
            one.own[F + S] = r.E;
            one.own[F + 2 * S] = r.P;
            one.own[F + 3 * S] = r.T;
        };
        // the rows that arrive in this step (a thread copies its own column)
        cp_async_wait<2>();
        if (STEADY || j <= R + 5) {
            const float2 *r = q0 + I * P;
            A[I] = make_rec(r[0], r[3 * P], r[6 * P], r[9 * P], gm1);
            publish(Int<0>{}, A[I]);
        }
        if (STEADY || (j >= 3 && j <= R + 6)) publish(Int<1>{}, B[I2]);
        if (STEADY || (j >= 6 && j <= R + 7)) publish(Int<2>{}, C[I2]);
        __syncthreads();
        if (STEADY || j + 3 <= R + 5) load_row(qnext + I * P);
        cp_async_commit();

        float2 L3[4], L2[4], L1[4];
        // in the steady state the three stages run without a branch between them:
        // their ILP hides the latency (one or two warps per scheduler)
        if constexpr (!STEADY && I == 1) {
            if (j == 7) march_rhs<P, I, 2, false>(cur, prev, one, C[I], C[I1], C[I2], u.inv_h, u.inv_2h, mu, kap, yf3, L3);
            if (j == 4) march_rhs<P, I, 1, false>(cur, prev, one, B[I], B[I1], B[I2], u.inv_h, u.inv_2h, mu, kap, yf2, L2);
            if (j == 1) march_rhs<P, I, 0, false>(cur, prev, one, A[I1], A[I2], A[I], u.inv_h, u.inv_2h, mu, kap, yf1, L1);
        }
        const bool run3 = STEADY || j >= 8, run2 = STEADY || (j >= 5 && j <= R + 6),
                   run1 = STEADY || (j >= 2 && j <= R + 5);
        if (run3) march_rhs<P, I, 2, true>(cur, prev, one, C[I], C[I1], C[I2], u.inv_h, u.inv_2h, mu, kap, yf3, L3);
        if (run3) {  // the new state's row y0 - 8 + j; u0's row arrived in step j - 5
            const float2 *R0 = I == 2 ? qprev : qnext + (I + 1) * P;
            const Rec &c = C[I1];
            const float2 q[4] = {c.rho, c.mx, c.my, c.E};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 base = R0[3 * k * P];
                const float2 res = fma2(f2(2.f / 3.f), fma2(dt, L3[k], sub2(q[k], base)), base);
                if (j < enda) u.h[0].out[k * plane + oa] = res.x;
                if (j < endb) u.h[1].out[k * plane + ob] = res.y;
            }
            oa += n;
            ob += n;
        }
        if (run2) march_rhs<P, I, 1, true>(cur, prev, one, B[I], B[I1], B[I2], u.inv_h, u.inv_2h, mu, kap, yf2, L2);
        if (run2) {  // row y0 - 6 + j of s2; u0's row arrived in step j - 3
            const float2 *R0 = qprev + I * P;
            const Rec &c = B[I1];
            const float2 q[4] = {c.rho, c.mx, c.my, c.E};
            float2 sv[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 base = R0[3 * k * P];
                sv[k] = fma2(f2(0.25f), fma2(dt, L2[k], sub2(q[k], base)), base);
            }
            C[I] = make_rec(sv[0], sv[1], sv[2], sv[3], gm1);
        }
        if (run1) march_rhs<P, I, 0, true>(cur, prev, one, A[I1], A[I2], A[I], u.inv_h, u.inv_2h, mu, kap, yf1, L1);
        if (run1) {  // row y0 - 4 + j of s1
            const Rec &c = A[I2];
            const float2 q[4] = {c.rho, c.mx, c.my, c.E};
            float2 sv[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) sv[k] = fma2(dt, L1[k], q[k]);
            B[I] = make_rec(sv[0], sv[1], sv[2], sv[3], gm1);
        }
    };
    using No = std::false_type;
    using Yes = std::true_type;
    for (int j = 0; j < R + 8; j += 3) {
        if (j >= 8 && j + 2 <= R + 5) {
            step(Int<0>{}, Yes{}, j);
            step(Int<1>{}, Yes{}, j + 1);
            step(Int<2>{}, Yes{}, j + 2);
        } else {
            step(Int<0>{}, No{}, j);
            if (j + 1 < R + 8) step(Int<1>{}, No{}, j + 1);
            if (j + 2 < R + 8) step(Int<2>{}, No{}, j + 2);
        }
        const Ring s = cur;
        cur = prev;
        prev = s;
        float2 *const q = qprev;
        qprev = q0;
        q0 = qnext;
        qnext = q;
    }
    cp_async_wait<0>();
}

// After an odd number of steps the states sit in the scratch buffers: copy
// them back (group blockIdx.y).
template <class Units>
__global__ void __launch_bounds__(256) ns2d_copy_back(Units src) {
    const NsGroup<float> G = src.group(blockIdx.y);
    const size_t count = (size_t)G.n * G.n * G.nprob;  // float4 per group: 4 n^2 nprob floats
    const float4 *s = reinterpret_cast<const float4 *>(G.s1);
    float4 *d = reinterpret_cast<float4 *>(G.u0);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
        d[i] = s[i];
}

// CTAs per launch of the persistent step kernel: resident CTAs per SM x SMs
// (per device: the attribute and the occupancy belong to a device context)
template <int TX, int H, int MINB, class Tiles>
static int step_grid(int total_tiles) {
    static OncePerDevice once;
    static int ctas[kMaxDevices];
    once.run([](int dev) {
        const size_t smem = StepSmem<TX, H>::bytes();
        int per_sm = 0, sms = 0;
        cudaError_t e = cudaFuncSetAttribute(ns2d_rk3_step<TX, H, MINB, Tiles>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ns2d_rk3_step<TX, H, MINB, Tiles>, 256, smem);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        ctas[dev] = std::max(per_sm, 1) * std::max(sms, 1);
        return e;
    });
    const int dev = OncePerDevice::current();
    const int c = dev >= 0 && ctas[dev] > 0 ? ctas[dev] : kNumSMs;
    return std::min(total_tiles, c);
}

template <int TX, int H, int MINB, class Tiles>
static void step_launch(const Tiles &src, int total_tiles, int parity, float gm1, float mu, float kap,
                        cudaStream_t s) {
    const int grid = step_grid<TX, H, MINB, Tiles>(total_tiles);
    // programmatic stream serialisation: the launch may start while the
    // previous kernel on the stream finishes; the kernel waits for it before
    // it touches the state (griddepcontrol.wait)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = StepSmem<TX, H>::bytes();
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, ns2d_rk3_step<TX, H, MINB, Tiles>, src, total_tiles, parity, gm1, mu, kap);
}

// nsteps steps of every tile (the states end in u0), FP32
template <int TX, int H, int MINB, class Tiles>
static void step_sequence(const Tiles &src, int ngroups, int total_tiles, int nsteps, float gm1, float mu,
                          float kap, cudaStream_t s) {
    for (int st = 0; st < nsteps; ++st) step_launch<TX, H, MINB>(src, total_tiles, st & 1, gm1, mu, kap, s);
    count_launches(nsteps);
    if (nsteps & 1) {
        ns2d_copy_back<Tiles><<<dim3(2 * kNumSMs, ngroups), 256, 0, s>>>(src);
        count_launches(1);
    }
}

template <int I>
static void march_launch(const MarchUnits &src, int units, int threads, int parity, float gm1, float mu, float kap,
                         cudaStream_t s) {
    constexpr int P = kMarchPitch[I];
    if constexpr (I + 1 < (int)(sizeof(kMarchPitch) / sizeof(kMarchPitch[0])))
        if (threads > P) return march_launch<I + 1>(src, units, threads, parity, gm1, mu, kap, s);
    static OncePerDevice once;
    once.run([](int) {
        return cudaFuncSetAttribute(ns2d_rk3_march<P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)march_smem_bytes(P));
    });
    // programmatic stream serialisation: the launch may start while the
    // previous kernel on the stream finishes; the kernel waits for it before
    // it touches the state (griddepcontrol.wait)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(units);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = march_smem_bytes(P);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, ns2d_rk3_march<P>, src, parity, gm1, mu, kap);
}

// nsteps steps of every unit (the states end in u0), FP32
static void march_sequence(const MarchUnits &src, int ngroups, int units, int threads, int nsteps, float gm1, float mu,
                           float kap, cudaStream_t s) {
    for (int st = 0; st < nsteps; ++st) march_launch<0>(src, units, threads, st & 1, gm1, mu, kap, s);
    count_launches(nsteps);
    if (nsteps & 1) {
        ns2d_copy_back<MarchUnits><<<dim3(2 * kNumSMs, ngroups), 256, 0, s>>>(src);
        count_launches(1);
    }
}

// rows per segment of the march for a choice (the batch's tuned "shape":
// shape mod kNsSegChoices the segment rows, shape / kNsSegChoices = 1 narrow
// bands)
int ns2d_seg_rows(int shape) {
    constexpr int rows[kNsSegChoices] = {32, 16, 64, 128, 256, 24, 48, 20};
    return rows[shape % kNsSegChoices];
}
bool ns2d_narrow(int shape) { return shape / kNsSegChoices == 1; }

void ns2d_march_layout(int n, int shape, int *bands, int *segs, int *threads) {
    const int S = std::min(n, ns2d_seg_rows(shape));
    const bool narrow = ns2d_narrow(shape);
    *bands = march_bands(n, narrow);
    *segs = (n + S - 1) / S;
    *threads = march_threads(n, narrow);
}

// Estimated time of a model step of all sizes at once, in march steps at two
// warps per scheduler.  A march step's time is its latency: about 0.65 us with
// one warp per scheduler and 1.05 us with two, which is all that the registers
// of an SM hold (248 a thread).  While every CTA of the launches is resident
// the longest march decides; beyond that the work does, plus a tenth of the
// longest march (and a little of each) for the ends of the launches.  CTAs of
// more than four warps have an SM to themselves: they lose a tenth at their
// barriers, and half with more than two sizes at once (two: the members and the
// fine run of one handle, or problems alike), as an SM whose large CTA has ended
// is then taken by small CTAs of other sizes before it is empty again.  (24
// problems of 64^2 .. 768^2, one choice for all: the estimates for 32, 48, 64,
// 128 and 256 rows, wide and narrow, are proportional to the measured 6.2 ..
// 7.9 ms within 5%; with the defaults 6.2 ms.)
static double march_estimate(int count, const int *n, const int *grids, const int *choice, int sms) {
    double load = 0, work = 0;
    int longest = 0, all = 0;
    bool large = false;
    for (int k = 0; k < count; ++k) {
        int bands = 0, segs = 0, threads = 0;
        ns2d_march_layout(n[k], choice[k], &bands, &segs, &threads);
        const int warps = (threads + 31) / 32, per_sm = std::max(1, 8 / warps);
        const double share = (((long long)bands * segs * grids[k] + 1) / 2) / ((double)per_sm * sms);
        const int steps = (n[k] + segs - 1) / segs + 8;
        load += share;
        all += steps;
        work += share * steps * (warps > 4 ? (count > 2 ? 1.5 : 1.1) : 1.0);
        if (steps > longest || (steps == longest && warps > 4)) large = warps > 4;
        longest = std::max(longest, steps);
    }
    if (load <= 1) return longest * (load <= 0.5 && !large ? 0.63 : 1.0);
    return std::max(work, (double)longest) + 0.1 * longest + 0.003 * all;
}

void ns2d_default_choices(int count, const int *n, const int *grids, int sms, int *choice) {
    std::vector<int> c(count);
    double best = 0;
    const int starts = count > 1 ? kNsSegChoices : 1;  // one size alone: every choice is tried in the first pass
    for (int rows = 0; rows < starts; ++rows) {
        // from segments of these rows everywhere, one size at a time until no
        // change of one choice helps
        for (int k = 0; k < count; ++k) c[k] = n[k] > 128 ? kNsSegChoices + rows : rows;
        double now = march_estimate(count, n, grids, c.data(), sms);
        bool better = true;
        for (int pass = 0; pass < (count > 1 ? 4 : 1) && better; ++pass) {
            better = false;
            for (int k = 0; k < count; ++k)
                for (int q = 0; q < kNsTileShapes; ++q) {
                    const int was = c[k];
                    c[k] = q;
                    const double t = march_estimate(count, n, grids, c.data(), sms);
                    if (t < now * (1 - 1e-9)) {
                        now = t;
                        better = true;
                    } else {
                        c[k] = was;
                    }
                }
        }
        if (rows == 0 || now < best * (1 - 1e-9)) {
            best = now;
            std::copy(c.begin(), c.end(), choice);
        }
    }
}

// strips of an n x n grid in the FP64 march, and the CTAs of `grids` grids cut
// into runs of `rows` rows
static int n64_strips(int n) { return ceil_div(n, kN64Threads); }
static long long n64_ctas(int n, int grids, int rows) {
    const int pitch = ceil_div(ceil_div(n, n64_strips(n)), 32) * 32, upc = kN64Threads / pitch;
    return ((long long)grids * n64_strips(n) * ceil_div(n, rows) + upc - 1) / upc;
}

template <int STAGE>
static cudaError_t n64_launch(const Ns64Args &A, long long ctas, int per_sm, cudaStream_t s) {
    static OncePerDevice once;
    once.run([](int) {
        return cudaFuncSetAttribute(ns2d_march64<STAGE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 120 * 1024);
    });
    count_launches(1);
    return launch_kernel(ns2d_march64<STAGE>, (unsigned)ctas, kN64Threads,
                         residency_smem(sizeof(double) * n64_smem_doubles(A.rows), per_sm), s, LaunchHow{}, A);
}

static cudaError_t n64_forecast(const NsGroup<double> (&g)[2], double gm1, double mu, double kappa, int nsteps,
                                cudaStream_t s) {
    Ns64Args A = {};
    static OncePerDevice once;
    static int sm_count[kMaxDevices];
    once.run([](int dev) { return cudaDeviceGetAttribute(&sm_count[dev], cudaDevAttrMultiProcessorCount, dev); });
    const int dev = OncePerDevice::current(), sms = dev >= 0 && sm_count[dev] > 0 ? sm_count[dev] : kNumSMs;
    auto ctas = [&](int rows) {
        long long c = 0;
        for (int k = 0; k < 2; ++k)
            if (g[k].nprob > 0) c += n64_ctas(g[k].n, g[k].nprob, rows);
        return c;
    };
    // rows per unit and CTAs per SM at once: the FP64 instructions of a CTA (80
    // per row, about 60 for the two extra rows) times the CTAs an SM runs; one,
    // two, three CTAs at a time leave 20%, 10%, 2% of the pipe idle at barriers
    // and loads (512^2: 1.62 ms with 14 rows, 1.56 with two of 7, 1.61 with three
    // of 5; 64^2 x 32 and 256^2: 1.31 with 11 rows, 1.37, 1.33)
    double best = 1e300;
    int per_sm = 1;
    const int nmax = std::max(g[0].nprob > 0 ? g[0].n : 0, g[1].nprob > 0 ? g[1].n : 0);
    for (int rows = 2; rows <= std::min(nmax, 64); ++rows) {
        const long long c = ctas(rows);
        for (int r = 1; r <= 3; ++r) {
            const double idle[3] = {1.2, 1.1, 1.02};
            const double t = (double)((c + (long long)sms * r - 1) / ((long long)sms * r)) * r * idle[r - 1] *
                             (80.0 * rows + 60.0);
            if (t < best) {
                best = t;
                A.rows = rows;
                per_sm = r;
            }
        }
    }
    for (int k = 0; k < 2; ++k) {
        A.g[k] = g[k];
        if (g[k].nprob <= 0) continue;
        A.g[k].tx = n64_strips(g[k].n);
        A.g[k].ty = ceil_div(g[k].n, A.rows);
        A.c1[k] = -g[k].dt * g[k].inv_2h;
        A.c2[k] = g[k].dt * mu * g[k].inv_h * g[k].inv_h;
    }
    A.gm1 = gm1;
    A.k2 = mu > 0.0 ? 2.0 * kappa / mu : 0.0;
    A.ctas0 = g[0].nprob > 0 ? (int)n64_ctas(g[0].n, g[0].nprob, A.rows) : 0;
    const long long total = ctas(A.rows);
    if (total > INT32_MAX) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaSuccess;
    for (int st = 0; st < nsteps && e == cudaSuccess; ++st) {
        e = n64_launch<0>(A, total, per_sm, s);
        if (e == cudaSuccess) e = n64_launch<1>(A, total, per_sm, s);
        if (e == cudaSuccess) e = n64_launch<2>(A, total, per_sm, s);
    }
    return e;
}

const char *ns2d_check_size(int n_whole, int n_split) {
    for (int n : {n_whole, n_split}) {
        if (n < 8 || n > 4096 || n % 8 != 0) return "NS-2D grids need 8 <= n <= 4096 points per side with n % 8 == 0";
    }
    return nullptr;
}

size_t ns2d_scratch_elems(int n_whole, int n_whole_probs, int n_split, int n_split_probs) {
    return 2 * 4 * ((size_t)n_whole * n_whole * n_whole_probs + (size_t)n_split * n_split * n_split_probs);
}

template <typename T>
cudaError_t ns2d_forecast_scratch(T *whole, int n_whole, int n_whole_probs, T *split, int n_split,
                                  int n_split_probs, double length, double dt, double mu,
                                  double gamma, double prandtl, int nsteps, T *scratch,
                                  cudaStream_t stream) {
    NsGroup<T> gr[2] = {};
    const int ns[2] = {n_whole, n_split}, np[2] = {n_whole_probs, n_split_probs};
    T *st[2] = {whole, split};
    T *sc = scratch;
    int tiles[2] = {0, 0};
    for (int g = 0; g < 2; ++g) {
        NsGroup<T> &G = gr[g];
        G.n = ns[g];
        G.nprob = np[g];
        G.u0 = st[g];
        const size_t sz = (size_t)4 * ns[g] * ns[g] * np[g];
        G.s1 = sc;
        G.s2 = sc + sz;
        sc += 2 * sz;
        if (np[g] > 0) {
            G.tx = ceil_div(ns[g], kNsTx);
            G.ty = ceil_div(ns[g], kNsTileRows);
            const double h = length / ns[g];
            G.inv_h = (T)(1.0 / h);
            G.inv_2h = (T)(1.0 / (2.0 * h));
            G.dt = (T)dt;
            tiles[g] = G.tx * G.ty * np[g];
        }
    }
    const T gm1 = (T)(gamma - 1.0), m = (T)mu, kappa = (T)(mu * gamma / ((gamma - 1.0) * prandtl));
    const int grid = tiles[0] + tiles[1];
    if (grid == 0 || nsteps == 0) return cudaSuccess;
    if constexpr (std::is_same<T, float>::value) {
        // the copy back moves float4
        if ((reinterpret_cast<uintptr_t>(whole) | reinterpret_cast<uintptr_t>(split) |
             reinterpret_cast<uintptr_t>(scratch)) & 15)
            return cudaErrorMisalignedAddress;
        if (n_split_probs > 0) {
            // a handle (members and fine run): both groups in one persistent
            // launch of the tile kernel per step
            PairTiles P{{gr[0], gr[1]}};
            P.g[0].tile_begin = 0;
            P.g[1].tile_begin = tiles[0];
            step_sequence<32, 16, 2>(P, 2, grid, nsteps, gm1, m, kappa, stream);
        } else {
            // grids of one size (truth runs, the stateless entry point): the
            // column march
            MarchUnits U{nullptr, 1, gr[0]};
            int bands = 0, segs = 0, threads = 0;
            int choice = 0;
            ns2d_default_choices(1, ns, np, kNumSMs, &choice);
            ns2d_march_layout(ns[0], choice, &bands, &segs, &threads);
            U.one.tx = bands;
            U.one.ty = segs;
            U.one.tile_begin = 0;
            march_sequence(U, 1, ns2d_group_units(U.one), threads, nsteps, gm1, m, kappa, stream);
        }
    } else {
        const cudaError_t e = n64_forecast(gr, gm1, m, kappa, nsteps, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t ns2d_forecast(T *whole, int n_whole, int n_whole_probs, T *split, int n_split,
                          int n_split_probs, double length, double dt, double mu, double gamma,
                          double prandtl, int nsteps, cudaStream_t stream) {
    // stream-ordered scratch for the stateless entry point
    const size_t elems = ns2d_scratch_elems(n_whole, n_whole_probs, n_split, n_split_probs);
    if (elems == 0 || nsteps == 0) return cudaSuccess;
    T *scratch = nullptr;
    cudaError_t e = cudaMallocAsync((void **)&scratch, elems * sizeof(T), stream);
    if (e != cudaSuccess) return e;
    e = ns2d_forecast_scratch<T>(whole, n_whole, n_whole_probs, split, n_split, n_split_probs, length, dt,
                                 mu, gamma, prandtl, nsteps, scratch, stream);
    cudaError_t e2 = cudaFreeAsync(scratch, stream);
    return e != cudaSuccess ? e : e2;
}

static cudaError_t table_steps(const NsGroup<float> *d_groups, int ngroups, int units, int n, int nsteps,
                               bool probe, double gamma, double mu, double prandtl, int shape, cudaStream_t s) {
    if (units == 0 || nsteps == 0) return cudaSuccess;
    const float gm1 = (float)(gamma - 1.0), m = (float)mu, kap = (float)(mu * gamma / ((gamma - 1.0) * prandtl));
    const MarchUnits src{d_groups, ngroups, {}};
    const int threads = march_threads(n, ns2d_narrow(shape));
    if (probe) {  // one step into the scratch buffers: the states stay as they are
        march_launch<0>(src, units, threads, 0, gm1, m, kap, s);
        count_launches(1);
    } else {
        march_sequence(src, ngroups, units, threads, nsteps, gm1, m, kap, s);
    }
    return cudaGetLastError();
}

cudaError_t ns2d_forecast_table(const NsGroup<float> *d_groups, int ngroups, int units, int n, int nsteps,
                                double gamma, double mu, double prandtl, int shape, cudaStream_t s) {
    return table_steps(d_groups, ngroups, units, n, nsteps, false, gamma, mu, prandtl, shape, s);
}

cudaError_t ns2d_probe_step(const NsGroup<float> *d_groups, int ngroups, int units, int n, double gamma,
                            double mu, double prandtl, int shape, cudaStream_t s) {
    return table_steps(d_groups, ngroups, units, n, 1, true, gamma, mu, prandtl, shape, s);
}

#define MGK_NS_INST(T)                                                                            \
    template cudaError_t ns2d_forecast<T>(T *, int, int, T *, int, int, double, double, double,    \
                                          double, double, int, cudaStream_t);                     \
    template cudaError_t ns2d_forecast_scratch<T>(T *, int, int, T *, int, int, double, double,    \
                                                  double, double, double, int, T *, cudaStream_t);

MGK_NS_INST(float)
MGK_NS_INST(double)
#undef MGK_NS_INST

}  // namespace mgk
