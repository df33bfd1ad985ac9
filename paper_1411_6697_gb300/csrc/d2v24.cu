// d2v24.cu -- the paper's own 24-velocity model (D2V24, Sec. II Eqs. (25)-(27)):
// kernels and the C ABI of include/lbkm24.h.
//
// The step is one fused kernel per time step, one thread per cell, in tiles (step_kernel):
// the 25 planes of a tile and its two-cell halo are staged in shared memory by asynchronous
// copies; rho, u, T of the tile's cells and u of its rim are formed in FP64 (an FP32 state sums
// its conserved moments as exact double-floats on the FP32 pipes first); the 20 non-conserved
// moments less their equilibrium, the relaxation, the back-transform, the chemical term of
// Eq. (24) and the NND update run in the storage type R (FP64 or FP32); the TNE statistics of
// the state being read gather per warp (sums in FP64 or as exact FP32 pairs, extremes exactly),
// and an 82-block kernel turns them into one history record.
//
// What bounds it. FP32: instruction issue (60 % of the slots; about 3500 instructions per warp
// and step, half of them the exact sums of the recovery). FP64: the FP64 unit (cellops.cuh);
// 720 of its instructions per warp and 1-D step, 240 more where a cell of the warp reacts.
// Measured per step, against one thread per cell reading its stencil through the cache, every
// sum normalised, the reaction in FP64 divisions and exponentials throughout: 2048^2 FP32 1.95
// -> 0.67 ms, the 5000-cell detonation FP64 54 -> 37 us, FP32 12.6 -> 6.6 us.
//
// M and M^-1 act in block form: butterflies inside each orbit of four velocities
// (axis: f1+f3, f2+f4, f1-f3, f2-f4; diagonal: the sum and the three sign patterns)
// split the 24 components by parity in (v_x, v_y), and the moments of each parity
// sector depend on that sector's components only. The sectors are 9 (even, even:
// m1 m4 m5 m7 m14 m16 m17 m19 m20), 6 (odd, even: m2 m8 m10 m12 m21 m23), 6 (even,
// odd: m3 m9 m11 m13 m22 m24) and 3 (odd, odd: m6 m15 m18), so one transform costs
// 162 multiply-adds instead of 576. The blocks and their inverses are built on the
// host from M itself (checking that everything outside the blocks vanishes) and
// reach the kernel as kernel-parameter (constant-bank) operands.
#include <cuda_runtime.h>
#include <float.h>
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <string>
#include <vector>

#include "cellops.cuh"
#include "kernels.cuh"
#include "lbkm24.h"

namespace v24 {

using lbk::DevCounters;
using lbk::ad;
using lbk::dbits;
using lbk::f2d_exact;
using lbk::fm;
using lbk::map_index;
using lbk::mu;
using lbk::reaction_increment;
using lbk::sub;

constexpr int NV = 24;
constexpr int NP = NV + 1;       // planes: f_1..f_24, lambda
constexpr int TK = NV - 4;       // non-conserved moments Delta_5..Delta_24
constexpr int NQ = 4 * TK + 2;   // TNE quantities: sum, |sum|, min, max of each, d, d^2
constexpr int BT = 128;          // threads per block of tne_kernel: 128 x 1 or 32 x 1 (1-D), 32 x 4
constexpr int GRAPH_CHUNK = 32;  // even: a replay leaves the ping-pong index unchanged

// signs of v_x, v_y of velocity i = 8 g + 4 o + j (speed group g, o = 0 axis orbit with
// (1,0) (0,1) (-1,0) (0,-1), o = 1 diagonal orbit with (1,1) (-1,1) (-1,-1) (1,-1)); the
// speeds are positive, so the upwind side of every plane is fixed at compile time
__host__ __device__ constexpr int vsign_x(int i)
{
    return ((i >> 2) & 1) == 0 ? ((i & 3) == 0 ? 1 : ((i & 3) == 2 ? -1 : 0))
                               : (((i & 3) == 0 || (i & 3) == 3) ? 1 : -1);
}
__host__ __device__ constexpr int vsign_y(int i)
{
    return ((i >> 2) & 1) == 0 ? ((i & 3) == 1 ? 1 : ((i & 3) == 3 ? -1 : 0)) : ((i & 3) < 2 ? 1 : -1);
}

// parity sectors: sizes, offsets of their blocks, and the moment (0-based) at each
// sector-ordered position p = 0..23 (ee 0..8, oe 9..14, eo 15..20, oo 21..23)
constexpr int NSEC = 4;
constexpr int NB = 162; // 81 + 36 + 36 + 9 block entries
__host__ __device__ constexpr int sec_n(int s) { return s == 0 ? 9 : (s == 3 ? 3 : 6); }
__host__ __device__ constexpr int sec_p(int s) { return s == 0 ? 0 : (s == 1 ? 9 : (s == 2 ? 15 : 21)); }
__host__ __device__ constexpr int sec_b(int s) { return s == 0 ? 0 : (s == 1 ? 81 : (s == 2 ? 117 : 153)); }
__host__ __device__ constexpr int mom_of(int p)
{
    constexpr int t[NV] = {0, 3, 4, 6, 13, 15, 16, 18, 19, 1, 7, 9, 11, 20, 22,
                           2, 8, 10, 12, 21, 23, 5, 14, 17};
    return t[p];
}

struct Record {
    double sum[NV], abs_sum[NV], min[NV], max[NV];
    double d_sum, d2_sum;
    int64_t step;
};
static_assert(sizeof(Record) == sizeof(lbkm24_tne_global), "record layout");

// Model constants, passed by value (constant bank). M is row-major [k][i]
// (moment k of velocity i), Minv row-major [i][k].
template <typename R>
struct Model {
    R Bf[NB];  // forward blocks, row-major [moment][component] per sector
    R Bi[NB];  // their inverses, row-major [component][moment]
    R Bis[NB]; // the inverses with the butterfly scales (1/2 axis, 1/4 diagonal orbits) folded in
    R vx[NV], vy[NV], eta2[NV], S[NV];
    R vxs[NV], vys[NV];              // v_x / dx and v_y / dy in R
    R dt_r, inv_dx_r, inv_dy_r, hdx_r, hdy_r, I_r, DI_r, inv_DI_r, A8c_r, A9c_r; // constants in R
    R c_r[6], chem_o[6];             // of each orbit: its speed, I v^2 + eta^2
    double kchem;                    // Q / (dt I (D + I))
    int32_t sides[4];                // condition of each side: 0 periodic, 1 zero gradient, 2
                                     // wall, 3 Dirichlet, 4 specular
    double vxd[NV], vyd[NV], wd[NV]; // FP64 copies for the conserved sums
    double cd[6], wod[6];            // speed and v^2 + eta^2 of each orbit (FP64)
    float cdh[6], cdl[6], wdh[6], wdl[6]; // the same split into hi + lo FP32 pairs
    double Minvd[NV * NV];           // FP64 M^-1 for the equilibrium start
    double I, DI, inv_DI, Q, omega1, omega2, T_ig, A8c, A9c;
    double dt, inv_dx, inv_dy;
    int nx, ny, pitch, bc_x, bc_y, pad_;
    int64_t plane;
    // Dirichlet sides: ghost cells hold the equilibrium f of the side's state and its lambda
    R sfeq[4][NP];
    // walls (code 2, y sides) by non-equilibrium extrapolation: the ghost rows take the
    // edge row's f plus wall[side][i][x] = [M^-1 (f_hat^eq(rho, u_w, T_w) -
    // f_hat^eq(rho, u, T))]_i, rho, u, T of the edge cell, refreshed before every step
    const R* wall;
    double wux[2], wuy[2], wT[2];
};

struct Args {
    const void* in;
    void* out;
    double* partials;  // [NQ][grid blocks]
    DevCounters* ctr;
    Record* hist;
    int hist_cap;
    int tne_every;
    double area;       // dx * dy
};

__device__ __forceinline__ double tcomb(int kind, double a, double b)
{
    return kind == 0 ? a + b : (kind == 1 ? fmin(a, b) : fmax(a, b));
}
// quantity q: [0, TK) sum, [TK, 2TK) |.| sum, [2TK, 3TK) min, [3TK, 4TK) max, 4TK d, 4TK+1 d^2
__host__ __device__ __forceinline__ int tkind(int q)
{
    return (q < 2 * TK || q >= 4 * TK) ? 0 : (q < 3 * TK ? 1 : 2);
}

// FP64 -> R: exact (double) or rounded to nearest on the integer pipe (float)
template <typename R>
__device__ __forceinline__ R to_r(double x);
template <>
__device__ __forceinline__ double to_r<double>(double x) { return x; }
template <>
__device__ __forceinline__ float to_r<float>(double x) { return lbk::d2f_rn(x); }

// the same for values known to be finite, branch-free
template <typename R>
__device__ __forceinline__ R to_fast(double x);
template <>
__device__ __forceinline__ double to_fast<double>(double x) { return x; }
template <>
__device__ __forceinline__ float to_fast<float>(double x) { return lbk::d2f_fast(x); }

__device__ __forceinline__ double to_f64(double x) { return x; }
// exact, on the integer pipe (the FP64 unit runs at 1/58 of the FP32 rate on GB300)
__device__ __forceinline__ double to_f64(float x) { return f2d_exact(x); }

// plane of the velocity with v_y reversed (axis orbits (c,0) (0,c) (-c,0) (0,-c);
// diagonal orbits (+,+) (-,+) (-,-) (+,-)); lambda maps to itself
__host__ __device__ __forceinline__ int mirror24(int i)
{
    if (i >= NV) return i;
    const int o = i / 4, j = i % 4;
    const int jm = (o & 1) ? 3 - j : (j == 1 ? 3 : (j == 3 ? 1 : j));
    return 4 * o + jm;
}

// rho, u_x, u_y and, if asked, T (FP64) at cell (x, y) of state `in`, boundary conditions
// applied (Eqs. (5)-(7)). The sums go orbit by orbit: an orbit of speed c adds its sum s
// to rho, c times its x and y differences to rho u, and (c^2 or 2 c^2) + eta^2 times s to
// the energy moment m_4; 1/rho comes from an FP32 seed and two Newton steps.
template <typename R>
__device__ __forceinline__ void conserved_at(const Model<R>& K, const R* __restrict__ in, int x,
                                             int y, double& rho, double& ux, double& uy,
                                             double* T = nullptr)
{
    x = map_index(x, K.nx, K.bc_x == 0 ? 0 : 1);
    y = map_index(y, K.ny, K.bc_y == 0 ? 0 : 1);
    const R* p = in + (size_t)y * K.pitch + x;
    auto ld = [&](int i) -> R { return __ldg(p + (size_t)i * K.plane); };
    double r = 0.0, jx = 0.0, jy = 0.0, e = 0.0;
    if constexpr (sizeof(R) == 4) {
        // FP32 state: the same sums as double-floats on the FP32 pipes (error-free
        // TwoSum butterflies, products with split constants, ~48 significant bits),
        // carried into FP64 once
        using lbk::df;
        df R0{0.f, 0.f}, R1{0.f, 0.f}, R2{0.f, 0.f}, R3{0.f, 0.f};
#pragma unroll
        for (int o = 0; o < 6; o++) {
            const float a = ld(4 * o), b = ld(4 * o + 1), c = ld(4 * o + 2), d = ld(4 * o + 3);
            const df sac = lbk::two_sum(a, c), sbd = lbk::two_sum(b, d);
            const df dac = lbk::two_sum(a, -c), dbd = lbk::two_sum(b, -d);
            const df sum = lbk::df_add(sac, sbd);
            df gx = dac, gy = dbd;
            if (o & 1) {
                gx = lbk::df_sub(dac, dbd);
                gy = lbk::df_add(dac, dbd);
            }
            const df co{K.cdh[o], K.cdl[o]};
            R0 = lbk::df_add(R0, sum);
            R1 = lbk::df_add(R1, lbk::df_mul(co, gx));
            R2 = lbk::df_add(R2, lbk::df_mul(co, gy));
            if (T) R3 = lbk::df_add(R3, lbk::df_mul(df{K.wdh[o], K.wdl[o]}, sum));
        }
        r = f2d_exact(R0.hi) + f2d_exact(R0.lo);
        jx = f2d_exact(R1.hi) + f2d_exact(R1.lo);
        jy = f2d_exact(R2.hi) + f2d_exact(R2.lo);
        if (T) e = f2d_exact(R3.hi) + f2d_exact(R3.lo);
    } else {
#pragma unroll
    for (int o = 0; o < 6; o++) {
        const double a = to_f64(ld(4 * o)), b = to_f64(ld(4 * o + 1));
        const double c = to_f64(ld(4 * o + 2)), d = to_f64(ld(4 * o + 3));
        const double sac = a + c, sbd = b + d, dac = a - c, dbd = b - d;
        const double sum = sac + sbd;
        double gx, gy;
        if ((o & 1) == 0) { // axis: (1,0) (0,1) (-1,0) (0,-1)
            gx = dac;
            gy = dbd;
        } else {            // diagonal: (1,1) (-1,1) (-1,-1) (1,-1)
            gx = dac - dbd;
            gy = dac + dbd;
        }
        r += sum;
        jx = fma(K.cd[o], gx, jx);
        jy = fma(K.cd[o], gy, jy);
        if (T) e = fma(K.wod[o], sum, e);
    }
    }
    double q = f2d_exact(lbk::rcp_approx(lbk::d2f_rn(r)));
    q = fma(q, fma(-r, q, 1.0), q);
    q = fma(q, fma(-r, q, 1.0), q);
    rho = r;
    ux = jx * q;
    uy = jy * q;
    if (T) *T = (e * q - (ux * ux + uy * uy)) * K.inv_DI;
}

// orbit butterflies: f (velocity order) -> g (sector order)
template <typename R>
__host__ __device__ __forceinline__ void butterfly(const R* f, R* g)
{
#pragma unroll
    for (int o = 0; o < 6; o++) {
        const R a = f[4 * o], b = f[4 * o + 1], c = f[4 * o + 2], d = f[4 * o + 3];
        const int e0 = (o / 2) * 3;
        if ((o & 1) == 0) { // axis orbit: (1,0) (0,1) (-1,0) (0,-1)
            g[e0] = a + c;
            g[e0 + 1] = b + d;
            g[9 + o] = a - c;
            g[15 + o] = b - d;
        } else {            // diagonal orbit: (1,1) (-1,1) (-1,-1) (1,-1)
            g[e0 + 2] = (a + c) + (b + d);
            g[9 + o] = (a - c) - (b - d);
            g[15 + o] = (a - c) + (b - d);
            g[21 + o / 2] = (a + c) - (b + d);
        }
    }
}

// inverse butterflies: g (sector order) -> f (velocity order)
template <typename R>
__host__ __device__ __forceinline__ void unbutterfly(const R* g, R* f)
{
#pragma unroll
    for (int o = 0; o < 6; o++) {
        const int e0 = (o / 2) * 3;
        if ((o & 1) == 0) {
            const R sx = g[e0], sy = g[e0 + 1], ax = g[9 + o], ay = g[15 + o];
            f[4 * o] = R(0.5) * (sx + ax);
            f[4 * o + 1] = R(0.5) * (sy + ay);
            f[4 * o + 2] = R(0.5) * (sx - ax);
            f[4 * o + 3] = R(0.5) * (sy - ay);
        } else {
            const R e = g[e0 + 2], ax = g[9 + o], ay = g[15 + o], od = g[21 + o / 2];
            f[4 * o] = R(0.25) * ((e + od) + (ax + ay));
            f[4 * o + 1] = R(0.25) * ((e - od) - (ax - ay));
            f[4 * o + 2] = R(0.25) * ((e + od) - (ax + ay));
            f[4 * o + 3] = R(0.25) * ((e - od) + (ax - ay));
        }
    }
}

// y = blockdiag(B) x over the four sectors (x, y in sector order)
template <typename R>
__device__ __forceinline__ void block_apply(const R* B, const R* x, R* y)
{
#pragma unroll
    for (int sct = 0; sct < NSEC; sct++) {
        const int n = sec_n(sct), p0 = sec_p(sct), b0 = sec_b(sct);
#pragma unroll
        for (int r = 0; r < n; r++) {
            R acc = R(0);
#pragma unroll
            for (int j = 0; j < n; j++) acc = fma(B[b0 + r * n + j], x[p0 + j], acc);
            y[p0 + r] = acc;
        }
    }
}

// f_hat^eq_1..24 (list after Eq. (16); entries 14 and 16 with the factor T of Eq. (11)),
// in the arithmetic type F
template <typename F>
__host__ __device__ __forceinline__ void feq24(F I, F DI, F rho, F ux, F uy, F T, F* q)
{
    const F u2 = ux * ux + uy * uy;
    const F A = (DI + F(2)) * T + u2, B = (DI + F(4)) * T + u2;
    const F rx = rho * ux, ry = rho * uy, IT = I * T;
    const F C = u2 * u2 + F(4) * (DI + F(4)) * T * T + (DI + F(10)) * u2 * T; // D = 2
    q[0] = rho;
    q[1] = rx;
    q[2] = ry;
    q[3] = rho * (DI * T + u2);
    q[4] = rho * (T + ux * ux);
    q[5] = rx * uy;
    q[6] = rho * (T + uy * uy);
    q[7] = rx * A;
    q[8] = ry * A;
    q[9] = rx * (F(3) * T + ux * ux);
    q[10] = ry * (T + ux * ux);
    q[11] = rx * (T + uy * uy);
    q[12] = ry * (F(3) * T + uy * uy);
    q[13] = rho * A * T + rx * ux * B;
    q[14] = rx * uy * B;
    q[15] = rho * A * T + ry * uy * B;
    q[16] = rho * IT * (T + ux * ux);
    q[17] = rx * uy * IT;
    q[18] = rho * IT * (T + uy * uy);
    q[19] = rho * IT * (u2 + (F(2) + F(3) * I) * T);
    q[20] = rx * C;
    q[21] = ry * C;
    q[22] = rx * IT * (u2 + (F(4) + F(3) * I) * T);
    q[23] = ry * IT * (u2 + (F(4) + F(3) * I) * T);
}

// Block reduction of the TNE quantities of the block's cells into partials
// [q * nblocks + b], q in the record's order (sums of Delta_k, of |Delta_k|, minima,
// maxima, sum of d, sum of d^2). Each thread leaves its cell's Delta_5..24, d and d^2
// (formed in R) in shared memory; each quantity is then reduced in three parts of a
// third of the block's cells (one thread per part; the block's threads take the parts
// in turn), in a fixed order: the 42 sums exactly (FP64, or FP32 TwoSum pairs for an
// FP32 state), the 40 extremes in R (exact); one thread per quantity joins the three
// parts in FP64. Deterministic for any block size <= BT.
template <typename R>
__device__ __forceinline__ void block_tne(const R* Dk, bool active, double* partials, int nblocks,
                                          int b)
{
    constexpr int LD = BT + 1;            // padded rows: the readers walk along a row
    constexpr int NS = 2 * TK + 2;        // sums: Delta_k, |Delta_k|, d, d^2
    constexpr int NE = 2 * TK;            // extremes: min and max of Delta_k
    __shared__ R sD[TK + 2][LD];
    __shared__ unsigned char sact[BT];
    __shared__ double spart[NQ][3];
    const int t = threadIdx.x + threadIdx.y * blockDim.x;
    const int nt = blockDim.x * blockDim.y;
    const int per = (nt + 2) / 3; // cells per part
    R d2 = R(0);
#pragma unroll
    for (int k = 0; k < TK; k++) {
        sD[k][t] = Dk[k];
        d2 = fma(Dk[k], Dk[k], d2);
    }
    sD[TK][t] = sqrt(d2);
    sD[TK + 1][t] = d2;
    sact[t] = active ? 1 : 0;
    __syncthreads();
    for (int w = t; w < 3 * NS; w += nt) {
        const int s = w / 3, part = w - 3 * s;
        const int q = s < 2 * TK ? s : 4 * TK + (s - 2 * TK);
        const int row = s < TK ? s : (s < 2 * TK ? s - TK : TK + (s - 2 * TK));
        const bool absv = s >= TK && s < 2 * TK;
        const int j1 = min((part + 1) * per, nt);
        if constexpr (sizeof(R) == 4) {
            // FP32 terms summed exactly: each addition's rounding error (TwoSum) goes to
            // a compensating term, the pair joined in FP64 once (the FP64 unit runs at
            // 1/58 of the FP32 rate on this part)
            float sum = 0.f, comp = 0.f;
            for (int j = part * per; j < j1; j++) {
                if (!sact[j]) continue;
                const float v = absv ? fabsf(sD[row][j]) : sD[row][j];
                const lbk::df t2 = lbk::two_sum(sum, v);
                sum = t2.hi;
                comp += t2.lo;
            }
            spart[q][part] = (double)sum + (double)comp;
        } else {
            double acc = 0.0;
            for (int j = part * per; j < j1; j++) {
                if (!sact[j]) continue;
                const double v = (double)sD[row][j];
                acc += absv ? fabs(v) : v;
            }
            spart[q][part] = acc;
        }
    }
    for (int w = t; w < 3 * NE; w += nt) {
        const int e = w / 3, part = w - 3 * e;
        const bool mn = e < TK;
        const int k = mn ? e : e - TK;
        const int j1 = min((part + 1) * per, nt);
        bool any = false;
        R m = R(0);
        for (int j = part * per; j < j1; j++) {
            if (!sact[j]) continue;
            const R v = sD[k][j];
            m = !any ? v : (mn ? fmin(m, v) : fmax(m, v));
            any = true;
        }
        spart[2 * TK + e][part] = any ? (double)m : (mn ? DBL_MAX : -DBL_MAX);
    }
    __syncthreads();
    for (int q = t; q < NQ; q += nt) {
        const int kind = tkind(q);
        partials[(size_t)q * nblocks + b] =
            tcomb(kind, tcomb(kind, spart[q][0], spart[q][1]), spart[q][2]);
    }
}

// ---- the step -----------------------------------------------------------------------
// conserved moments of one cell from its butterflies g, then rho, u, T (Eqs. (5)-(7)); FP64
struct Macro {
    double rho, ux, uy, T;
    bool hot, ok; // T > T_ig; rho, T > 0 and finite
};
__device__ __forceinline__ Macro recover24(const Model<double>& K, const double* f, const double* g)
{
    double P[6];
#pragma unroll
    for (int o = 0; o < 6; o++) P[o] = (o & 1) ? g[(o / 2) * 3 + 2] : ad(g[(o / 2) * 3], g[(o / 2) * 3 + 1]);
    Macro m;
    m.rho = ad(ad(ad(P[0], P[1]), ad(P[2], P[3])), ad(P[4], P[5]));
    double jx = mu(K.cd[0], g[9]), jy = mu(K.cd[0], g[15]), e = mu(K.wod[0], P[0]);
#pragma unroll
    for (int o = 1; o < 6; o++) {
        jx = fm(K.cd[o], g[9 + o], jx);
        jy = fm(K.cd[o], g[15 + o], jy);
        e = fm(K.wod[o], P[o], e);
    }
    const double q = lbk::recip64(m.rho);
    m.ux = mu(jx, q);
    m.uy = mu(jy, q);
    m.T = mu(fm(e, q, -fm(m.ux, m.ux, mu(m.uy, m.uy))), K.inv_DI);
    const long long rb = dbits(m.rho), tb = dbits(m.T), big = dbits(DBL_MAX);
    m.ok = rb > 0 && rb <= big && tb > 0 && tb <= big;
    m.hot = tb > dbits(K.T_ig);
    return m;
}
// the same of an FP32 state: the sums exact double-floats on the FP32 pipes, carried into FP64
__device__ __forceinline__ Macro recover24(const Model<float>& K, const float* f, const float*)
{
    using lbk::S1;
    S1 r{0.f, 0.f}, jx{0.f, 0.f}, jy{0.f, 0.f}, e{0.f, 0.f};
#pragma unroll
    for (int o = 0; o < 6; o++) {
        const float a = f[4 * o], b = f[4 * o + 1], c = f[4 * o + 2], d = f[4 * o + 3];
        const S1 sac = lbk::s_sum(a, c), sbd = lbk::s_sum(b, d);
        const S1 dac = lbk::s_sum(a, -c), dbd = lbk::s_sum(b, -d);
        const S1 sum = lbk::s_add(sac, sbd);
        const S1 gx = (o & 1) ? lbk::s_sub(dac, dbd) : dac, gy = (o & 1) ? lbk::s_add(dac, dbd) : dbd;
        const S1 px = lbk::s_mul(gx, K.cdh[o], K.cdl[o]), py = lbk::s_mul(gy, K.cdh[o], K.cdl[o]);
        const S1 pe = lbk::s_mul(sum, K.wdh[o], K.wdl[o]);
        r = o ? lbk::s_add(r, sum) : sum;
        jx = o ? lbk::s_add(jx, px) : px;
        jy = o ? lbk::s_add(jy, py) : py;
        e = o ? lbk::s_add(e, pe) : pe;
    }
    r = lbk::s_norm(r);
    jx = lbk::s_norm(jx);
    jy = lbk::s_norm(jy);
    e = lbk::s_norm(e);
    Macro m;
    m.rho = lbk::df_to_f64_fast(r.hi, r.lo);
    lbk::recover_one_f64_fast(r.hi, r.lo, m.rho, lbk::df_to_f64_fast(jx.hi, jx.lo),
                              lbk::df_to_f64_fast(jy.hi, jy.lo), lbk::df_to_f64_fast(e.hi, e.lo), K.inv_DI,
                              m.ux, m.uy, m.T);
    const long long tb = dbits(m.T), big = dbits(DBL_MAX);
    m.ok = r.hi > 0.f && r.hi <= FLT_MAX && fabsf(jx.hi) <= FLT_MAX && fabsf(jy.hi) <= FLT_MAX &&
           fabsf(e.hi) <= FLT_MAX && tb > 0 && tb <= big;
    m.hot = tb > dbits(K.T_ig);
    return m;
}

// rows r of sector sct of B applied to x, columns j0.. only
template <typename R>
__device__ __forceinline__ R row_dot(const R* B, int sct, int r, int j0, const R* x)
{
    const int n = sec_n(sct), b0 = sec_b(sct) + r * n, p0 = sec_p(sct);
    R acc = mu(B[b0 + j0], x[p0 + j0]);
#pragma unroll
    for (int j = 1; j < 9; j++)
        if (j0 + j < n) acc = fm(B[b0 + j0 + j], x[p0 + j0 + j], acc);
    return acc;
}
// the first moments of the sectors ee (m1, m4), oe (m2), eo (m3) are conserved
__host__ __device__ constexpr int sec_cons(int s) { return s == 0 ? 2 : (s == 3 ? 0 : 1); }

// velocity space from sector components whose butterfly scales B has folded in
template <typename R>
__device__ __forceinline__ void unfly(const R* g, R* f)
{
#pragma unroll
    for (int o = 0; o < 6; o++) {
        const int e0 = (o / 2) * 3;
        if ((o & 1) == 0) {
            f[4 * o] = ad(g[e0], g[9 + o]);
            f[4 * o + 1] = ad(g[e0 + 1], g[15 + o]);
            f[4 * o + 2] = ad(g[e0], -g[9 + o]);
            f[4 * o + 3] = ad(g[e0 + 1], -g[15 + o]);
        } else {
            const R ep = ad(g[e0 + 2], g[21 + o / 2]), em = ad(g[e0 + 2], -g[21 + o / 2]);
            const R xp = ad(g[9 + o], g[15 + o]), xm = ad(g[9 + o], -g[15 + o]);
            f[4 * o] = ad(ep, xp);
            f[4 * o + 1] = ad(em, -xm);
            f[4 * o + 2] = ad(ep, -xp);
            f[4 * o + 3] = ad(em, xm);
        }
    }
}
// M^-1 applied to w (sector order); CONS: the conserved entries are zero and left out
template <bool CONS, typename R>
__device__ __forceinline__ void inverse24(const Model<R>& K, const R* w, R* f)
{
    R g[NV];
#pragma unroll
    for (int sct = 0; sct < NSEC; sct++)
#pragma unroll
        for (int r = 0; r < 9; r++)
            if (r < sec_n(sct)) g[sec_p(sct) + r] = row_dot(K.Bis, sct, r, CONS ? sec_cons(sct) : 0, w);
    unfly(g, f);
}

// the products that f_hat^eq is made of
template <typename R>
struct Eq24 {
    R m1, m2, m3, ux, uy, T, u2, Ta, Tb, A, B, pT, rIT, IT, C, G, H;
};
template <typename R>
__device__ __forceinline__ Eq24<R> eq24(const Model<R>& K, R rho, R ux, R uy, R T)
{
    Eq24<R> e;
    e.m1 = rho;
    e.ux = ux;
    e.uy = uy;
    e.T = T;
    e.m2 = mu(rho, ux);
    e.m3 = mu(rho, uy);
    constexpr bool F4 = sizeof(R) == 4; // each of u^2, T + u^2, (D+I+4) T + u^2 rounded once
    const R ux2 = mu(ux, ux), uy2 = mu(uy, uy), I3 = mu(R(3), K.I_r);
    e.u2 = F4 ? fm(ux, ux, uy2) : ad(ux2, uy2);
    e.Ta = F4 ? fm(ux, ux, T) : ad(T, ux2);
    e.Tb = F4 ? fm(uy, uy, T) : ad(T, uy2);
    e.A = fm(ad(K.DI_r, R(2)), T, e.u2);
    e.B = F4 ? fm(ad(K.DI_r, R(4)), T, e.u2) : fm(R(2), T, e.A);
    e.pT = mu(rho, T);
    e.IT = mu(K.I_r, T);
    e.rIT = mu(rho, e.IT);
    e.C = fm(e.u2, e.u2, mu(T, fm(ad(K.DI_r, R(10)), e.u2, mu(mu(R(4), ad(K.DI_r, R(4))), T))));
    e.G = mu(e.IT, fm(ad(R(4), I3), T, e.u2));
    e.H = fm(ad(R(2), I3), T, e.u2);
    return e;
}
// h - a b of a moment h and its equilibrium: FP64 one FMA, FP32 the product rounded like the moment
// (deltas, cellops.cuh)
__device__ __forceinline__ double less(double h, double a, double b) { return fm(-a, b, h); }
__device__ __forceinline__ float less(float h, float a, float b) { return sub(h, mu(a, b)); }
// h - (m1 A T + a B) and 3 T + u^2
__device__ __forceinline__ double less4(const Eq24<double>& e, double h, double a) { return fm(-a, e.B, fm(-e.pT, e.A, h)); }
__device__ __forceinline__ float less4(const Eq24<float>& e, float h, float a)
{
    return sub(h, fm(mu(e.m1, e.A), e.T, mu(a, e.B)));
}
__device__ __forceinline__ double three(double T, double Ta, double) { return fm(2.0, T, Ta); }
__device__ __forceinline__ float three(float T, float, float u) { return fm(3.f, T, mu(u, u)); }
// h - f_hat^eq of moment k (0-based)
template <typename R>
__device__ __forceinline__ R minus_eq(const Eq24<R>& e, int k, R h)
{
    switch (k) {
    case 4: return less(h, e.m1, e.Ta);
    case 5: return less(h, e.m2, e.uy);
    case 6: return less(h, e.m1, e.Tb);
    case 7: return less(h, e.m2, e.A);
    case 8: return less(h, e.m3, e.A);
    case 9: return less(h, e.m2, three(e.T, e.Ta, e.ux));
    case 10: return less(h, e.m3, e.Ta);
    case 11: return less(h, e.m2, e.Tb);
    case 12: return less(h, e.m3, three(e.T, e.Tb, e.uy));
    case 13: return less4(e, h, mu(e.m2, e.ux));
    case 14: return less(h, mu(e.m2, e.uy), e.B);
    case 15: return less4(e, h, mu(e.m3, e.uy));
    case 16: return less(h, e.rIT, e.Ta);
    case 17: return less(h, mu(e.m2, e.uy), e.IT);
    case 18: return less(h, e.rIT, e.Tb);
    case 19: return less(h, e.rIT, e.H);
    case 20: return less(h, e.m2, e.C);
    case 21: return less(h, e.m3, e.C);
    case 22: return less(h, e.m2, e.G);
    default: return less(h, e.m3, e.G);
    }
}

template <typename R>
__device__ __forceinline__ R eq_moment(const Model<R>& K, const Eq24<R>& e, int k)
{
    return k == 0 ? e.m1 : k == 1 ? e.m2 : k == 2 ? e.m3 : k == 3 ? mu(e.m1, fm(K.DI_r, e.T, e.u2)) : -minus_eq(e, k, R(0));
}

// Per-warp TNE statistics of a tile row: row k of td (stride ld) holds Delta_{k+5} (k < TK), d
// and d^2 of the block's cells; the lanes take one quantity each over the warp's cells in
// `mask`, first the signed sums and minima, then the sums of |Delta| and maxima, and join them
// to the launch's statistics acc [NQ]. FP64 terms add in FP64, FP32 terms as exact pairs.
template <typename R>
__device__ __forceinline__ void warp_tne24(const R* td, int ld, unsigned mask, double* acc)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int pass = 0; pass < 2; pass++) {
        if (lane >= (pass ? TK : TK + 2)) continue;
        const R* p = td + lane * ld;
        double sum;
        R m = R(0);
        bool any = false;
        if constexpr (sizeof(R) == 8) {
            sum = 0.0;
            const long long keep = pass ? 0x7fffffffffffffffll : -1ll, flip = pass ? -1ll : 0ll;
            long long v = lbk::order64(DBL_MAX);
            for (int j = 0; j < 32; j++) {
                if (!(mask >> j & 1u)) continue;
                sum += __longlong_as_double(__double_as_longlong(p[j]) & keep);
                const long long k = lbk::order64(p[j]) ^ flip;
                v = k < v ? k : v;
            }
            any = mask != 0;
            m = lbk::unorder64(v ^ flip);
        } else {
            float s = 0.f, c = 0.f, v = FLT_MAX;
            const float sign = pass ? -1.f : 1.f;
            for (int j = 0; j < 32; j++) {
                if (!(mask >> j & 1u)) continue;
                const lbk::df t = lbk::two_sum(s, pass ? fabsf(p[j]) : p[j]);
                s = t.hi;
                c += t.lo;
                v = fminf(v, sign * p[j]);
            }
            sum = (double)s + (double)c;
            any = mask != 0;
            m = sign * v;
        }
        const int qs = lane < TK ? (pass ? TK : 0) + lane : 3 * TK + lane; // d, d^2 at 4 TK, 4 TK + 1
        acc[qs] += sum;
        if (lane < TK && any) {
            const int qm = (pass ? 3 * TK : 2 * TK) + lane;
            acc[qm] = pass ? fmax(acc[qm], (double)m) : fmin(acc[qm], (double)m);
        }
    }
}

// Tiles of 32 x 8 (FP32) or 32 x 4 cells (2-D), 32 cells (1-D), one cell per thread.
template <typename R, bool TWO_D>
struct Tile24 {
    static constexpr int TX = 32, TY = !TWO_D ? 1 : (sizeof(R) == 8 ? 4 : 8), TT = TX * TY;
    static constexpr int HY = TWO_D ? 2 : 0, SW = TX + 4, SH = TY + 2 * HY, PS = SW * SH;
    static constexpr int UW = TX + 2, UH = TWO_D ? TY + 2 : 1; // u of the tile and its rim
    static constexpr size_t smem(bool tne)
    {
        return sizeof(R) * ((size_t)NP * PS + 2 * UW * UH) +
               (tne ? sizeof(double) * (size_t)TY * NQ + sizeof(R) * (TK + 2) * (TT + 1) : 0);
    }
};

// SRT: the single-relaxation-time fast path (all R_5..R_24 equal, no TNE due): with one
// rate the moment-space relaxation is -R (f - M^-1 f_hat^eq) in velocity space (the SRT
// form of Sec. V) and A_hat vanishes, so the forward transform of f is skipped and only
// f^eq = M^-1 f_hat^eq is formed (it also feeds the chemical term of Eq. (24)).
//
// Each block walks tiles (grid-stride loop): the 25 planes of the tile and its two-cell halo
// are staged in shared memory by asynchronous copies, all in flight together; rho, u, T of the
// own cells and u of the rim are recovered; the cells are updated from registers and shared
// memory.
template <typename R, bool SRT, bool TWO_D, bool TNE>
__global__ void __launch_bounds__((Tile24<R, TWO_D>::TT), (TWO_D ? 2 : 1))
    step_kernel(const __grid_constant__ Model<R> K, const __grid_constant__ Args a)
{
    using C = Tile24<R, TWO_D>;
    constexpr int TX = C::TX, TY = C::TY, TT = C::TT, SW = C::SW, SH = C::SH, PS = C::PS, HY = C::HY,
                  UW = C::UW, UH = C::UH;
    extern __shared__ __align__(16) unsigned char smem[];
    R* sf = reinterpret_cast<R*>(smem);                        // [25][SH][SW]
    R* su = sf + NP * PS;                                      // u_x, u_y  [2][UH][UW]
    double* acc = reinterpret_cast<double*>(su + 2 * UH * UW); // the launch's statistics [TY][NQ]
    R* td = reinterpret_cast<R*>(acc + TY * NQ);               // [TK + 2][TT + 1]

    const int t = threadIdx.x, lx = t & 31, ly = t >> 5; // a warp is a row of the tile
    const R* __restrict__ in = static_cast<const R*>(a.in);
    R* __restrict__ out = static_cast<R*>(a.out);
    const bool tne = TNE && a.tne_every > 0;
    const int64_t step = tne ? a.ctr->step : 0;
    const bool do_tne = tne && step % a.tne_every == 0;
    if (do_tne)
        for (int i = lx; i < NQ; i += 32) acc[ly * NQ + i] = tkind(i) == 0 ? 0.0 : (tkind(i) == 1 ? DBL_MAX : -DBL_MAX);
    int bad = 0;

    const int tiles_x = (K.nx + TX - 1) / TX, ntiles = tiles_x * ((K.ny + TY - 1) / TY);
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int x0 = (tile % tiles_x) * TX, y0 = (tile / tiles_x) * TY;
        __syncthreads(); // the previous tile is done with shared memory
        lbk::stage_tile<NP, SH, SW, TY, TWO_D>(in, sf, x0 - 2, y0 - HY, K.nx, K.ny, K.pitch, K.plane, K.sides,
                                               K.sfeq, [](int p) { return mirror24(p); });
        lbk::cp_commit();
        lbk::cp_wait<0>();
        __syncthreads();
        if (TWO_D && K.wall && (y0 - HY < 0 || y0 + TY + HY > K.ny)) {
            // walls: the staged ghost rows hold copies of the edge row; add its correction
            for (int c = t; c < SW * SH; c += TT) {
                const int r = c / SW, y = y0 - HY + r, side = y < 0 ? 0 : 1;
                if ((y >= 0 && y < K.ny) || K.sides[2 + side] != 2) continue;
                bool m_;
                const int sx = lbk::source(x0 - 2 + c - r * SW, K.nx, K.sides, 0, m_);
                if (sx < 0) continue; // a corner, never read
                for (int i = 0; i < NV; i++) sf[i * PS + c] += K.wall[((size_t)side * NV + i) * K.nx + sx];
            }
            __syncthreads();
        }
        const int x = x0 + lx, y = y0 + ly;
        const bool active = x < K.nx && y < K.ny;
        const R* s0 = sf + (ly + HY) * SW + lx + 2;
        R g[NV];
        Macro m;
        if (y < K.ny) { // whole warps past the last row have nothing to do
            R f[NV];
#pragma unroll
            for (int i = 0; i < NV; i++) f[i] = s0[i * PS];
            butterfly(f, g);
            m = recover24(K, f, g);
            if (active && !m.ok) bad = 1;
            su[(ly + (TWO_D ? 1 : 0)) * UW + lx + 1] = to_fast<R>(m.ux);
            su[(UH + ly + (TWO_D ? 1 : 0)) * UW + lx + 1] = to_fast<R>(m.uy);
        }
        if (!SRT) { // u of the rim; the row past the grid is one of a ragged tile's own
            const int rows = TWO_D ? 2 * UW : 0, rim = rows + 2 * TY;
            for (int c = t; c < rim || (TWO_D && y0 + TY > K.ny && c < rim + TX); c += TT) {
                int rx, ry;
                if (c < rows) rx = c % UW, ry = c < UW ? 0 : UH - 1;
                else if (c < rim) rx = (c & 1) ? UW - 1 : 0, ry = (TWO_D ? 1 : 0) + (c - rows) / 2;
                else rx = 1 + c - rim, ry = K.ny - y0 + 1;
                const R* sr = sf + (ry + (TWO_D ? 1 : 0)) * SW + rx + 1;
                R f[NV], h[NV];
#pragma unroll
                for (int i = 0; i < NV; i++) f[i] = sr[i * PS];
                butterfly(f, h);
                const Macro r = recover24(K, f, h);
                su[ry * UW + rx] = to_fast<R>(r.ux);
                su[(UH + ry) * UW + rx] = to_fast<R>(r.uy);
            }
        }
        __syncthreads();
        if (y >= K.ny) continue;

        const R rr = to_fast<R>(m.rho), uxr = to_fast<R>(m.ux), uyr = to_fast<R>(m.uy), Tr = to_fast<R>(m.T);
        const Eq24<R> e = eq24(K, rr, uxr, uyr, Tr);
        const R lam0 = s0[NV * PS];
        // reaction over dt with p and T frozen at t_n (Eq. (28), m = n = 1), in FP64
        const bool hot = m.hot && lam0 != R(1);
        const bool react = __any_sync(0xffffffffu, hot);
        R dlam = R(0), chem = R(0);
        if (react && hot) {
            const double pT = mu(m.rho, m.T);
            const double d = reaction_increment<double>((double)lam0, mu(K.omega1, pT), mu(K.omega2, pT), K.dt);
            const double rT = lbk::recip64(m.T);
            dlam = to_fast<R>(d);
            chem = to_fast<R>(mu(mu(K.kchem, d), mu(rT, rT))); // Q lambda' / (I (D+I) T^2)
        }
        R W[NV], fe[NV];
        if constexpr (SRT) {
            R w[NV];
#pragma unroll
            for (int p = 0; p < NV; p++) w[p] = eq_moment(K, e, mom_of(p));
            inverse24<false>(K, w, fe);
#pragma unroll
            for (int i = 0; i < NV; i++) W[i] = mu(-K.S[4], sub(s0[i * PS], fe[i]));
        } else {
            // Delta of the non-conserved moments, in sector order
            R w[NV];
#pragma unroll
            for (int sct = 0; sct < NSEC; sct++)
#pragma unroll
                for (int r = 0; r < 9; r++)
                    if (r < sec_n(sct)) {
                        const int p = sec_p(sct) + r;
                        w[p] = r < sec_cons(sct) ? R(0) : minus_eq(e, mom_of(p), row_dot(K.Bf, sct, r, 0, g));
                    }
            if (do_tne) {
                R d2 = R(0);
#pragma unroll
                for (int p = 0; p < NV; p++)
                    if (mom_of(p) >= 4) {
                        td[(mom_of(p) - 4) * (TT + 1) + t] = w[p];
                        d2 = fm(w[p], w[p], d2);
                    }
                td[TK * (TT + 1) + t] = sqrt(d2);
                td[(TK + 1) * (TT + 1) + t] = d2;
                const unsigned mask = __ballot_sync(0xffffffffu, active);
                __syncwarp();
                warp_tne24(td + ly * 32, TT + 1, mask, acc + ly * NQ);
            }
            if (react) { // f^eq for the chemical term
                if constexpr (sizeof(R) == 8) { // f - M^-1 Delta: no conserved entries, no f_hat^eq
                    inverse24<true>(K, w, fe);
#pragma unroll
                    for (int i = 0; i < NV; i++) fe[i] = sub(s0[i * PS], fe[i]);
                } else { // M^-1 f_hat^eq: free of the rounding that Delta's cancellation brings in FP32
                    R q[NV];
#pragma unroll
                    for (int p = 0; p < NV; p++) q[p] = eq_moment(K, e, mom_of(p));
                    inverse24<false>(K, q, fe);
                }
            }
            // relaxation with A_hat_8, A_hat_9 (Eqs. (3)-(4), sign as in Eq. (29)) and back
#pragma unroll
            for (int p = 0; p < NV; p++) w[p] = mom_of(p) >= 4 ? mu(-K.S[mom_of(p)], w[p]) : R(0);
            {
                const R* u0 = su + (ly + (TWO_D ? 1 : 0)) * UW + lx + 1;
                const R* v0 = u0 + UH * UW;
                const R gxx = mu(sub(u0[1], u0[-1]), K.hdx_r), gyx = mu(sub(v0[1], v0[-1]), K.hdx_r);
                const R gxy = TWO_D ? mu(sub(u0[TWO_D ? UW : 0], u0[TWO_D ? -UW : 0]), K.hdy_r) : R(0);
                const R gyy = TWO_D ? mu(sub(v0[TWO_D ? UW : 0], v0[TWO_D ? -UW : 0]), K.hdy_r) : R(0);
                const R th = mu(TWO_D ? ad(gxx, gyy) : gxx, K.inv_DI_r), sh = mu(R(2), TWO_D ? ad(gyx, gxy) : gyx);
                w[10] = fm(mu(e.pT, K.A8c_r), fm(uyr, sh, mu(mu(R(4), uxr), sub(gxx, th))), w[10]);  // m8
                w[16] = fm(mu(e.pT, K.A9c_r), fm(uxr, sh, mu(mu(R(4), uyr), sub(gyy, th))), w[16]);  // m9
            }
            inverse24<true>(K, w, W);
        }
        if (react) {
            // C_i = f_i^eq chem [-(1 + D) I T + I (v_i - u)^2 + eta_i^2] (Eq. (24)), the square
            // multiplied out: per orbit a - b_x s_x - b_y s_y
            const R base = fm(K.I_r, e.u2, mu(R(-3), e.IT)), i2 = mu(R(2), K.I_r);
#pragma unroll
            for (int o = 0; o < 6; o++) {
                const R ao = mu(chem, ad(base, K.chem_o[o])), cc = mu(chem, mu(i2, K.c_r[o]));
                const R bx = mu(cc, uxr), by = mu(cc, uyr);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int i = 4 * o + j, sx = vsign_x(i), sy = vsign_y(i);
                    R k = ao;
                    if (sx) k = sx > 0 ? sub(k, bx) : ad(k, bx);
                    if (sy) k = sy > 0 ? sub(k, by) : ad(k, by);
                    W[i] = fm(fe[i], k, W[i]);
                }
            }
        }

        // NND flux differences (upwind side fixed per velocity), Euler update; one rounding at
        // the size of f
        auto nnd = [&](const R* q, R q0, int d, bool neg) -> R {
            const R l = q[-d], r = q[d];
            return neg ? lbk::nnd3(sub(q0, l), sub(r, q0), sub(q[2 * d], r), true)
                       : lbk::nnd3(sub(l, q[-2 * d]), sub(q0, l), sub(r, q0), false);
        };
        auto nnd_by = [&](const R* q, R q0, int d, bool neg) -> R { // the side known at run time
            const R* c = neg ? q + d : q;
            const R c0 = neg ? *c : q0, l = c[-d];
            return lbk::nnd3(sub(l, c[-2 * d]), sub(c0, l), sub(c[d], c0), neg);
        };
        const size_t gi = (size_t)y * K.pitch + x;
#pragma unroll
        for (int i = 0; i < NV; i++) {
            const R f0 = s0[i * PS];
            R w = W[i];
            if (vsign_x(i)) w = fm(-K.vxs[i], nnd(s0 + i * PS, f0, 1, vsign_x(i) < 0), w);
            if (TWO_D && vsign_y(i)) w = fm(-K.vys[i], nnd(s0 + i * PS, f0, SW, vsign_y(i) < 0), w);
            if (active) out[(size_t)i * K.plane + gi] = fm(K.dt_r, w, f0);
        }
        // lambda: u . grad(lambda) with NND interface values, then the update
        const R* sl = s0 + NV * PS;
        R la = fm(mu(mu(-K.dt_r, K.inv_dx_r), uxr), nnd_by(sl, lam0, 1, lbk::negative(uxr)), dlam);
        if (TWO_D) la = fm(mu(mu(-K.dt_r, K.inv_dy_r), uyr), nnd_by(sl, lam0, SW, lbk::negative(uyr)), la);
        if (active) out[(size_t)NV * K.plane + gi] = lbk::clamp01(ad(lam0, la));
    }

    // status, TNE partials, step counter: without TNE no block reads the counter, so block 0
    // moves it on; with TNE the last block to finish does
    if (__syncthreads_or(bad) && t == 0) atomicOr(&a.ctr->status, 1);
    if (do_tne)
        for (int q = t; q < NQ; q += TT) {
            double v = acc[q];
            for (int w = 1; w < TY; w++) v = tcomb(tkind(q), v, acc[w * NQ + q]);
            a.partials[(size_t)q * gridDim.x + blockIdx.x] = v;
        }
    if (!tne) {
        if (blockIdx.x == 0 && t == 0) {
            a.ctr->tne_pending = 0;
            a.ctr->step += 1;
        }
    } else if (t == 0) {
        if (atomicAdd(&a.ctr->arrivals, 1u) == gridDim.x - 1) {
            if (do_tne) {
                a.ctr->hist_count += 1;
                a.ctr->tne_step = step;
            }
            a.ctr->tne_pending = do_tne ? 1 : 0;
            a.ctr->step = step + 1;
            a.ctr->arrivals = 0u;
        }
    }
}

template <typename R, bool SRT, bool TWO_D, bool TNE>
cudaError_t step_prepare()
{
    static cudaError_t done = cudaFuncSetAttribute(step_kernel<R, SRT, TWO_D, TNE>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)Tile24<R, TWO_D>::smem(TNE));
    return done;
}
// blocks of a launch: all tiles, or as many as the SMs hold at a time
template <typename R, bool SRT, bool TWO_D, bool TNE>
int step_blocks(int nx, int ny, int sms)
{
    using C = Tile24<R, TWO_D>;
    static int per_sm = -1;
    if (per_sm < 0) {
        if (step_prepare<R, SRT, TWO_D, TNE>() != cudaSuccess) return -1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, step_kernel<R, SRT, TWO_D, TNE>, C::TT,
                                                          C::smem(TNE)) != cudaSuccess)
            return -1;
        if (per_sm < 1) per_sm = 1;
    }
    const int64_t tiles = (int64_t)((nx + C::TX - 1) / C::TX) * ((ny + C::TY - 1) / C::TY);
    const int64_t g = (int64_t)per_sm * sms;
    return (int)(tiles < g ? tiles : g);
}
template <typename R, bool SRT, bool TWO_D, bool TNE>
cudaError_t step_launch(const Model<R>& K, const Args& a, int blocks, cudaStream_t s)
{
    using C = Tile24<R, TWO_D>;
    const cudaError_t e = step_prepare<R, SRT, TWO_D, TNE>();
    if (e != cudaSuccess) return e;
    step_kernel<R, SRT, TWO_D, TNE><<<blocks, C::TT, C::smem(TNE), s>>>(K, a);
    return cudaGetLastError();
}
// the step variant of a handle: CALL(R, SRT, TWO_D, TNE) of its precision, collision, shape and
// records
#define V24_VARIANT(CALL, f64, srt, two_d, tne)                                                    \
    ((f64) ? ((two_d) ? ((srt) ? CALL(double, true, true, false)                                   \
                         : (tne) ? CALL(double, false, true, true) : CALL(double, false, true, false)) \
                      : ((srt) ? CALL(double, true, false, false)                                  \
                         : (tne) ? CALL(double, false, false, true) : CALL(double, false, false, false))) \
           : ((two_d) ? ((srt) ? CALL(float, true, true, false)                                    \
                         : (tne) ? CALL(float, false, true, true) : CALL(float, false, true, false)) \
                      : ((srt) ? CALL(float, true, false, false)                                   \
                         : (tne) ? CALL(float, false, false, true) : CALL(float, false, false, false))))

// ---- short 1-D grids in FP64: four warps to a window of 32 cells -----------------
// One warp to 32 cells leaves three quarters of each SM's FP64 unit idle on a grid of a few
// thousand cells. Here warps 0..2 hold the velocities of one speed group each, warp 3 lambda; the moment
// sectors are shared out as ee (first rows) to warp 0, oe to 1, eo to 2, ee (last rows) and oo to
// 3. Butterflies, the ee entries and the back-transformed sectors pass through shared memory,
// three barriers a step; what neighbouring cells provide stays within a warp (shuffles). Up to
// `kmax` steps run in one launch, of the window all but 2 kmax cells at either end being right
// after them. The operations and their order are those of step_kernel.
constexpr int SPLIT_EE = 5; // inverse rows 0..4 of ee in warp 0, Delta rows 2..5; the rest in warp 3

struct SplitShared {
    double g[NV][32], dx[9][32], dy[9][32], go[NV][32], ge[NV][32], lam[32];
};
__device__ __forceinline__ void join_warps() // a barrier that the four warps reach from their own code
{
    asm volatile("bar.sync 1, 128;" ::: "memory");
}

template <int Q>
__device__ __forceinline__ void split24_steps(const Model<double>& K, const Args& a, int nsteps, int kmax,
                                              SplitShared& sh)
{
    const unsigned all = 0xffffffffu;
    constexpr int n = 32;
    const int t = threadIdx.x & 31, h = 2 * kmax, own = n - 2 * h;
    const int nx = K.nx, x0 = blockIdx.x * own - h, x = x0 + t;
    const double* in = static_cast<const double*>(a.in);
    int gx = x, dir = -1;
    bool fixed = false;
    if (x < 0 || x >= nx) {
        const int s = x < 0 ? 0 : 1, code = K.sides[s];
        if (code == 0) {
            gx = x % nx;
            gx = gx < 0 ? gx + nx : gx;
        } else {
            gx = x < 0 ? 0 : nx - 1;
            fixed = true;
            if (code == 3) dir = s;
        }
    }
    const int lo = K.sides[0] == 1 && -x0 > 0 ? (-x0 < n ? -x0 : n - 1) : 0;
    const int hi = K.sides[1] == 1 && nx - 1 - x0 < n - 1 ? (nx - 1 - x0 > 0 ? nx - 1 - x0 : 0) : n - 1;
    auto at = [&](int j) { return j < lo ? lo : (j > hi ? hi : j); };
    const int jm1 = at(t - 1), j0 = at(t), jp1 = at(t + 1);
    const int dm2 = t >= 2 ? t - 2 : 0, dm1 = t >= 1 ? t - 1 : 0, dp1 = t + 1 < n ? t + 1 : n - 1;
    const bool mine = t >= h && t < h + own && x < nx;
    auto slope3 = [&](double q, double& l2, double& l1, double& d, double& r1) {
        d = sub(__shfl_sync(all, q, jp1), __shfl_sync(all, q, j0));
        l2 = __shfl_sync(all, d, dm2);
        l1 = __shfl_sync(all, d, dm1);
        r1 = __shfl_sync(all, d, dp1);
    };

    constexpr int G = Q < 3 ? Q : 0; // the speed group (warp 3: none)
    double f[8], lam = dir >= 0 ? K.sfeq[dir][NV] : in[(size_t)NV * K.plane + gx];
    if constexpr (Q < 3) {
#pragma unroll
        for (int j = 0; j < 8; j++) f[j] = dir >= 0 ? K.sfeq[dir][8 * G + j] : in[(size_t)(8 * G + j) * K.plane + gx];
    }
    int bad = 0;
    for (int s = 0; s < nsteps; s++) {
        if constexpr (Q < 3) {
            const double s02 = f[0] + f[2], s13 = f[1] + f[3];
            sh.g[3 * G][t] = s02;
            sh.g[3 * G + 1][t] = s13;
            sh.g[9 + 2 * G][t] = f[0] - f[2];
            sh.g[15 + 2 * G][t] = f[1] - f[3];
            const double ac = f[4] + f[6], bd = f[5] + f[7], am = f[4] - f[6], bm = f[5] - f[7];
            sh.g[3 * G + 2][t] = ac + bd;
            sh.g[10 + 2 * G][t] = am - bm;
            sh.g[16 + 2 * G][t] = am + bm;
            sh.g[21 + G][t] = ac - bd;
        } else {
            sh.lam[t] = lam;
        }
        join_warps();
        double g[NV];
#pragma unroll
        for (int p = 0; p < NV; p++) g[p] = sh.g[p][t];
        if constexpr (Q < 3) lam = sh.lam[t];
        const Macro m = recover24(K, nullptr, g);
        if (mine && !m.ok) bad = 1;
        const Eq24<double> e = eq24(K, m.rho, m.ux, m.uy, m.T);
        const bool hot = m.hot && dbits(lam) != dbits(1.0);
        const bool react = __any_sync(all, hot);
        double dlam = 0.0, chem = 0.0;
        if (react && hot) {
            const double pT = mu(m.rho, m.T);
            dlam = reaction_increment<double>(lam, mu(K.omega1, pT), mu(K.omega2, pT), K.dt);
            const double rT = lbk::recip64(m.T);
            chem = mu(mu(K.kchem, dlam), mu(rT, rT));
        }
        // this warp's Delta (y) and relaxed entries (w), in sector order
        double w[NV], y[NV];
        auto delta = [&](int sct, int r) {
            const int p = sec_p(sct) + r;
            y[p] = minus_eq(e, mom_of(p), row_dot(K.Bf, sct, r, 0, g));
            w[p] = mu(-K.S[mom_of(p)], y[p]);
        };
        if constexpr (Q == 0) {
#pragma unroll
            for (int r = 2; r < 6; r++) delta(0, r);
        } else if constexpr (Q == 3) {
#pragma unroll
            for (int r = 6; r < 9; r++) delta(0, r);
#pragma unroll
            for (int r = 0; r < 3; r++) delta(3, r);
        } else {
#pragma unroll
            for (int r = 1; r < 6; r++) delta(Q, r);
            const double gxx = mu(sub(__shfl_sync(all, m.ux, jp1), __shfl_sync(all, m.ux, jm1)), K.hdx_r);
            const double gyx = mu(sub(__shfl_sync(all, m.uy, jp1), __shfl_sync(all, m.uy, jm1)), K.hdx_r);
            const double th = mu(gxx, K.inv_DI_r), shr = mu(2.0, gyx);
            if constexpr (Q == 1)
                w[10] = fm(mu(e.pT, K.A8c_r), fm(m.uy, shr, mu(mu(4.0, m.ux), sub(gxx, th))), w[10]);
            else
                w[16] = fm(mu(e.pT, K.A9c_r), fm(m.ux, shr, mu(mu(4.0, m.uy), sub(0.0, th))), w[16]);
        }
        if constexpr (Q == 0 || Q == 3) { // the ee entries, wanted by both
#pragma unroll
            for (int p = 2; p < 9; p++)
                if ((p < 6) == (Q == 0)) {
                    sh.dx[p][t] = w[p];
                    if (react) sh.dy[p][t] = y[p];
                }
        }
        join_warps();
        if constexpr (Q == 0 || Q == 3) {
#pragma unroll
            for (int p = 2; p < 9; p++)
                if ((p < 6) != (Q == 0)) {
                    w[p] = sh.dx[p][t];
                    if (react) y[p] = sh.dy[p][t];
                }
        }
        auto rows = [&](const double* v, double (*to)[32]) {
            if constexpr (Q == 0 || Q == 3) {
#pragma unroll
                for (int r = 0; r < 9; r++)
                    if ((r < SPLIT_EE) == (Q == 0)) to[r][t] = row_dot(K.Bis, 0, r, 2, v);
            }
            if constexpr (Q == 3) {
#pragma unroll
                for (int r = 0; r < 3; r++) to[21 + r][t] = row_dot(K.Bis, 3, r, 0, v);
            } else if constexpr (Q != 0) {
#pragma unroll
                for (int r = 0; r < 6; r++) to[sec_p(Q) + r][t] = row_dot(K.Bis, Q, r, 1, v);
            }
        };
        rows(w, sh.go);
        if (react) rows(y, sh.ge);
        join_warps();
        // back to this group's velocities; chemical term, NND differences, Euler update
        double nlam = lam;
        if constexpr (Q < 3) {
            auto back = [&](const double (*c)[32], double* v) {
                const double e0 = c[3 * G][t], e1 = c[3 * G + 1][t], ax = c[9 + 2 * G][t], ay = c[15 + 2 * G][t];
                v[0] = ad(e0, ax);
                v[1] = ad(e1, ay);
                v[2] = ad(e0, -ax);
                v[3] = ad(e1, -ay);
                const double e2 = c[3 * G + 2][t], o = c[21 + G][t], bx = c[10 + 2 * G][t], by = c[16 + 2 * G][t];
                const double ep = ad(e2, o), em = ad(e2, -o), xp = ad(bx, by), xm = ad(bx, -by);
                v[4] = ad(ep, xp);
                v[5] = ad(em, -xm);
                v[6] = ad(ep, -xp);
                v[7] = ad(em, xm);
            };
            double W[8];
            back(sh.go, W);
            if (react) {
                double fe[8];
                back(sh.ge, fe);
                const double base = fm(K.I_r, e.u2, mu(-3.0, e.IT)), i2 = mu(2.0, K.I_r);
#pragma unroll
                for (int o = 0; o < 2; o++) {
                    const double ao = mu(chem, ad(base, K.chem_o[2 * G + o])), cc = mu(chem, mu(i2, K.c_r[2 * G + o]));
                    const double bx = mu(cc, m.ux), by = mu(cc, m.uy);
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const int i = 8 * G + 4 * o + j, sx = vsign_x(i), sy = vsign_y(i);
                        double k = ao;
                        if (sx) k = sx > 0 ? sub(k, bx) : ad(k, bx);
                        if (sy) k = sy > 0 ? sub(k, by) : ad(k, by);
                        W[4 * o + j] = fm(sub(f[4 * o + j], fe[4 * o + j]), k, W[4 * o + j]);
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const int i = 8 * G + j;
                if (vsign_x(i)) {
                    double l2, l1, d, r1;
                    slope3(f[j], l2, l1, d, r1);
                    const double X = vsign_x(i) < 0 ? lbk::nnd3(l1, d, r1, true) : lbk::nnd3(l2, l1, d, false);
                    W[j] = fm(-K.vxs[i], X, W[j]);
                }
                W[j] = fm(K.dt_r, W[j], f[j]);
                if (!fixed) f[j] = W[j];
            }
        } else {
            double l2, l1, d, r1;
            slope3(lam, l2, l1, d, r1);
            const bool neg = lbk::negative(m.ux);
            const double X = lbk::nnd3(neg ? l1 : l2, neg ? d : l1, neg ? r1 : d, neg);
            nlam = lbk::clamp01(ad(lam, fm(mu(mu(-K.dt_r, K.inv_dx_r), m.ux), X, dlam)));
            if (!fixed) lam = nlam;
        }
    }
    if (mine) {
        double* out = static_cast<double*>(a.out) + x;
        if constexpr (Q < 3) {
#pragma unroll
            for (int j = 0; j < 8; j++) out[(size_t)(8 * G + j) * K.plane] = f[j];
        } else {
            out[(size_t)NV * K.plane] = lam;
        }
    }
    if (Q == 3 && __any_sync(all, bad) && t == 0) atomicOr(&a.ctr->status, 1);
}

__global__ void __launch_bounds__(128)
    split_kernel(const __grid_constant__ Model<double> K, const __grid_constant__ Args a, int nsteps, int kmax)
{
    __shared__ SplitShared sh;
    switch (threadIdx.x >> 5) {
    case 0: split24_steps<0>(K, a, nsteps, kmax, sh); break;
    case 1: split24_steps<1>(K, a, nsteps, kmax, sh); break;
    case 2: split24_steps<2>(K, a, nsteps, kmax, sh); break;
    default: split24_steps<3>(K, a, nsteps, kmax, sh); break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctr->tne_pending = 0;
        a.ctr->step += nsteps;
    }
}

// TNE of a state on demand: Delta fields (optional) and block partials.
template <typename R>
__global__ void __launch_bounds__(BT) tne_kernel(const Model<R> K, const R* __restrict__ in,
                                                 double* delta, double* partials)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const bool active = x < K.nx && y < K.ny;
    R Dk[TK];
#pragma unroll
    for (int k = 0; k < TK; k++) Dk[k] = R(0);
    if (active) {
        const size_t g = (size_t)y * K.pitch + x;
        double rho, ux, uy, T;
        conserved_at(K, in, x, y, rho, ux, uy, &T);
        R q[NV];
        feq24<R>(K.I_r, K.DI_r, to_r<R>(rho), to_r<R>(ux), to_r<R>(uy), to_r<R>(T), q);
        R f[NV], gv[NV], h[NV];
#pragma unroll
        for (int i = 0; i < NV; i++) f[i] = __ldg(in + (size_t)i * K.plane + g);
        butterfly(f, gv);
        block_apply(K.Bf, gv, h);
#pragma unroll
        for (int p = 0; p < NV; p++)
            if (mom_of(p) >= 4) Dk[mom_of(p) - 4] = h[p] - q[mom_of(p)];
        if (delta) {
            const size_t n = (size_t)K.nx * K.ny, c = (size_t)y * K.nx + x;
#pragma unroll
            for (int k = 0; k < NV; k++) delta[k * n + c] = k < 4 ? 0.0 : (double)Dk[k - 4];
        }
    }
    block_tne(Dk, active, partials, gridDim.x * gridDim.y, blockIdx.x + blockIdx.y * gridDim.x);
}

// Record of a grid's partials: block q reduces quantity q in a fixed order.
// rec == nullptr: the step's record, into history slot (hist_count - 1) % cap,
// only when the step left partials (ctr->tne_pending).
__global__ void __launch_bounds__(256)
    finish_kernel(const double* __restrict__ partials, int nblocks, Record* hist, int hist_cap,
                  const DevCounters* ctr, Record* rec_out, double area)
{
    if (!rec_out && !ctr->tne_pending) return;
    __shared__ double wsum[8];
    const int q = blockIdx.x, t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int kind = tkind(q);
    double acc = kind == 0 ? 0.0 : (kind == 1 ? DBL_MAX : -DBL_MAX);
    const double* pq = partials + (size_t)q * nblocks;
    for (int b = t; b < nblocks; b += 256) acc = tcomb(kind, acc, __ldcg(pq + b));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc = tcomb(kind, acc, __shfl_xor_sync(0xffffffffu, acc, o));
    if (lane == 0) wsum[w] = acc;
    __syncthreads();
    if (t != 0) return;
    for (int k = 1; k < 8; k++) acc = tcomb(kind, acc, wsum[k]);
    Record* rec = rec_out ? rec_out : hist + (ctr->hist_count - 1) % hist_cap;
    if (q < TK) rec->sum[q + 4] = acc * area;
    else if (q < 2 * TK) rec->abs_sum[q - TK + 4] = acc * area;
    else if (q < 3 * TK) rec->min[q - 2 * TK + 4] = acc;
    else if (q < 4 * TK) rec->max[q - 3 * TK + 4] = acc;
    else if (q == 4 * TK) rec->d_sum = acc * area;
    else rec->d2_sum = acc * area;
    if (q == 0) {
        for (int k = 0; k < 4; k++) rec->sum[k] = rec->abs_sum[k] = rec->min[k] = rec->max[k] = 0.0;
        rec->step = rec_out ? ctr->step : ctr->tne_step;
    }
}

// The wall corrections of the edge rows (non-equilibrium extrapolation, Sec. IV.D):
// thread (side, x) forms rho, u, T of the edge cell in FP64 and
// M^-1 [f_hat^eq(rho, u_w, T_w) - f_hat^eq(rho, u, T)] in FP64, stored in R.
template <typename R>
__global__ void wall_kernel(const Model<R> K, const R* __restrict__ in, R* wall)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 2 * K.nx) return;
    const int side = t / K.nx, x = t % K.nx;
    if (K.sides[2 + side] != 2) return;
    double rho, ux, uy, T;
    conserved_at(K, in, x, side ? K.ny - 1 : 0, rho, ux, uy, &T);
    double qw[NV], qf[NV];
    feq24<double>(K.I, K.DI, rho, K.wux[side], K.wuy[side], K.wT[side], qw);
    feq24<double>(K.I, K.DI, rho, ux, uy, T, qf);
#pragma unroll 4
    for (int i = 0; i < NV; i++) {
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < NV; k++) acc = fma(K.Minvd[i * NV + k], qw[k] - qf[k], acc);
        wall[((size_t)side * NV + i) * K.nx + x] = (R)acc;
    }
}

// f = M^-1 f_hat^eq in block form, FP64 (162 multiply-adds of the transform, not 576)
template <typename R>
__global__ void init_kernel(const __grid_constant__ Model<double> K, const double* rho, const double* ux,
                            const double* uy, const double* T, const double* lam, R* state)
{
    const int64_t n = (int64_t)K.nx * K.ny;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n;
         c += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(c % K.nx), y = (int)(c / K.nx);
        const double t = T[c];
        const Eq24<double> e = eq24(K, rho[c], ux[c], uy[c], t);
        double w[NV], f[NV];
#pragma unroll
        for (int p = 0; p < NV; p++) w[p] = eq_moment(K, e, mom_of(p));
        inverse24<false>(K, w, f);
        const size_t g = (size_t)y * K.pitch + x;
#pragma unroll
        for (int i = 0; i < NV; i++) state[(size_t)i * K.plane + g] = (R)f[i];
        state[(size_t)NV * K.plane + g] = lam ? (R)lam[c] : R(0);
    }
}

template <typename R>
__global__ void macros_kernel(const Model<R> K, const R* __restrict__ in, double* rho,
                              double* ux, double* uy, double* T, double* p, double* lam)
{
    const int64_t n = (int64_t)K.nx * K.ny;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n;
         c += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(c % K.nx), y = (int)(c / K.nx);
        double r, u, v, t;
        conserved_at(K, in, x, y, r, u, v, &t);
        if (rho) rho[c] = r;
        if (ux) ux[c] = u;
        if (uy) uy[c] = v;
        if (T) T[c] = t;
        if (p) p[c] = r * t;
        if (lam) lam[c] = (double)in[(size_t)NV * K.plane + (size_t)y * K.pitch + x];
    }
}

// ---------------------------------------------------------------- host side

// velocities of the paper's D2V24 (Eqs. (25)-(27))
void velocity_table(const double v[3], const double eta[3], double* vx, double* vy, double* e)
{
    static const int AX[4][2] = {{1, 0}, {0, 1}, {-1, 0}, {0, -1}};
    static const int DG[4][2] = {{1, 1}, {-1, 1}, {-1, -1}, {1, -1}};
    for (int g = 0; g < 3; g++)
        for (int o = 0; o < 2; o++)
            for (int j = 0; j < 4; j++) {
                const int i = 8 * g + 4 * o + j;
                vx[i] = v[g] * (o == 0 ? AX[j][0] : DG[j][0]);
                vy[i] = v[g] * (o == 0 ? AX[j][1] : DG[j][1]);
                e[i] = eta[g];
            }
}

// rows m_1..m_24 (list after Eq. (16)) at the discrete velocities
void moment_rows(const double* vx, const double* vy, const double* e, double* M)
{
    for (int i = 0; i < NV; i++) {
        const double a = vx[i], b = vy[i], e2 = e[i] * e[i], v2 = a * a + b * b, w = v2 + e2;
        const double col[NV] = {1.0,       a,         b,         w,         a * a,
                                a * b,     b * b,     w * a,     w * b,     a * a * a,
                                a * a * b, a * b * b, b * b * b, w * a * a, w * a * b,
                                w * b * b, e2 * a * a, e2 * a * b, e2 * b * b, w * e2,
                                w * v2 * a, w * v2 * b, w * e2 * a, w * e2 * b};
        for (int k = 0; k < NV; k++) M[k * NV + i] = col[k];
    }
}

// The inverse of an n x n matrix (n <= 24) by LU factorisation with partial pivoting
// in long double, one step of iterative refinement per column. Returns max |A Ainv - 1|,
// or -1 if singular.
double invert(const double* M, double* Minv, int n = NV)
{
    long double lu[NV][NV];
    int perm[NV];
    long double amax = 0;
    for (int r = 0; r < n; r++) {
        perm[r] = r;
        for (int c = 0; c < n; c++) {
            lu[r][c] = M[r * n + c];
            amax = fmaxl(amax, fabsl(lu[r][c]));
        }
    }
    for (int k = 0; k < n; k++) {
        int p = k;
        for (int r = k + 1; r < n; r++)
            if (fabsl(lu[r][k]) > fabsl(lu[p][k])) p = r;
        if (fabsl(lu[p][k]) < 1e-13L * amax) return -1.0;
        if (p != k) {
            for (int c = 0; c < n; c++) {
                long double t = lu[k][c];
                lu[k][c] = lu[p][c];
                lu[p][c] = t;
            }
            int t = perm[k];
            perm[k] = perm[p];
            perm[p] = t;
        }
        for (int r = k + 1; r < n; r++) {
            lu[r][k] /= lu[k][k];
            for (int c = k + 1; c < n; c++) lu[r][c] -= lu[r][k] * lu[k][c];
        }
    }
    auto solve = [&](const long double* rhs, long double* x) {
        long double z[NV];
        for (int r = 0; r < n; r++) {
            long double s = rhs[perm[r]];
            for (int c = 0; c < r; c++) s -= lu[r][c] * z[c];
            z[r] = s;
        }
        for (int r = n - 1; r >= 0; r--) {
            long double s = z[r];
            for (int c = r + 1; c < n; c++) s -= lu[r][c] * x[c];
            x[r] = s / lu[r][r];
        }
    };
    for (int col = 0; col < n; col++) {
        long double e[NV], x[NV], res[NV], dx[NV];
        for (int r = 0; r < n; r++) e[r] = r == col ? 1.0L : 0.0L;
        solve(e, x);
        for (int r = 0; r < n; r++) {
            long double s = e[r];
            for (int c = 0; c < n; c++) s -= (long double)M[r * n + c] * x[c];
            res[r] = s;
        }
        solve(res, dx);
        for (int r = 0; r < n; r++) Minv[r * n + col] = (double)(x[r] + dx[r]);
    }
    double worst = 0.0;
    for (int r = 0; r < n; r++)
        for (int c = 0; c < n; c++) {
            long double s = 0;
            for (int k = 0; k < n; k++) s += (long double)M[r * n + k] * Minv[k * n + c];
            worst = fmax(worst, fabs((double)(s - (r == c ? 1.0L : 0.0L))));
        }
    return worst;
}

// The sector blocks of M (column j of a sector = M applied to the inverse butterfly of
// that sector's j-th unit component, restricted to the sector's moments) and their
// inverses. Returns the largest |entry| M produces outside the blocks relative to the
// largest inside, or -1 if a block is singular.
double build_blocks(const double* M, double* Bf, double* Bi)
{
    double leak = 0.0, big = 0.0;
    for (int sct = 0; sct < NSEC; sct++) {
        const int n = sec_n(sct), p0 = sec_p(sct);
        double blk[NV * NV], inv[NV * NV];
        for (int j = 0; j < n; j++) {
            double gv[NV] = {0}, f[NV], col[NV];
            gv[p0 + j] = 1.0;
            unbutterfly(gv, f);
            for (int k = 0; k < NV; k++) {
                col[k] = 0.0;
                for (int i = 0; i < NV; i++) col[k] += M[k * NV + i] * f[i];
            }
            for (int p = 0; p < NV; p++) {
                const bool inside = p >= p0 && p < p0 + n;
                if (inside) {
                    blk[(p - p0) * n + j] = col[mom_of(p)];
                    big = fmax(big, fabs(col[mom_of(p)]));
                } else {
                    leak = fmax(leak, fabs(col[mom_of(p)]));
                }
            }
        }
        const double res = invert(blk, inv, n);
        if (res < 0.0 || res > 1e-9) return -1.0;
        for (int k = 0; k < n * n; k++) {
            Bf[sec_b(sct) + k] = blk[k];
            Bi[sec_b(sct) + k] = inv[k];
        }
    }
    return leak / big;
}

template <typename R>
void fill_model(const lbkm24_params& p, const double* Bf, const double* Bi, const double* Minv,
                const double* vx, const double* vy, const double* e, int pitch,
                const int* sbc, const double (*sfeq)[NP], Model<R>* K)
{
    memset(K, 0, sizeof(*K));
    for (int sd = 0; sd < 4; sd++) {
        const int dir = sd < 2 ? p.bc_x : p.bc_y;
        K->sides[sd] = dir == LBKM_BC_SIDES ? sbc[sd] : dir;
        for (int i = 0; i < NP; i++) K->sfeq[sd][i] = (R)sfeq[sd][i];
    }
    for (int sct = 0; sct < NSEC; sct++)
        for (int r = 0; r < sec_n(sct); r++) {
            // orbit parity of component r: ee (sx, sy, e) per group, oe and eo one per orbit
            const bool diag = sct == 0 ? r % 3 == 2 : (sct == 3 ? true : r & 1);
            for (int j = 0; j < sec_n(sct); j++) {
                const int k = sec_b(sct) + r * sec_n(sct) + j;
                K->Bis[k] = (R)(Bi[k] * (diag ? 0.25 : 0.5));
            }
        }
    for (int k = 0; k < NB; k++) {
        K->Bf[k] = (R)Bf[k];
        K->Bi[k] = (R)Bi[k];
    }
    for (int k = 0; k < NV * NV; k++) K->Minvd[k] = Minv[k];
    for (int i = 0; i < NV; i++) {
        K->vx[i] = (R)vx[i];
        K->vy[i] = (R)vy[i];
        K->eta2[i] = (R)(e[i] * e[i]);
        K->S[i] = (R)p.S[i];
        K->vxd[i] = vx[i];
        K->vyd[i] = vy[i];
        K->wd[i] = vx[i] * vx[i] + vy[i] * vy[i] + e[i] * e[i];
    }
    for (int o = 0; o < 6; o++) {
        const double c = p.v[o / 2], et = p.eta[o / 2];
        K->cd[o] = c;
        K->wod[o] = c * c * ((o & 1) ? 2.0 : 1.0) + et * et;
        K->cdh[o] = (float)c;
        K->cdl[o] = (float)(c - (double)K->cdh[o]);
        K->wdh[o] = (float)K->wod[o];
        K->wdl[o] = (float)(K->wod[o] - (double)K->wdh[o]);
    }
    K->I = 2.0 / (p.gamma - 1.0) - 2.0;
    K->DI = 2.0 + K->I;
    K->kchem = p.Q / (p.dt * K->I * K->DI);
    K->inv_DI_r = (R)(1.0 / K->DI);
    for (int o = 0; o < 6; o++) {
        const double c = p.v[o / 2], et = p.eta[o / 2];
        K->c_r[o] = (R)c;
        K->chem_o[o] = (R)(K->I * c * c * ((o & 1) ? 2.0 : 1.0) + et * et);
    }
    K->inv_DI = 1.0 / K->DI;
    K->Q = p.Q;
    K->omega1 = p.omega1;
    K->omega2 = p.omega2;
    K->T_ig = p.T_ig;
    K->A8c = (p.S[4] - p.S[7]) / p.S[4];
    K->A9c = (p.S[6] - p.S[8]) / p.S[6];
    K->dt = p.dt;
    K->inv_dx = 1.0 / p.dx;
    K->inv_dy = 1.0 / p.dy;
    for (int i = 0; i < NV; i++) {
        K->vxs[i] = (R)(vx[i] / p.dx);
        K->vys[i] = (R)(vy[i] / p.dy);
    }
    K->dt_r = (R)p.dt;
    K->inv_dx_r = (R)(1.0 / p.dx);
    K->inv_dy_r = (R)(1.0 / p.dy);
    K->hdx_r = (R)(0.5 / p.dx);
    K->hdy_r = (R)(0.5 / p.dy);
    K->I_r = (R)K->I;
    K->DI_r = (R)K->DI;
    K->A8c_r = (R)K->A8c;
    K->A9c_r = (R)K->A9c;
    K->nx = p.nx;
    K->ny = p.ny;
    K->pitch = pitch;
    K->bc_x = p.bc_x;
    K->bc_y = p.bc_y;
    K->plane = (int64_t)pitch * p.ny;
}

thread_local std::string g_create_error;

} // namespace v24

using namespace v24;

struct lbkm24 {
    lbkm24_params p;
    Model<double> Kd;
    Model<float> Kf;
    int pitch;
    size_t elem, plane_elems;
    cudaStream_t stream, capture_stream;
    void* buf[2];
    int cur;
    double* partials;
    int nblocks;       // of tne_kernel
    dim3 grid, block;
    int sblocks;       // of a step
    int split;         // > 0: steps per launch of split_kernel (short FP64 1-D grids)
    DevCounters* ctr;
    Record* hist;
    Record* tne_out;
    bool initialized;
    bool srt;  // the single-relaxation-time fast path runs the steps
    bool has_wall;
    void* wallbuf;  // [2][24][nx] wall corrections in the state's precision
    int64_t host_steps;
    cudaGraphExec_t graph[2];
    std::string err;
};

namespace {

lbkm_status fail(lbkm24_t h, lbkm_status st, const char* fmt, ...)
{
    char b[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(b, sizeof(b), fmt, ap);
    va_end(ap);
    (h ? h->err : g_create_error) = b;
    return st;
}

#define TRY24(h, call)                                                                        \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess)                                                                \
            return fail((h), e_ == cudaErrorMemoryAllocation ? LBKM_ENOMEM : LBKM_ECUDA,      \
                        "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
    } while (0)

// one step from buf[from], or up to h->split steps in one launch of split_kernel: n comes in as
// the steps wanted and goes out as the steps launched
cudaError_t launch_steps(const lbkm24* h, int from, int64_t& n, cudaStream_t st)
{
    Args a;
    a.in = h->buf[from];
    a.out = h->buf[1 - from];
    a.partials = h->partials;
    a.ctr = h->ctr;
    a.hist = h->hist;
    a.hist_cap = h->p.tne_capacity;
    a.tne_every = h->p.tne_every;
    a.area = h->p.dx * h->p.dy;
    if (h->split) {
        if (n > h->split) n = h->split;
        const int own = 32 - 4 * h->split;
        split_kernel<<<(h->p.nx + own - 1) / own, 128, 0, st>>>(h->Kd, a, (int)n, h->split);
        return cudaGetLastError();
    }
    n = 1;
    if (h->has_wall) {
        const int g = (2 * h->p.nx + 127) / 128;
        if (h->p.precision == LBKM_F64)
            wall_kernel<double><<<g, 128, 0, st>>>(h->Kd, (const double*)a.in, (double*)h->wallbuf);
        else
            wall_kernel<float><<<g, 128, 0, st>>>(h->Kf, (const float*)a.in, (float*)h->wallbuf);
        const cudaError_t we = cudaGetLastError();
        if (we != cudaSuccess) return we;
    }
    const bool f64 = h->p.precision == LBKM_F64;
#define V24_LAUNCH(R_, SRT_, D2_, TNE_) \
    step_launch<R_, SRT_, D2_, TNE_>(*static_cast<const Model<R_>*>(f64 ? (const void*)&h->Kd : &h->Kf), a, h->sblocks, st)
    cudaError_t e = V24_VARIANT(V24_LAUNCH, f64, h->srt, h->p.ny > 1, h->p.tne_every > 0);
#undef V24_LAUNCH
    if (e == cudaSuccess && h->p.tne_every > 0) {
        finish_kernel<<<NQ, 256, 0, st>>>(h->partials, h->sblocks, h->hist, h->p.tne_capacity,
                                          h->ctr, nullptr, a.area);
        e = cudaGetLastError();
    }
    return e;
}

// Steps per launch of split_kernel, or 0 where it does not apply: FP64, 1-D, moment form, no
// records, and at most three windows an SM (a window's four warps use all of an SM's FP64 unit,
// step_kernel's one warp a quarter). us per step, this against step_kernel: 5000 and 8400 cells, two
// windows on some or all SMs, 21.6 and 37; 9000 to 12700 cells, three, 24 to 28.1 and 37.
int split_steps_for(const lbkm24* h, int sms)
{
    if (h->p.precision != LBKM_F64 || h->p.ny != 1 || h->srt || h->p.tne_every > 0) return 0;
    const int nx = h->p.nx;
    for (int k = 4; k >= 1; k /= 2)
        if ((nx + 31 - 4 * k) / (32 - 4 * k) <= sms) return k;
    return (nx + 27) / 28 <= 3 * sms ? 1 : 0;
}

// streaming multiprocessors of the current device (152 on GB300, the value taken if the
// query fails)
int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        sms < 1) {
        cudaGetLastError();
        return 152;
    }
    return sms;
}

int elementwise_blocks(int64_t n)
{
    const int64_t b = (n + 255) / 256, cap = (int64_t)sm_count() * 16;
    return (int)(b < cap ? (b < 1 ? 1 : b) : cap);
}

lbkm_status check(lbkm24_t h)
{
    TRY24(h, cudaStreamSynchronize(h->stream));
    int st = 0;
    TRY24(h, cudaMemcpy(&st, &h->ctr->status, sizeof(int), cudaMemcpyDeviceToHost));
    if (st & 1)
        return fail(h, LBKM_EUNSTABLE,
                    "a cell reached a non-finite or non-positive density or temperature");
    return LBKM_OK;
}

void to_global(const Record& r, lbkm24_tne_global* g) { memcpy(g, &r, sizeof(r)); }

} // namespace

extern "C" {

void lbkm24_default_params(lbkm24_params* p)
{
    if (!p) return;
    memset(p, 0, sizeof(*p));
    p->precision = LBKM_F64;
    p->gamma = 1.4;
    p->v[0] = 2.7;
    p->v[1] = 2.2;
    p->v[2] = 1.2;
    p->eta[0] = 5.0;
    p->eta[1] = 3.0;
    p->eta[2] = 1.1;
    for (int k = 0; k < NV; k++) p->S[k] = (k >= 4 && k <= 6) ? 1e4 : 1e5;
    p->Q = 1.0;
    p->T_ig = 1.1;
    p->dx = p->dy = 2e-4;
    p->dt = 5e-6;
    p->bc_x = LBKM_BC_ZERO_GRADIENT;
    p->bc_y = LBKM_BC_PERIODIC;
    p->tne_capacity = 1;
}

const char* lbkm24_last_error(lbkm24_t h) { return h ? h->err.c_str() : g_create_error.c_str(); }

lbkm_status lbkm24_create(const lbkm24_params* pin, void* cuda_stream, lbkm24_t* out)
{
    if (!out) return fail(nullptr, LBKM_EINVAL, "out is NULL");
    *out = nullptr;
    if (!pin) return fail(nullptr, LBKM_EINVAL, "params is NULL");
    const lbkm24_params& p = *pin;
    if (p.nx < 1 || p.ny < 1 || (int64_t)p.nx * p.ny > (int64_t)1 << 30)
        return fail(nullptr, LBKM_EINVAL, "nx, ny must be >= 1 (at most 2^30 cells)");
    if (p.precision != LBKM_F64 && p.precision != LBKM_F32)
        return fail(nullptr, LBKM_EINVAL, "precision must be LBKM_F64 or LBKM_F32");
    if (!(p.gamma > 1.0) || !(2.0 / (p.gamma - 1.0) - 2.0 > 0.0))
        return fail(nullptr, LBKM_EINVAL, "gamma must give I = 2/(gamma-1) - 2 > 0");
    for (int g = 0; g < 3; g++) {
        if (!(p.v[g] > 0.0) || !isfinite(p.v[g]))
            return fail(nullptr, LBKM_EINVAL, "v[%d] must be finite and > 0", g);
        if (!(p.eta[g] >= 0.0) || !isfinite(p.eta[g]))
            return fail(nullptr, LBKM_EINVAL, "eta[%d] must be finite and >= 0", g);
    }
    double smax = 0.0;
    for (int k = 4; k < NV; k++) {
        if (!(p.S[k] > 0.0) || !isfinite(p.S[k]))
            return fail(nullptr, LBKM_EINVAL, "S[%d] must be finite and > 0", k);
        smax = fmax(smax, p.S[k]);
    }
    if (!(p.dx > 0) || !(p.dy > 0) || !(p.dt > 0))
        return fail(nullptr, LBKM_EINVAL, "dx, dy, dt must be > 0");
    if (!(p.dt * smax < 2.0))
        return fail(nullptr, LBKM_EINVAL, "dt * max S = %g must be < 2", p.dt * smax);
    const double vmax = fmax(p.v[0], fmax(p.v[1], p.v[2])); // per-axis component of the diagonals
    const double cfl = vmax * p.dt * (1.0 / p.dx + (p.ny > 1 ? 1.0 / p.dy : 0.0));
    if (!(cfl <= 1.0))
        return fail(nullptr, LBKM_EINVAL, "CFL number %g of the fastest velocity exceeds 1", cfl);
    if (!(p.omega1 >= 0) || !(p.omega2 >= 0) || !isfinite(p.Q))
        return fail(nullptr, LBKM_EINVAL, "omega1, omega2 must be >= 0 and Q finite");
    if (!(p.T_ig >= 0) || !isfinite(p.T_ig))
        return fail(nullptr, LBKM_EINVAL, "T_ig must be finite and >= 0");
    for (int d = 0; d < 2; d++) {
        const int bc = d == 0 ? p.bc_x : p.bc_y;
        if (bc != LBKM_BC_PERIODIC && bc != LBKM_BC_ZERO_GRADIENT && bc != LBKM_BC_SIDES)
            return fail(nullptr, LBKM_EINVAL, "%s must be periodic, zero gradient or sides",
                        d == 0 ? "bc_x" : "bc_y");
    }
    for (int sd = 0; sd < 4; sd++) {
        if ((sd < 2 ? p.bc_x : p.bc_y) != LBKM_BC_SIDES) continue;
        const int code = p.side_bc[sd];
        const bool ok = code == LBKM_BC_ZERO_GRADIENT || code == LBKM_BC_DIRICHLET ||
                        ((code == LBKM_BC_SPECULAR || code == LBKM_BC_WALL) && sd >= 2);
        if (!ok)
            return fail(nullptr, LBKM_EINVAL,
                        "side_bc[%d]: zero gradient, Dirichlet, or specular / wall (y sides only)",
                        sd);
        if ((code == LBKM_BC_SPECULAR || code == LBKM_BC_WALL) && p.ny < 2)
            return fail(nullptr, LBKM_EINVAL, "a specular or wall side needs ny >= 2");
        if (code == LBKM_BC_WALL &&
            (!(p.side_T[sd] > 0) || !isfinite(p.side_T[sd]) || !isfinite(p.side_ux[sd]) ||
             !isfinite(p.side_uy[sd])))
            return fail(nullptr, LBKM_EINVAL, "side %d: a wall needs T > 0 and a finite velocity",
                        sd);
        if (code == LBKM_BC_DIRICHLET &&
            (!(p.side_rho[sd] > 0) || !(p.side_T[sd] > 0) || !isfinite(p.side_rho[sd]) ||
             !isfinite(p.side_T[sd]) || !isfinite(p.side_ux[sd]) || !isfinite(p.side_uy[sd]) ||
             !(p.side_lam[sd] >= 0 && p.side_lam[sd] <= 1)))
            return fail(nullptr, LBKM_EINVAL,
                        "side %d: Dirichlet state needs rho > 0, T > 0, finite u, lambda in [0, 1]",
                        sd);
    }
    if (p.tne_every < 0 || (p.tne_every > 0 && p.tne_capacity < 1))
        return fail(nullptr, LBKM_EINVAL, "tne_every >= 0 and tne_capacity >= 1");
    if (p.collision != 0 && p.collision != 1)
        return fail(nullptr, LBKM_EINVAL, "collision must be 0 (fast path allowed) or 1");

    double vx[NV], vy[NV], e[NV], M[NV * NV], Minv[NV * NV], Bf[NB], Bi[NB];
    velocity_table(p.v, p.eta, vx, vy, e);
    moment_rows(vx, vy, e, M);
    const double res = invert(M, Minv);
    const double leak = res < 0.0 ? -1.0 : build_blocks(M, Bf, Bi);
    if (res < 0.0 || res > 1e-9 || leak < 0.0)
        return fail(nullptr, LBKM_ESINGULAR, "the D2V24 velocity set gives a singular M");
    if (leak > 1e-12)
        return fail(nullptr, LBKM_ESINGULAR, "M is not block-diagonal under the butterflies");

    lbkm24* h = new lbkm24();
    h->p = p;
    if (h->p.tne_capacity < 1) h->p.tne_capacity = 1;
    h->stream = (cudaStream_t)cuda_stream;
    h->elem = p.precision == LBKM_F64 ? 8 : 4;
    h->pitch = (p.nx + 31) / 32 * 32;
    h->plane_elems = (size_t)h->pitch * p.ny;
    bool equal = true;
    for (int k = 5; k < NV; k++) equal = equal && p.S[k] == p.S[4];
    h->srt = equal && p.tne_every == 0 && p.collision == 0;
    // Dirichlet sides: ghost f = M^-1 f_hat^eq(side state), ghost lambda = the side's
    int sbc[4] = {0, 0, 0, 0};
    double sfeq[4][NP];
    memset(sfeq, 0, sizeof(sfeq));
    const double Ih = 2.0 / (p.gamma - 1.0) - 2.0;
    for (int sd = 0; sd < 4; sd++) {
        if ((sd < 2 ? p.bc_x : p.bc_y) != LBKM_BC_SIDES) continue;
        sbc[sd] = p.side_bc[sd];
        if (sbc[sd] != LBKM_BC_DIRICHLET) continue;
        double q[NV];
        feq24<double>(Ih, 2.0 + Ih, p.side_rho[sd], p.side_ux[sd], p.side_uy[sd], p.side_T[sd], q);
        for (int i = 0; i < NV; i++) {
            double acc = 0.0;
            for (int k = 0; k < NV; k++) acc += Minv[i * NV + k] * q[k];
            sfeq[sd][i] = acc;
        }
        sfeq[sd][NV] = p.side_lam[sd];
    }
    fill_model(p, Bf, Bi, Minv, vx, vy, e, h->pitch, sbc, sfeq, &h->Kd);
    fill_model(p, Bf, Bi, Minv, vx, vy, e, h->pitch, sbc, sfeq, &h->Kf);
    h->has_wall = p.bc_y == LBKM_BC_SIDES && (sbc[2] == LBKM_BC_WALL || sbc[3] == LBKM_BC_WALL);
    for (int w = 0; w < 2; w++) {
        h->Kd.wux[w] = h->Kf.wux[w] = p.side_ux[2 + w];
        h->Kd.wuy[w] = h->Kf.wuy[w] = p.side_uy[2 + w];
        h->Kd.wT[w] = h->Kf.wT[w] = p.side_T[2 + w];
    }
    // (the TNE of a state on demand: short 1-D grids in blocks of one warp, for more SMs)
    const bool narrow = p.ny == 1 && (p.nx + BT - 1) / BT < 2 * sm_count();
    h->block = p.ny > 1 ? dim3(32, BT / 32) : dim3(narrow ? 32 : BT, 1);
    h->grid = dim3((p.nx + h->block.x - 1) / h->block.x, (p.ny + h->block.y - 1) / h->block.y);
    h->nblocks = (int)(h->grid.x * h->grid.y);
    auto bail = [&](cudaError_t ce, const char* what) {
        lbkm24_destroy(h);
        return fail(nullptr, ce == cudaErrorMemoryAllocation ? LBKM_ENOMEM : LBKM_ECUDA, "%s: %s",
                    what, cudaGetErrorString(ce));
    };
    cudaError_t ce;
    const int sms = sm_count();
#define V24_BLOCKS(R_, SRT_, D2_, TNE_) step_blocks<R_, SRT_, D2_, TNE_>(p.nx, p.ny, sms)
    h->sblocks = V24_VARIANT(V24_BLOCKS, p.precision == LBKM_F64, h->srt, p.ny > 1, p.tne_every > 0);
#undef V24_BLOCKS
    if (h->sblocks < 1) return bail(cudaGetLastError(), "step kernel");
    h->split = split_steps_for(h, sms);
    const size_t sb = (size_t)NP * h->plane_elems * h->elem;
    for (int k = 0; k < 2; k++)
        if ((ce = cudaMalloc(&h->buf[k], sb)) != cudaSuccess) return bail(ce, "state");
    if ((ce = cudaMalloc((void**)&h->partials, sizeof(double) * NQ * (h->nblocks > h->sblocks ? h->nblocks : h->sblocks))) !=
        cudaSuccess)
        return bail(ce, "partials");
    if (h->has_wall) {
        const size_t wb = sizeof(double) * 2 * NV * (size_t)p.nx;
        if ((ce = cudaMalloc(&h->wallbuf, wb)) != cudaSuccess) return bail(ce, "walls");
        if ((ce = cudaMemset(h->wallbuf, 0, wb)) != cudaSuccess) return bail(ce, "walls");
        h->Kd.wall = static_cast<const double*>(h->wallbuf);
        h->Kf.wall = static_cast<const float*>(h->wallbuf);
    }
    if ((ce = cudaMalloc((void**)&h->ctr, sizeof(DevCounters))) != cudaSuccess)
        return bail(ce, "counters");
    if ((ce = cudaMalloc((void**)&h->hist, sizeof(Record) * h->p.tne_capacity)) != cudaSuccess)
        return bail(ce, "history");
    if ((ce = cudaMalloc((void**)&h->tne_out, sizeof(Record))) != cudaSuccess)
        return bail(ce, "record");
    if ((ce = cudaStreamCreateWithFlags(&h->capture_stream, cudaStreamNonBlocking)) != cudaSuccess)
        return bail(ce, "capture stream");
    if ((ce = cudaMemset(h->buf[0], 0, sb)) != cudaSuccess ||
        (ce = cudaMemset(h->buf[1], 0, sb)) != cudaSuccess ||
        (ce = cudaMemset(h->ctr, 0, sizeof(DevCounters))) != cudaSuccess)
        return bail(ce, "clear");
    *out = h;
    return LBKM_OK;
}

void lbkm24_destroy(lbkm24_t h)
{
    if (!h) return;
    if (h->stream || h->buf[0]) cudaStreamSynchronize(h->stream);
    for (int i = 0; i < 2; i++) {
        if (h->graph[i]) cudaGraphExecDestroy(h->graph[i]);
        if (h->buf[i]) cudaFree(h->buf[i]);
    }
    if (h->capture_stream) cudaStreamDestroy(h->capture_stream);
    if (h->partials) cudaFree(h->partials);
    if (h->ctr) cudaFree(h->ctr);
    if (h->hist) cudaFree(h->hist);
    if (h->tne_out) cudaFree(h->tne_out);
    if (h->wallbuf) cudaFree(h->wallbuf);
    delete h;
}

lbkm_status lbkm24_init_fields(lbkm24_t h, const double* rho, const double* ux, const double* uy,
                               const double* T, const double* lambda, int on_device)
{
    if (!h) return LBKM_EINVAL;
    if (!rho || !ux || !uy || !T) return fail(h, LBKM_EINVAL, "rho, ux, uy and T are required");
    const size_t n = (size_t)h->p.nx * h->p.ny, nb = n * sizeof(double);
    const double* src[5] = {rho, ux, uy, T, lambda};
    const double* dev[5] = {rho, ux, uy, T, lambda};
    double* tmp = nullptr;
    if (!on_device) {
        TRY24(h, cudaMallocAsync((void**)&tmp, nb * 5, h->stream));
        for (int k = 0; k < 5; k++) {
            if (!src[k]) {
                dev[k] = nullptr;
                continue;
            }
            TRY24(h, cudaMemcpyAsync(tmp + k * n, src[k], nb, cudaMemcpyHostToDevice, h->stream));
            dev[k] = tmp + k * n;
        }
    }
    const int g = elementwise_blocks((int64_t)n);
    if (h->p.precision == LBKM_F64)
        init_kernel<double><<<g, 256, 0, h->stream>>>(h->Kd, dev[0], dev[1], dev[2], dev[3],
                                                      dev[4], (double*)h->buf[0]);
    else
        init_kernel<float><<<g, 256, 0, h->stream>>>(h->Kd, dev[0], dev[1], dev[2], dev[3],
                                                     dev[4], (float*)h->buf[0]);
    TRY24(h, cudaGetLastError());
    h->cur = 0;
    TRY24(h, cudaMemsetAsync(h->ctr, 0, sizeof(DevCounters), h->stream));
    if (tmp) TRY24(h, cudaFreeAsync(tmp, h->stream));
    TRY24(h, cudaStreamSynchronize(h->stream));
    h->initialized = true;
    h->host_steps = 0;
    return LBKM_OK;
}

lbkm_status lbkm24_step(lbkm24_t h, int64_t n)
{
    if (!h) return LBKM_EINVAL;
    if (!h->initialized) return fail(h, LBKM_ESTATE, "lbkm24_step before lbkm24_init_fields");
    if (n < 0) return fail(h, LBKM_EINVAL, "n must be >= 0");
    while (n >= GRAPH_CHUNK) {
        cudaGraphExec_t& ex = h->graph[h->cur];
        if (!ex) {
            cudaGraph_t gr;
            TRY24(h, cudaStreamBeginCapture(h->capture_stream, cudaStreamCaptureModeThreadLocal));
            cudaError_t le = cudaSuccess;
            int c = h->cur;
            for (int64_t left = GRAPH_CHUNK, m; left > 0 && le == cudaSuccess; left -= m, c = 1 - c) {
                m = left;
                le = launch_steps(h, c, m, h->capture_stream);
            }
            cudaError_t ce = cudaStreamEndCapture(h->capture_stream, &gr);
            if (le != cudaSuccess || ce != cudaSuccess) {
                if (ce == cudaSuccess) cudaGraphDestroy(gr);
                return fail(h, LBKM_ECUDA, "graph capture: %s",
                            cudaGetErrorString(le != cudaSuccess ? le : ce));
            }
            cudaError_t ie = cudaGraphInstantiate(&ex, gr, 0);
            cudaGraphDestroy(gr);
            if (ie != cudaSuccess)
                return fail(h, LBKM_ECUDA, "graph instantiate: %s", cudaGetErrorString(ie));
        }
        TRY24(h, cudaGraphLaunch(ex, h->stream));
        n -= GRAPH_CHUNK;
        h->host_steps += GRAPH_CHUNK;
    }
    while (n > 0) {
        int64_t m = n;
        TRY24(h, launch_steps(h, h->cur, m, h->stream));
        h->cur = 1 - h->cur;
        h->host_steps += m;
        n -= m;
    }
    return LBKM_OK;
}

lbkm_status lbkm24_sync(lbkm24_t h)
{
    if (!h) return LBKM_EINVAL;
    return check(h);
}

int64_t lbkm24_steps_taken(lbkm24_t h) { return h ? h->host_steps : -1; }

lbkm_status lbkm24_macros(lbkm24_t h, double* rho, double* ux, double* uy, double* T, double* p,
                          double* lambda, int on_device)
{
    if (!h) return LBKM_EINVAL;
    if (!h->initialized) return fail(h, LBKM_ESTATE, "lbkm24_macros before lbkm24_init_fields");
    const size_t n = (size_t)h->p.nx * h->p.ny, nb = n * sizeof(double);
    double* outs[6] = {rho, ux, uy, T, p, lambda};
    double* dev[6] = {rho, ux, uy, T, p, lambda};
    double* tmp = nullptr;
    if (!on_device) {
        TRY24(h, cudaMallocAsync((void**)&tmp, nb * 6, h->stream));
        for (int k = 0; k < 6; k++) dev[k] = outs[k] ? tmp + k * n : nullptr;
    }
    const int g = elementwise_blocks((int64_t)n);
    if (h->p.precision == LBKM_F64)
        macros_kernel<double><<<g, 256, 0, h->stream>>>(h->Kd, (const double*)h->buf[h->cur],
                                                        dev[0], dev[1], dev[2], dev[3], dev[4],
                                                        dev[5]);
    else
        macros_kernel<float><<<g, 256, 0, h->stream>>>(h->Kf, (const float*)h->buf[h->cur], dev[0],
                                                       dev[1], dev[2], dev[3], dev[4], dev[5]);
    TRY24(h, cudaGetLastError());
    if (!on_device) {
        for (int k = 0; k < 6; k++)
            if (outs[k])
                TRY24(h, cudaMemcpyAsync(outs[k], dev[k], nb, cudaMemcpyDeviceToHost, h->stream));
        TRY24(h, cudaFreeAsync(tmp, h->stream));
    }
    return check(h);
}

lbkm_status lbkm24_tne(lbkm24_t h, double* delta, lbkm24_tne_global* g, int on_device)
{
    if (!h) return LBKM_EINVAL;
    if (!h->initialized) return fail(h, LBKM_ESTATE, "lbkm24_tne before lbkm24_init_fields");
    const size_t n = (size_t)h->p.nx * h->p.ny, nb = (size_t)NV * n * sizeof(double);
    double* dd = delta;
    double* tmp = nullptr;
    if (delta && !on_device) {
        TRY24(h, cudaMallocAsync((void**)&tmp, nb, h->stream));
        dd = tmp;
    }
    if (h->p.precision == LBKM_F64)
        tne_kernel<double><<<h->grid, h->block, 0, h->stream>>>(
            h->Kd, (const double*)h->buf[h->cur], dd, h->partials);
    else
        tne_kernel<float><<<h->grid, h->block, 0, h->stream>>>(
            h->Kf, (const float*)h->buf[h->cur], dd, h->partials);
    TRY24(h, cudaGetLastError());
    finish_kernel<<<NQ, 256, 0, h->stream>>>(h->partials, h->nblocks, nullptr, 1, h->ctr,
                                             h->tne_out, h->p.dx * h->p.dy);
    TRY24(h, cudaGetLastError());
    if (tmp) {
        TRY24(h, cudaMemcpyAsync(delta, tmp, nb, cudaMemcpyDeviceToHost, h->stream));
        TRY24(h, cudaFreeAsync(tmp, h->stream));
    }
    Record r;
    TRY24(h, cudaMemcpyAsync(&r, h->tne_out, sizeof(r), cudaMemcpyDeviceToHost, h->stream));
    lbkm_status st = check(h);
    if (st != LBKM_OK) return st;
    if (g) to_global(r, g);
    return LBKM_OK;
}

lbkm_status lbkm24_tne_history(lbkm24_t h, lbkm24_tne_global* out, int32_t max_records,
                               int32_t* n_out)
{
    if (!h || !n_out || (max_records > 0 && !out)) return LBKM_EINVAL;
    *n_out = 0;
    lbkm_status st = check(h);
    if (st != LBKM_OK) return st;
    DevCounters c;
    TRY24(h, cudaMemcpy(&c, h->ctr, sizeof(c), cudaMemcpyDeviceToHost));
    const int cap = h->p.tne_capacity;
    const int64_t have = c.hist_count < cap ? c.hist_count : cap;
    const int64_t take = have < max_records ? have : max_records;
    for (int64_t k = 0; k < take; k++) {
        Record r;
        TRY24(h, cudaMemcpy(&r, h->hist + (c.hist_count - have + k) % cap, sizeof(r),
                            cudaMemcpyDeviceToHost));
        to_global(r, out + k);
    }
    *n_out = (int32_t)take;
    return LBKM_OK;
}

size_t lbkm24_state_bytes(lbkm24_t h)
{
    return h ? (size_t)NP * h->p.nx * h->p.ny * h->elem + sizeof(int64_t) : 0;
}

lbkm_status lbkm24_get_state(lbkm24_t h, void* dst, int on_device)
{
    if (!h || !dst) return LBKM_EINVAL;
    if (!h->initialized) return fail(h, LBKM_ESTATE, "lbkm24_get_state before init_fields");
    const size_t row = (size_t)h->p.nx * h->elem, plane = row * h->p.ny;
    if (on_device && lbk::can_pack((int)h->elem, h->buf[h->cur], dst)) {
        TRY24(h, lbk::launch_pack((int)h->elem, NP, h->buf[h->cur], (int64_t)h->plane_elems, h->pitch, h->p.nx,
                                  h->p.ny, dst, h->host_steps, h->stream));
        return check(h);
    }
    const cudaMemcpyKind k = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    for (int pl = 0; pl < NP; pl++)
        TRY24(h, cudaMemcpy2DAsync((char*)dst + pl * plane, row,
                                   (const char*)h->buf[h->cur] + pl * h->plane_elems * h->elem,
                                   h->pitch * h->elem, row, h->p.ny, k, h->stream));
    const int64_t s = h->host_steps;
    TRY24(h, cudaMemcpyAsync((char*)dst + NP * plane, &s, sizeof(s),
                             on_device ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost,
                             h->stream));
    return check(h);
}

lbkm_status lbkm24_set_state(lbkm24_t h, const void* src, int on_device)
{
    if (!h || !src) return LBKM_EINVAL;
    const size_t row = (size_t)h->p.nx * h->elem, plane = row * h->p.ny;
    const cudaMemcpyKind k = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    h->cur = 0;
    for (int pl = 0; pl < NP; pl++)
        TRY24(h, cudaMemcpy2DAsync((char*)h->buf[0] + pl * h->plane_elems * h->elem,
                                   h->pitch * h->elem, (const char*)src + pl * plane, row, row,
                                   h->p.ny, k, h->stream));
    int64_t s = 0;
    TRY24(h, cudaMemcpyAsync(&s, (const char*)src + NP * plane, sizeof(s),
                             on_device ? cudaMemcpyDeviceToHost : cudaMemcpyHostToHost,
                             h->stream));
    TRY24(h, cudaStreamSynchronize(h->stream));
    DevCounters c;
    memset(&c, 0, sizeof(c));
    c.step = s;
    TRY24(h, cudaMemcpy(h->ctr, &c, sizeof(c), cudaMemcpyHostToDevice));
    h->host_steps = s;
    h->initialized = true;
    return LBKM_OK;
}

} // extern "C"
