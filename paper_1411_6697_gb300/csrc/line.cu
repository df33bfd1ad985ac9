// line.cu -- the 1-D step (Ny = 1), FP64 and FP32: several time steps in one launch.
//
// A block holds a window of `threads` cells, one per thread, and carries them through
// `nsteps` time steps in registers; neighbours meet in shared memory once per step. A
// step reaches two cells to each side, so of a window only the cells 2 nsteps away from
// its ends are right after nsteps: those are the block's own, the rest overlaps with the
// neighbour blocks' windows. No block waits for another, and the state passes through
// memory once per launch instead of once per step.
//
// What bounds it. FP64: the FP64 unit. One FP64 warp instruction (add, multiply, FMA or
// compare alike) holds its quarter of the SM for 64 cycles whatever its lanes do, so the
// time of a step is the number of FP64 instructions of one warp times 64..76 cycles, and
// everything that can leave that unit does: minmod, comparisons and clamps work on the bit
// patterns (integer pipe), each difference of neighbouring cells is formed once and
// exchanged, the factor 1/2 of four moments is folded into the matrix, f_hat^eq enters
// Delta_k as the product of an FMA, the reciprocal is an FP32 seed with one third-order
// correction, and the terms of the reaction and of A_hat are left out of warps and models
// where they vanish: 298 FP64 instructions per warp and step (ncu, 16384-cell detonation). FP32:
// the latency of one warp's chain of about 900 instructions; the conserved sums are exact
// double-floats, which keeps all but 14 FP64 instructions off that unit.
//
// Measured per step, against one launch per step of a tile kernel with the plain formulas
// (every stencil's differences, FP64 minmod and FP64 sums of an FP32 state): Sod tube of 400
// cells FP64 29.8 -> 11.7 us; detonation of 16384 cells FP32 13.3 -> 2.1 us, FP64 with records
// at every step 58.9 -> 24.9 us.
//
// Boundaries: lanes past a zero-gradient end are read through the index of the end cell,
// lanes past a Dirichlet end hold the side's equilibrium, and on a periodic grid every lane
// stands for the cell its position wraps to.
#include <float.h>

#include "cell.cuh"
#include "line.cuh"
#include "pair.cuh"
#include "reduce.cuh"

namespace lbk {

namespace {

constexpr int NMOVE = 12;          // planes with v_x != 0
constexpr int NX = NMOVE + 1;      // and lambda: what neighbours read
constexpr int LINE_THREADS = 256;      // threads of a block

// plane of slot s: v_x > 0 in the first six, v_x < 0 in the next six, then lambda
__host__ __device__ constexpr int slot_plane(int s)
{
    constexpr int t[NX] = {0, 4, 7, 8, 12, 15, 2, 5, 6, 10, 13, 14, 16};
    return t[s];
}
__host__ __device__ constexpr int slot_of(int plane) // -1: v_x = 0
{
    constexpr int t[16] = {0, -1, 6, -1, 1, 7, 8, 2, 3, -1, 9, -1, 4, 10, 11, 5};
    return t[plane];
}

template <typename R>
struct LineConst {
    R h2[4], h3[4], ha[4]; // rows of the ES and EA blocks of m_5, m_7, m_14, m_16, halved
    R c8x, c8y, c9x, c9y;  // A_hat_8, A_hat_9 = rho T (c.x u du_x + c.y u' du_y), raw differences
    R cdx[4], dtdx;        // c / dx (FP32: dt c / dx) of each orbit, dt / dx
    R di2;                 // D + I + 2
    int a_hat;             // A_hat does not vanish
};

// ---- FP64 values as bit patterns (integer pipe) ---------------------------------
__device__ __forceinline__ double mm64(double a, double b)
{
    const unsigned long long ia = (unsigned long long)__double_as_longlong(a);
    const unsigned long long ib = (unsigned long long)__double_as_longlong(b);
    const unsigned long long m = 0x7fffffffffffffffull;
    const unsigned long long r = (ia & m) <= (ib & m) ? ia : ib;
    return __longlong_as_double((long long)((long long)(ia ^ ib) < 0 ? 0ull : r));
}
__device__ __forceinline__ long long order64(double x) // monotonic in x
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double unorder64(long long k)
{
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
}
// 1/x: FP32 estimate (22 bits), then q + q (e + e^2), e = 1 - x q
__device__ __forceinline__ double recip64(double x)
{
    const double q = f2d_fast(rcp_approx(d2f_fast(x)));
    const double e = __fma_rn(-x, q, 1.0);
    return __fma_rn(q, __fma_rn(e, e, e), q);
}

// Rounded operations that the compiler must not merge: every path through the step then
// rounds alike, whichever instantiation (with records or without) it runs in.
__device__ __forceinline__ double fm(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fm(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mu(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mu(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double ad(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float ad(float a, float b) { return __fadd_rn(a, b); }

__device__ __forceinline__ bool negative(double x) { return dbits(x) < 0; }
__device__ __forceinline__ bool negative(float x) { return x < 0.f; }
// x clamped to [0, 1]; NaN stays
__device__ __forceinline__ double clamp01(double x)
{
    const long long b = dbits(x), inf = 0x7ff0000000000000ll;
    if ((b & 0x7fffffffffffffffll) > inf) return x;
    return b < 0 ? 0.0 : (b > dbits(1.0) ? 1.0 : x);
}
__device__ __forceinline__ float clamp01(float x) { return x < 0.f ? 0.f : (x > 1.f ? 1.f : x); }

// The orbit butterflies of one cell (sums and differences that all its moments share).
template <typename R>
struct Fly {
    R P0, P2, e1, e3, M0, M2, ax0, ax2, ax1, ax3, ay0, ay2, ay1, ay3, o1, o3;
};
template <typename R>
__device__ __forceinline__ Fly<R> butterflies(const R* f)
{
    Fly<R> b;
    const R sx0 = f[0] + f[2], sy0 = f[1] + f[3], sx2 = f[8] + f[10], sy2 = f[9] + f[11];
    b.ax0 = f[0] - f[2];
    b.ay0 = f[1] - f[3];
    b.ax2 = f[8] - f[10];
    b.ay2 = f[9] - f[11];
    b.P0 = sx0 + sy0;
    b.M0 = sx0 - sy0;
    b.P2 = sx2 + sy2;
    b.M2 = sx2 - sy2;
    const R s01 = f[4] + f[5], d01 = f[4] - f[5], s23 = f[6] + f[7], d23 = f[6] - f[7];
    const R t01 = f[12] + f[13], u01 = f[12] - f[13], t23 = f[14] + f[15], u23 = f[14] - f[15];
    b.e1 = s01 + s23;
    b.ay1 = s01 - s23;
    b.ax1 = d01 - d23;
    b.o1 = d01 + d23;
    b.e3 = t01 + t23;
    b.ay3 = t01 - t23;
    b.ax3 = u01 - u23;
    b.o3 = u01 + u23;
    return b;
}
template <typename R>
__device__ __forceinline__ R dot4(const R* c, R w, R x, R y, R z)
{
    return fm(c[3], z, fm(c[2], y, fm(c[1], x, mu(c[0], w))));
}

// Delta_5..16 = f_hat - f_hat^eq, the equilibrium entering as the product of an FMA
// (m1 = rho, m2 = rho u_x, m3 = rho u_y)
template <typename R>
__device__ __forceinline__ void deltas(const ModelConst<R>& K, const LineConst<R>& E, const Fly<R>& b,
                                       R m1, R m2, R m3, R ux, R uy, R ux2, R uy2, R u2, R T, R pT, R* D)
{
    const R Ta = ad(T, ux2), Tb = ad(T, uy2);
    const R A = fm(E.di2, T, u2), B = fm(R(2), T, A);
    const R p2 = dot4(E.h2, b.P0, b.P2, b.e1, b.e3), p3 = dot4(E.h3, b.P0, b.P2, b.e1, b.e3);
    const R a0 = fm(E.ha[1], b.M2, mu(E.ha[0], b.M0)), a1 = fm(E.ha[3], b.M2, mu(E.ha[2], b.M0));
    D[0] = fm(-m1, Ta, ad(p2, a0));
    D[2] = fm(-m1, Tb, ad(p2, -a0));
    D[9] = fm(-mu(m2, ux), B, fm(-pT, A, ad(p3, a1)));
    D[11] = fm(-mu(m3, uy), B, fm(-pT, A, ad(p3, -a1)));
    D[1] = fm(-m2, uy, fm(K.Boo[1], b.o3, mu(K.Boo[0], b.o1)));
    D[10] = fm(-mu(m2, uy), B, fm(K.Boo[3], b.o3, mu(K.Boo[2], b.o1)));
    D[3] = fm(-m2, A, dot4(K.Bodd + 4, b.ax0, b.ax2, b.ax1, b.ax3));
    D[5] = fm(-m2, fm(R(2), T, Ta), dot4(K.Bodd + 8, b.ax0, b.ax2, b.ax1, b.ax3));
    D[7] = fm(-m2, Tb, dot4(K.Bodd + 12, b.ax0, b.ax2, b.ax1, b.ax3));
    D[4] = fm(-m3, A, dot4(K.Bodd + 4, b.ay0, b.ay2, b.ay1, b.ay3));
    D[8] = fm(-m3, fm(R(2), T, Tb), dot4(K.Bodd + 8, b.ay0, b.ay2, b.ay1, b.ay3));
    D[6] = fm(-m3, Ta, dot4(K.Bodd + 12, b.ay0, b.ay2, b.ay1, b.ay3));
}

// W = Omega = M^-1 [-S Delta + A_hat + C_hat] in block form (Omega_hat_1..3 vanish). dux,
// duy: differences of u between the right and the left neighbour; cr: dlambda times the
// chemical constant, `react` (warp-uniform) if it is nonzero anywhere in the warp.
template <typename R>
__device__ __forceinline__ void collide(const ModelConst<R>& K, const LineConst<R>& E, const R* D, R m1,
                                        R m2, R m3, R ux, R uy, R u2, R T, R pT, R dux, R duy, bool react,
                                        R cr, R* W)
{
    R Om[16]; // Omega_hat; the ES and EA sectors already joined (es, ea)
#pragma unroll
    for (int k = 4; k < 16; k++)
        if (k != 6 && k != 15) Om[k] = mu(-K.S[k], D[k - 4]);
    R es2 = fm(-K.S[6], D[2], Om[4]), ea0 = fm(K.S[6], D[2], Om[4]);
    R es3 = fm(-K.S[15], D[11], Om[13]), ea1 = fm(K.S[15], D[11], Om[13]);
    if (E.a_hat) { // A_hat_8, A_hat_9 (Eqs. (3)-(4))
        Om[7] = fm(pT, fm(E.c8y, mu(uy, duy), mu(E.c8x, mu(ux, dux))), Om[7]);
        Om[8] = fm(pT, fm(E.c9y, mu(ux, duy), mu(E.c9x, mu(uy, dux))), Om[8]);
    }
    R pes[4], pea[2], px[4], py[4], po[2], e1 = R(0); // e1: Omega_hat_4
    if (react) { // C_hat = d f_hat^eq / dT cr (Eqs. (19)-(23))
        const R dA = fm(R(2) * E.di2, T, u2), pd = mu(m1, dA), c4 = E.di2 + R(2);
        const R xx = mu(mu(m2, ux), c4), yy = mu(mu(m3, uy), c4), xy = mu(mu(m2, uy), c4);
        e1 = mu(mu(m1, K.DI), cr);
        es2 = fm(R(2) * m1, cr, es2);
        es3 = fm(ad(R(2) * pd, ad(xx, yy)), cr, es3);
        ea1 = fm(ad(xx, -yy), cr, ea1);
        Om[7] = fm(mu(E.di2, m2), cr, Om[7]);
        Om[8] = fm(mu(E.di2, m3), cr, Om[8]);
        Om[9] = fm(mu(R(3), m2), cr, Om[9]);
        Om[10] = fm(m3, cr, Om[10]);
        Om[11] = fm(m2, cr, Om[11]);
        Om[12] = fm(mu(R(3), m3), cr, Om[12]);
        Om[14] = fm(xy, cr, Om[14]);
    }
#pragma unroll
    for (int r = 0; r < 4; r++) {
        pes[r] = fm(K.Ies[4 * r + 3], es3, mu(K.Ies[4 * r + 2], es2));
        px[r] = fm(K.Iodd[4 * r + 3], Om[11], fm(K.Iodd[4 * r + 2], Om[9], mu(K.Iodd[4 * r + 1], Om[7])));
        py[r] = fm(K.Iodd[4 * r + 3], Om[10], fm(K.Iodd[4 * r + 2], Om[12], mu(K.Iodd[4 * r + 1], Om[8])));
    }
    if (react) {
#pragma unroll
        for (int r = 0; r < 4; r++) pes[r] = fm(K.Ies[4 * r + 1], e1, pes[r]);
    }
#pragma unroll
    for (int r = 0; r < 2; r++) {
        pea[r] = fm(K.Iea[2 * r + 1], ea1, mu(K.Iea[2 * r], ea0));
        po[r] = fm(K.Ioo[2 * r + 1], Om[14], mu(K.Ioo[2 * r], Om[5]));
    }
#pragma unroll
    for (int c = 0; c < 2; c++) {
        const R pp = ad(pes[c], pea[c]), pm = ad(pes[c], -pea[c]);
        W[8 * c] = ad(pp, px[c]);
        W[8 * c + 2] = ad(pp, -px[c]);
        W[8 * c + 1] = ad(pm, py[c]);
        W[8 * c + 3] = ad(pm, -py[c]);
        const R eo = ad(pes[2 + c], po[c]), em = ad(pes[2 + c], -po[c]);
        const R xp = ad(px[2 + c], py[2 + c]), xm = ad(px[2 + c], -py[2 + c]);
        W[4 + 8 * c] = ad(eo, xp);
        W[5 + 8 * c] = ad(em, -xm);
        W[6 + 8 * c] = ad(eo, -xp);
        W[7 + 8 * c] = ad(em, xm);
    }
}

// ---- per-warp TNE statistics ----------------------------------------------------
// Row k of td (stride ld) holds Delta_{k+5} (k < 12), d and d^2 of the block's cells. The
// warp's lanes take the 26 sums over the warp's own cells (those in `mask`), one quantity
// per lane, and on the way the 24 extremes (of the integer images, in the gaps of the FP64
// unit): 32 FP64 additions instead of the 130 of one shuffle tree per quantity. Results in
// the order of the partials, [TNE_PART].
__device__ __forceinline__ void warp_tne(const double* td, int ld, unsigned mask, double* out)
{
    const int lane = threadIdx.x & 31, row = lane < TNE_K ? lane : lane - TNE_K;
    if (lane >= NSUM) return;
    const bool second = lane >= TNE_K && lane < NMM; // |Delta| and the maximum
    const long long keep = second ? 0x7fffffffffffffffll : -1ll, flip = second ? -1ll : 0ll;
    const double* p = td + row * ld;
    double s = 0.0;
    long long v = order64(DBL_MAX); // the maximum as the minimum of the complements
    for (int j = 0; j < 32; j++) {
        if (!(mask >> j & 1u)) continue;
        const double x = p[j];
        s += __longlong_as_double(__double_as_longlong(x) & keep);
        const long long k = order64(x) ^ flip;
        v = k < v ? k : v;
    }
    out[lane < NMM ? lane : 2 * TNE_K + lane] = s;
    if (lane < NMM) out[2 * TNE_K + lane] = unorder64(v ^ flip);
}
// the same of FP32 terms: exact pairs (TwoSum), joined in FP64 once
__device__ __forceinline__ void warp_tne(const float* td, int ld, unsigned mask, double* out)
{
    const int lane = threadIdx.x & 31, row = lane < TNE_K ? lane : lane - TNE_K;
    if (lane >= NSUM) return;
    const bool second = lane >= TNE_K && lane < NMM;
    const unsigned keep = second ? 0x7fffffffu : 0xffffffffu;
    const float sign = second ? -1.f : 1.f; // the maximum as the minimum of the negated
    const float* p = td + row * ld;
    float s = 0.f, c = 0.f, v = FLT_MAX;
    for (int j = 0; j < 32; j++) {
        if (!(mask >> j & 1u)) continue;
        const float x = p[j];
        const df t = two_sum(s, __uint_as_float(__float_as_uint(x) & keep));
        s = t.hi;
        c += t.lo;
        v = fminf(v, sign * x);
    }
    out[lane < NMM ? lane : 2 * TNE_K + lane] = (double)s + (double)c;
    if (lane < NMM) out[2 * TNE_K + lane] = mask ? (double)(sign * v) : (second ? -DBL_MAX : DBL_MAX);
}

// scalar form of conserved_pair_u: the conserved moments as exact double-float sums
struct S1 {
    float hi, lo;
};
__device__ __forceinline__ S1 s_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ S1 s_add(S1 a, S1 b)
{
    const S1 s = s_sum(a.hi, b.hi);
    return {s.hi, __fadd_rn(__fadd_rn(a.lo, b.lo), s.lo)};
}
__device__ __forceinline__ S1 s_sub(S1 a, S1 b) { return s_add(a, {-b.hi, -b.lo}); }
__device__ __forceinline__ S1 s_mul(S1 a, float ch, float cl)
{
    const float p = __fmul_rn(a.hi, ch);
    float e = __fmaf_rn(a.hi, ch, -p);
    e = __fmaf_rn(a.hi, cl, e);
    e = __fmaf_rn(a.lo, ch, e);
    return {p, e};
}
__device__ __forceinline__ S1 s_norm(S1 a)
{
    const float s = __fadd_rn(a.hi, a.lo);
    return {s, __fsub_rn(a.lo, __fsub_rn(s, a.hi))};
}

// rho, u, T of one FP32 cell: exact conserved sums, then FP64 (REC = 0) or double-float
// (REC = 1); ig = T > T_ig in that precision, ok = rho, T > 0 and everything finite
template <int REC>
__device__ __forceinline__ void recover32(const ModelConst<float>& K, const float* f, float& rho,
                                          float& ux, float& uy, float& T, bool& ig, bool& ok)
{
    if constexpr (REC == 1) {
        double r, u, v, t;
        recover_df32(K.cd, K.wd, K.inv_DId, f, r, u, v, t);
        rho = (float)r;
        ux = (float)u;
        uy = (float)v;
        T = (float)t;
        ig = t > K.T_igd;
        ok = rho > 0.f && t > 0.0 && isfinite(ux + uy + rho) && isfinite(t);
    } else {
        S1 P[2], E[2], AX[4], AY[4];
#pragma unroll
        for (int a = 0; a < 2; a++) {
            const int b = 8 * a;
            P[a] = s_add(s_sum(f[b], f[b + 2]), s_sum(f[b + 1], f[b + 3]));
            AX[a] = s_sum(f[b], -f[b + 2]);
            AY[a] = s_sum(f[b + 1], -f[b + 3]);
        }
#pragma unroll
        for (int d = 0; d < 2; d++) {
            const int b = 4 + 8 * d;
            const S1 s01 = s_sum(f[b], f[b + 1]), d01 = s_sum(f[b], -f[b + 1]);
            const S1 s23 = s_sum(f[b + 2], f[b + 3]), d23 = s_sum(f[b + 2], -f[b + 3]);
            E[d] = s_add(s01, s23);
            AY[2 + d] = s_sub(s01, s23);
            AX[2 + d] = s_sub(d01, d23);
        }
        const S1 m1 = s_norm(s_add(s_add(P[0], P[1]), s_add(E[0], E[1])));
        const S1 m2 = s_norm(s_add(s_add(s_mul(AX[0], K.cdh[0], K.cdl[0]), s_mul(AX[1], K.cdh[2], K.cdl[2])),
                                   s_add(s_mul(AX[2], K.cdh[1], K.cdl[1]), s_mul(AX[3], K.cdh[3], K.cdl[3]))));
        const S1 m3 = s_norm(s_add(s_add(s_mul(AY[0], K.cdh[0], K.cdl[0]), s_mul(AY[1], K.cdh[2], K.cdl[2])),
                                   s_add(s_mul(AY[2], K.cdh[1], K.cdl[1]), s_mul(AY[3], K.cdh[3], K.cdl[3]))));
        const S1 m4 = s_norm(s_add(s_add(s_mul(P[0], K.wdh[0], K.wdl[0]), s_mul(P[1], K.wdh[2], K.wdl[2])),
                                   s_add(s_mul(E[0], K.wdh[1], K.wdl[1]), s_mul(E[1], K.wdh[3], K.wdl[3]))));
        double u, v, t;
        const double r = df_to_f64_fast(m1.hi, m1.lo);
        recover_one_f64_fast(m1.hi, m1.lo, r, df_to_f64_fast(m2.hi, m2.lo), df_to_f64_fast(m3.hi, m3.lo),
                             df_to_f64_fast(m4.hi, m4.lo), K.inv_DId, u, v, t);
        rho = m1.hi;
        ux = d2f_fast(u);
        uy = d2f_fast(v);
        T = d2f_fast(t);
        ig = dbits(t) > dbits(K.T_igd);
        ok = fabsf(m1.hi) <= FLT_MAX && fabsf(m2.hi) <= FLT_MAX && fabsf(m3.hi) <= FLT_MAX &&
             fabsf(m4.hi) <= FLT_MAX && m1.hi > 0.f && dbits(t) > 0 && dbits(t) <= dbits(DBL_MAX);
    }
}

// shared memory of a block of n threads: [NX + 2][n] published planes, u_x, u_y (twice for
// FP32, whose single barrier per step lets the next step's values be written early), FP64:
// [NX][n] differences; with TNE [14][n + 1] and 50 results per warp
template <typename R>
__host__ __device__ constexpr size_t line_smem(int n, bool tne)
{
    const size_t pub = (size_t)(NX + 2) * n * sizeof(R);
    const size_t rest = sizeof(R) == 8 ? (size_t)NX * n * sizeof(R) : pub;
    return pub + rest + (tne ? (size_t)(n / 32) * TNE_PART * 8 + (size_t)14 * (n + 1) * sizeof(R) + 16 : 0);
}

// TNE = false leaves the records' code out (12 % of an FP32 step)
template <typename R, int REC, bool TNE>
__global__ void __launch_bounds__(LINE_THREADS)
    line_kernel(const __grid_constant__ ModelConst<R> K, const __grid_constant__ LineConst<R> E,
                const __grid_constant__ LineArgs a, int kmax)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int n = blockDim.x, t = threadIdx.x, h = 2 * kmax, own = n - 2 * h;
    R* pub = reinterpret_cast<R*>(smem);               // [NX + 2][n]
    R* dif = pub + (NX + 2) * n;                       // FP64: [NX][n]; FP32: the second pub
    double* wres = reinterpret_cast<double*>(dif + (sizeof(R) == 8 ? NX : NX + 2) * n);
    R* td = reinterpret_cast<R*>(wres + (n / 32) * TNE_PART); // [14][n + 1]

    const int nx = K.nx;
    const int64_t plane = K.plane;
    const int x0 = blockIdx.x * own - h, x = x0 + t;
    const R* in = static_cast<const R*>(a.in);

    // the cell this lane stands for, and the ends of the index range that neighbours are
    // read through (a zero-gradient end inside the window closes it)
    int gx = x, dir = -1;
    bool fixed = false; // a ghost lane: never updated
    if (x < 0 || x >= nx) {
        const int s = x < 0 ? 0 : 1, code = K.sbc[s];
        if (code == 0) {
            gx = x % nx;
            gx = gx < 0 ? gx + nx : gx;
        } else {
            gx = x < 0 ? 0 : nx - 1;
            fixed = true;
            if (code == 3) dir = s;
        }
    }
    const int lo = K.sbc[0] == 1 && -x0 > 0 ? (-x0 < n ? -x0 : n - 1) : 0;
    const int hi = K.sbc[1] == 1 && nx - 1 - x0 < n - 1 ? (nx - 1 - x0 > 0 ? nx - 1 - x0 : 0) : n - 1;
    auto at = [&](int j) { return j < lo ? lo : (j > hi ? hi : j); };
    const int jm2 = at(t - 2), jm1 = at(t - 1), j0 = at(t), jp1 = at(t + 1), jp2 = at(t + 2);
    const int dm2 = t >= 2 ? t - 2 : 0, dm1 = t >= 1 ? t - 1 : 0, dp1 = t + 1 < n ? t + 1 : n - 1;
    const bool mine = t >= h && t < h + own && x < nx;

    R f[16], lam;
#pragma unroll
    for (int i = 0; i < 16; i++) f[i] = dir >= 0 ? K.sfeq[dir][i] : in[i * plane + gx];
    lam = dir >= 0 ? K.sfeq[dir][16] : in[16 * plane + gx];

    const bool tne = TNE && a.tne_every > 0;
    const int64_t step0 = tne ? a.ctr->step : 0;
    int bad = 0;
    for (int s = 0; s < a.nsteps; s++) {
        const bool do_tne = tne && (step0 + s) % a.tne_every == 0;
        R nf[16], nlam;
        R m1, m2, m3, ux, uy, T, dux, duy;
        bool hot; // the cell reacts; a burnt one adds nothing
        const Fly<R> b = butterflies(f);
        R* P = sizeof(R) == 4 && (s & 1) ? dif : pub; // what this step publishes
        R ux2, uy2, u2;
        if constexpr (sizeof(R) == 8) {
            // recovery (Eqs. (5)-(7)) from the butterflies the moments share
            m1 = (b.P0 + b.P2) + (b.e1 + b.e3);
            m2 = fm(K.cd[3], b.ax3, fm(K.cd[1], b.ax1, fm(K.cd[2], b.ax2, mu(K.cd[0], b.ax0))));
            m3 = fm(K.cd[3], b.ay3, fm(K.cd[1], b.ay1, fm(K.cd[2], b.ay2, mu(K.cd[0], b.ay0))));
            const double m4 = fm(K.wd[3], b.e3, fm(K.wd[1], b.e1, fm(K.wd[2], b.P2, mu(K.wd[0], b.P0))));
            const double q = recip64(m1);
            ux = mu(m2, q);
            uy = mu(m3, q);
            ux2 = mu(ux, ux);
            uy2 = mu(uy, uy);
            u2 = ad(ux2, uy2);
            T = mu(fm(m4, q, -u2), K.inv_DId);
            const long long tb = dbits(T), big = dbits(DBL_MAX);
            if (mine && !(dbits(m1) > 0 && dbits(m1) <= big && tb > 0 && tb <= big)) bad = 1;
            hot = tb > dbits(K.T_igd) && dbits(lam) != dbits(1.0);
        } else {
            bool ok;
            recover32<REC>(K, f, m1, ux, uy, T, hot, ok);
            if (mine && !ok) bad = 1;
            hot = hot && lam != 1.f;
            m2 = mu(m1, ux);
            m3 = mu(m1, uy);
            ux2 = mu(ux, ux);
            uy2 = mu(uy, uy);
            u2 = ad(ux2, uy2);
        }
#pragma unroll
        for (int k = 0; k < NX; k++) P[k * n + t] = slot_plane(k) == 16 ? lam : f[slot_plane(k) & 15];
        P[NX * n + t] = ux;
        P[(NX + 1) * n + t] = uy;
        __syncthreads();
        if constexpr (sizeof(R) == 8) {
            // each lane forms the differences to its right neighbour
#pragma unroll
            for (int k = 0; k < NX; k++) dif[k * n + t] = P[k * n + jp1] - P[k * n + j0];
        }
        dux = P[NX * n + jp1] - P[NX * n + jm1];
        duy = P[(NX + 1) * n + jp1] - P[(NX + 1) * n + jm1];
        R D[TNE_K], W[16];
        const R pT = mu(m1, T);
        deltas(K, E, b, m1, m2, m3, ux, uy, ux2, uy2, u2, T, pT, D);
        if (do_tne) {
            R d2 = mu(D[0], D[0]);
            td[t] = D[0];
#pragma unroll
            for (int k = 1; k < TNE_K; k++) {
                td[k * (n + 1) + t] = D[k];
                d2 = fm(D[k], D[k], d2);
            }
            td[12 * (n + 1) + t] = sqrt(d2);
            td[13 * (n + 1) + t] = d2;
        }
        // reaction over dt (Eq. (28)), and the collision
        const bool react = __any_sync(0xffffffffu, hot);
        R dlam = R(0);
        if (react && hot) dlam = reaction_increment(lam, mu(K.omega1, pT), mu(K.omega2, pT), K.dt);
        collide(K, E, D, m1, m2, m3, ux, uy, u2, T, pT, dux, duy, react, mu(dlam, K.chem), W);
        // NND differences (v > 0 from d_{j-2}, d_{j-1}, d_j; v < 0 from d_{j-1}, d_j, d_{j+1};
        // d_j = q_{j+1} - q_j) and the Euler update; lambda's side by the sign of u_x
        if constexpr (sizeof(R) == 8) __syncthreads();
        auto nnd = [&](int k, R q, bool neg) -> R {
            if constexpr (sizeof(R) == 8) {
                const double* d = dif + k * n;
                const double dl = d[neg ? dm1 : dm2], dc = d[neg ? t : dm1], dr = d[neg ? dp1 : t];
                const double m01 = mm64(dl, dc), m12 = mm64(dc, dr);
                return fm(neg ? -0.5 : 0.5, ad(m12, -m01), dc);
            } else {
                const float* r = P + k * n;
                const float a0 = r[neg ? jp2 : jm2], l = r[jm1], h_ = r[jp1];
                const float d1 = q - l, d2 = h_ - q, dx = neg ? a0 - h_ : l - a0;
                const float c = neg ? d2 : d1, m12 = mmag(d1, d2), mx = mmag(dx, c);
                // neg: d2 - (mm23 - mm12)/2, else d1 + (mm12 - mm01)/2, both of sign(c)
                return fm(0.5f, sgnmul(ad(m12, -mx), c), c);
            }
        };
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const int k = slot_of(i);
            const R c = k >= 6 ? E.cdx[i >> 2] : -E.cdx[i >> 2];
            if constexpr (sizeof(R) == 8) { // two FMAs
                if (k >= 0) W[i] = fm(c, nnd(k, f[i], k >= 6), W[i]);
                nf[i] = fm(K.dt, W[i], f[i]);
            } else { // the increment first: one rounding at the size of f
                W[i] = mu(K.dt, W[i]);
                if (k >= 0) W[i] = fm(c, nnd(k, f[i], k >= 6), W[i]);
                nf[i] = ad(f[i], W[i]);
            }
        }
        nlam = ad(lam, fm(mu(-E.dtdx, ux), nnd(12, lam, negative(ux)), dlam));
        nlam = clamp01(nlam);
        if (do_tne) {
            const int warp = t >> 5;
            const unsigned mask = __ballot_sync(0xffffffffu, mine);
            __syncwarp(); // the warp's own columns of td are written
            warp_tne(td + warp * 32, n + 1, mask, wres + warp * TNE_PART);
            __syncthreads();
            if (t < TNE_PART) {
                const int kind = tne_kind(t);
                double v = wres[t];
                for (int w = 1; w < n / 32; w++) v = tne_comb(kind, v, wres[w * TNE_PART + t]);
                a.partials[((size_t)s * TNE_PART + t) * gridDim.x + blockIdx.x] = v;
            }
        }
        const bool last = s == a.nsteps - 1;
        if (mine && (last || a.out_stride > 0)) {
            R* out = static_cast<R*>(a.out) + (a.out_stride > 0 ? s * a.out_stride : 0) + x;
            if (a.stage >= 2) { // a later SSP Runge-Kutta stage: weighted with u^n
                const R* prev = static_cast<const R*>(a.prev) + x;
                const R wp = (R)a.wprev, wn = (R)a.wnew;
#pragma unroll
                for (int i = 0; i < 16; i++) out[i * plane] = fm(wp, prev[i * plane], mu(wn, nf[i]));
                out[16 * plane] = fm(wp, prev[16 * plane], mu(wn, nlam));
            } else {
#pragma unroll
                for (int i = 0; i < 16; i++) out[i * plane] = nf[i];
                out[16 * plane] = nlam;
            }
        }
        if (!fixed) {
#pragma unroll
            for (int i = 0; i < 16; i++) f[i] = nf[i];
            lam = nlam;
        }
    }

    // status and step counter. Without TNE no block reads the counter, so block 0 moves it
    // on; with TNE the last block to finish does
    if (__syncthreads_or(bad) && t == 0) atomicOr(&a.ctr->status, 1);
    const bool counts = a.stage == 0 || a.stage == 2;
    if (!tne) {
        if (blockIdx.x == 0 && t == 0) {
            if (a.stage < 2) a.ctr->tne_pending = 0;
            if (counts) a.ctr->step += a.nsteps;
        }
    } else if (t == 0) {
        if (atomicAdd(&a.ctr->arrivals, 1u) == gridDim.x - 1) {
            const int64_t e = a.tne_every, last = step0 + a.nsteps - 1;
            const int64_t due = last / e - (step0 + e - 1) / e + 1;
            a.ctr->hist_count += due;
            a.ctr->tne_step = step0;
            a.ctr->tne_pending = due > 0 ? a.nsteps : 0;
            if (counts) a.ctr->step = step0 + a.nsteps;
            a.ctr->arrivals = 0u;
        }
    }
}

template <typename R>
void line_const(const ModelConst<R>& K, LineConst<R>* E)
{
    for (int j = 0; j < 4; j++) {
        E->h2[j] = R(0.5) * K.Bes[8 + j];
        E->h3[j] = R(0.5) * K.Bes[12 + j];
        E->ha[j] = R(0.5) * K.Bea[j];
        E->cdx[j] = sizeof(R) == 8 ? K.c[j] * K.inv_dx : K.dt * K.c[j] * K.inv_dx;
    }
    // theta = inv_DI du_x/dx; 4 u_x (du_x/dx - theta), -4 u_y theta, 2 u du_y/dx
    const R g = K.half_inv_dx;
    E->c8x = K.A8c * R(4) * (R(1) - K.inv_DI) * g;
    E->c8y = K.A8c * R(2) * g;
    E->c9x = K.A9c * R(-4) * K.inv_DI * g;
    E->c9y = K.A9c * R(2) * g;
    E->dtdx = K.dt * K.inv_dx;
    E->di2 = K.DI + R(2);
    E->a_hat = K.A8c != R(0) || K.A9c != R(0);
}

template <typename R, int REC, bool TNE>
cudaError_t line_launch_t(const ModelConst<R>& K, const LinePlan& p, const LineArgs& a, cudaStream_t s)
{
    const size_t bytes = line_smem<R>(p.threads, a.tne_every > 0);
    static cudaError_t done = cudaFuncSetAttribute(line_kernel<R, REC, TNE>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)line_smem<R>(LINE_THREADS, true));
    if (done != cudaSuccess) return done;
    LineConst<R> E;
    line_const(K, &E);
    line_kernel<R, REC, TNE><<<p.grid, p.threads, bytes, s>>>(K, E, a, p.steps);
    return cudaGetLastError();
}

} // namespace

// The cut of a 1-D grid: the (threads, steps) with the least time per step as measured over
// 19 cuts of seven lengths from 400 to 2^20 cells, modelled by the warps w an SM gets. FP64:
// an SM's FP64 units pass 3.0 us of warps one after another once its four quarters are busy
// (us per step: w = 3 12.8, 4 13.9, 5 16.3, 6 17.5, 8 24.1, 16 44.7) and a launch costs
// 1.5 us beside its steps. FP32: latency first, issue from about 20 warps on (w = 4 1.29,
// 6 1.63, 8 1.93, 16 2.95, 230 40.5), a launch 2.0 us. So short grids take 16 steps per
// launch (400 cells, FP32: 1.42 us per step against 3.3 with one), 16384 cells 4 steps of
// 128 threads, one block per SM (FP32 1.80, FP64 14.2; 8 steps, whose 171 blocks no longer
// fit one per SM, 2.19 and 23.3), and a million cells two FP32 steps (41.5; one 48.3, eight
// 46.2), one FP64 step (622; four 683).
LinePlan line_plan(int precision, int nx)
{
    static int sms = -1;
    if (sms < 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 152;
    }
    LinePlan best = {128, 1, (nx + 123) / 124};
    double t_best = 1e300;
    for (int threads = 32; threads <= LINE_THREADS; threads += 32)
        for (int steps = 1; steps <= 16; steps *= 2) {
            const int own = threads - 4 * steps;
            if (own < 16) continue;
            const int grid = (nx + own - 1) / own;
            const double w = (double)((grid + sms - 1) / sms) * (threads / 32);
            const double t = precision == 0 ? (w > 4.25 ? 3.0 * w : 12.8) + 1.5 / steps
                                            : (w > 21.0 ? 0.17 * w : 0.85 + 0.131 * w) + 2.0 / steps;
            if (t < t_best) t_best = t, best = {threads, steps, grid};
        }
    return best;
}

cudaError_t launch_line(int precision, int recovery, const void* K, const LinePlan& p,
                        const LineArgs& a, cudaStream_t s)
{
    if (a.nsteps < 1 || a.nsteps > p.steps) return cudaErrorInvalidValue;
    LineArgs b = a;
    if (a.stage >= 2) b.tne_every = 0; // only u^n has records
    if (precision == 0) {
        const ModelConst<double>& Kd = *static_cast<const ModelConst<double>*>(K);
        return b.tne_every > 0 ? line_launch_t<double, 0, true>(Kd, p, b, s) : line_launch_t<double, 0, false>(Kd, p, b, s);
    }
    const ModelConst<float>& Kf = *static_cast<const ModelConst<float>*>(K);
    if (b.tne_every > 0)
        return recovery == 1 ? line_launch_t<float, 1, true>(Kf, p, b, s) : line_launch_t<float, 0, true>(Kf, p, b, s);
    return recovery == 1 ? line_launch_t<float, 1, false>(Kf, p, b, s) : line_launch_t<float, 0, false>(Kf, p, b, s);
}

} // namespace lbk
