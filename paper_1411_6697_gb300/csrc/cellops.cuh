// cellops.cuh -- one cell's step on one thread, FP64 or FP32 (line.cu, tile.cu): exact
// rounding order, as few FP64 instructions as the formulas allow.
//
// One FP64 warp instruction (add, multiply, FMA or compare alike) holds its quarter of a GB300
// SM for 64 cycles, whatever its lanes do and whether or not it depends on the one before; an
// integer or FP32 instruction takes one. So minmod, comparisons, clamps and extremes of FP64
// values work on their bit patterns, the factors 1/2 of four moments are folded into the
// matrix, the FP64 f_hat^eq enters Delta_k as the product of an FMA, the reciprocal is an FP32 seed with
// one third-order correction, and the terms of the reaction and of A_hat are left out of warps
// and models where they vanish.
#pragma once
#include <float.h>

#include "cell.cuh"
#include "pair.cuh"
#include "reduce.cuh"

namespace lbk {

template <typename R>
struct StepConst {
    R h2[4], h3[4], ha[4]; // rows of the ES and EA blocks of m_5, m_7, m_14, m_16, halved
    R c8, c9, gx, gy;      // A8c, A9c, 1/(2 dx), 1/(2 dy)
    R cdx[4], cdy[4];      // c / dx, c / dy of each orbit
    R dtdx, dtdy, inv_DI;
    R di2, di4;            // D + I + 2, D + I + 4
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
// 1/x: FP32 estimate (22 bits), then q + q (e + e^2), e = 1 - x q, of x scaled to [1, 2) by its
// exponent field; the exponent goes back into the result on the integer pipe. NaN where the result
// or x is not a normal number (x zero, subnormal, from 2^1022 on or not finite), so that the tests
// on T see it.
__device__ __forceinline__ double recip64(double x)
{
    const int hi = __double2hiint(x), e2 = hi & 0x7ff00000;
    const double s = __hiloint2double(hi - e2 + 0x3ff00000, __double2loint(x));
    const double q = f2d_fast(rcp_approx(d2f_fast(s)));
    const double e = __fma_rn(-s, q, 1.0), r = __fma_rn(q, __fma_rn(e, e, e), q);
    const bool normal = (unsigned)(e2 - 0x00100000) < 0x7fc00000u;
    return __hiloint2double(normal ? __double2hiint(r) + 0x3ff00000 - e2 : 0x7ff80000, __double2loint(r));
}

// Rounded operations that the compiler must not merge: every path through the step then
// rounds alike, whichever instantiation (with records or without) it runs in.
__device__ __forceinline__ double fm(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fm(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mu(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mu(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double ad(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float ad(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }

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

// Delta_5..16 = f_hat - f_hat^eq (m1 = rho, m2 = rho u_x, m3 = rho u_y). FP64: the equilibrium
// enters as the product of an FMA.
template <bool>
__device__ __forceinline__ void deltas(const ModelConst<double>& K, const StepConst<double>& E,
                                       const Fly<double>& b, double m1, double m2, double m3, double ux, double uy,
                                       double ux2, double uy2, double u2, double T, double pT, double* D)
{
    const double Ta = ad(T, ux2), Tb = ad(T, uy2);
    const double A = fm(E.di2, T, u2), B = fm(2.0, T, A);
    const double p2 = dot4(E.h2, b.P0, b.P2, b.e1, b.e3), p3 = dot4(E.h3, b.P0, b.P2, b.e1, b.e3);
    const double a0 = fm(E.ha[1], b.M2, mu(E.ha[0], b.M0)), a1 = fm(E.ha[3], b.M2, mu(E.ha[2], b.M0));
    D[0] = fm(-m1, Ta, ad(p2, a0));
    D[2] = fm(-m1, Tb, ad(p2, -a0));
    D[9] = fm(-mu(m2, ux), B, fm(-pT, A, ad(p3, a1)));
    D[11] = fm(-mu(m3, uy), B, fm(-pT, A, ad(p3, -a1)));
    D[1] = fm(-m2, uy, fm(K.Boo[1], b.o3, mu(K.Boo[0], b.o1)));
    D[10] = fm(-mu(m2, uy), B, fm(K.Boo[3], b.o3, mu(K.Boo[2], b.o1)));
    D[3] = fm(-m2, A, dot4(K.Bodd + 4, b.ax0, b.ax2, b.ax1, b.ax3));
    D[5] = fm(-m2, fm(2.0, T, Ta), dot4(K.Bodd + 8, b.ax0, b.ax2, b.ax1, b.ax3));
    D[7] = fm(-m2, Tb, dot4(K.Bodd + 12, b.ax0, b.ax2, b.ax1, b.ax3));
    D[4] = fm(-m3, A, dot4(K.Bodd + 4, b.ay0, b.ay2, b.ay1, b.ay3));
    D[8] = fm(-m3, fm(2.0, T, Tb), dot4(K.Bodd + 8, b.ay0, b.ay2, b.ay1, b.ay3));
    D[6] = fm(-m3, Ta, dot4(K.Bodd + 12, b.ay0, b.ay2, b.ay1, b.ay3));
}
// FP32. The equilibria of the even moments are rounded before they are subtracted, like the moments
// themselves: in a uniform gas the two roundings then mostly cancel and the cell keeps its bits. As
// products of an FMA they leave the moment's own rounding in Delta, the same one step after step, and
// the run drifts (mean error of the state over 40 states: Sod tube of 400 cells, 600 steps 3.9e-7,
// with FMAs throughout 5.7e-7; batched detonations, 100 steps 2.7e-7 and 3.2e-7).
// FUSE: where products join sums in one FMA (the 1-D steps); without it each is rounded (the tiles).
template <bool FUSE>
__device__ __forceinline__ float mad(float a, float b, float c) { return FUSE ? fm(a, b, c) : ad(mu(a, b), c); }
template <bool FUSE>
__device__ __forceinline__ float less(float m, float a, float b) { return FUSE ? fm(-a, b, m) : sub(m, mu(a, b)); }
template <bool FUSE>
__device__ __forceinline__ void deltas(const ModelConst<float>& K, const StepConst<float>& E, const Fly<float>& b,
                                       float m1, float m2, float m3, float ux, float uy, float ux2, float uy2,
                                       float u2, float T, float, float* D)
{
    const float T3 = mu(3.f, T);
    const float Ta = mad<FUSE>(ux, ux, T), Tb = mad<FUSE>(uy, uy, T);
    const float A = mad<FUSE>(E.di2, T, u2), B = mad<FUSE>(E.di4, T, u2), q3 = mu(mu(m1, A), T), xy = mu(m2, uy);
    const float p2 = dot4(E.h2, b.P0, b.P2, b.e1, b.e3), p3 = dot4(E.h3, b.P0, b.P2, b.e1, b.e3);
    const float a0 = fm(E.ha[1], b.M2, mu(E.ha[0], b.M0)), a1 = fm(E.ha[3], b.M2, mu(E.ha[2], b.M0));
    D[0] = sub(ad(p2, a0), mu(m1, Ta));
    D[2] = sub(ad(p2, -a0), mu(m1, Tb));
    D[9] = sub(ad(p3, a1), mad<FUSE>(mu(m2, ux), B, q3));
    D[11] = sub(ad(p3, -a1), mad<FUSE>(mu(m3, uy), B, q3));
    D[1] = sub(fm(K.Boo[1], b.o3, mu(K.Boo[0], b.o1)), xy);
    D[10] = less<FUSE>(fm(K.Boo[3], b.o3, mu(K.Boo[2], b.o1)), xy, B);
    D[3] = less<FUSE>(dot4(K.Bodd + 4, b.ax0, b.ax2, b.ax1, b.ax3), m2, A);
    D[5] = less<FUSE>(dot4(K.Bodd + 8, b.ax0, b.ax2, b.ax1, b.ax3), m2, mad<FUSE>(ux, ux, T3));
    D[7] = less<FUSE>(dot4(K.Bodd + 12, b.ax0, b.ax2, b.ax1, b.ax3), m2, Tb);
    D[4] = less<FUSE>(dot4(K.Bodd + 4, b.ay0, b.ay2, b.ay1, b.ay3), m3, A);
    D[8] = less<FUSE>(dot4(K.Bodd + 8, b.ay0, b.ay2, b.ay1, b.ay3), m3, mad<FUSE>(uy, uy, T3));
    D[6] = less<FUSE>(dot4(K.Bodd + 12, b.ay0, b.ay2, b.ay1, b.ay3), m3, Ta);
}

// W = Omega = M^-1 [-S Delta + A_hat + C_hat] in block form (Omega_hat_1..3 vanish). S: the
// rates; w8 A8, w9 A9: A_hat_8 and A_hat_9 (a_hat); cr: dlambda times the chemical constant,
// `react` (warp-uniform) if it is nonzero anywhere in the warp. FP64 joins the rows that m_5 and m_7
// (m_14 and m_16) share with FMAs; FP32 rounds each row, then their sum and difference.
template <typename R>
struct Sectors { // M^-1 Omega_hat before the back butterflies
    R es[4], ea[2], ox[4], oy[4], oo[2];
};
template <bool, typename R>
__device__ __forceinline__ void sectors(const ModelConst<R>& K, const StepConst<R>& E, const R* S, const R* D, R m1,
                                        R m2, R m3, R ux, R uy, R u2, R T, R w8, R w9, R A8, R A9, bool react,
                                        R cr, Sectors<R>& z)
{
    R Om[16]; // Omega_hat; the ES and EA sectors already joined (es, ea)
#pragma unroll
    for (int k = 4; k < 16; k++)
        if (k != 6 && k != 15) Om[k] = mu(-S[k], D[k - 4]);
    R es2 = fm(-S[6], D[2], Om[4]), ea0 = fm(S[6], D[2], Om[4]);
    R es3 = fm(-S[15], D[11], Om[13]), ea1 = fm(S[15], D[11], Om[13]);
    if (E.a_hat) { // Eqs. (3)-(4)
        Om[7] = fm(w8, A8, Om[7]);
        Om[8] = fm(w9, A9, Om[8]);
    }
    R *pes = z.es, *pea = z.ea, *px = z.ox, *py = z.oy, *po = z.oo, e1 = R(0); // e1: Omega_hat_4
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
}
template <bool FUSE>
__device__ __forceinline__ void sectors(const ModelConst<float>& K, const StepConst<float>& E, const float* S,
                                        const float* D, float m1, float m2, float m3, float ux, float uy, float u2,
                                        float T, float w8, float w9, float A8, float A9, bool react, float cr,
                                        Sectors<float>& z)
{
    float Om[16] = {}, e1 = 0.f;
    if (react) { // C_hat = d f_hat^eq / dT cr
        const float dA = mad<FUSE>(2.f * E.di2, T, u2), c4 = E.di4, pd = mu(m1, dA);
        e1 = mu(mu(m1, K.DI), cr);
        Om[4] = Om[6] = mu(m1, cr);
        Om[7] = mu(mu(m2, E.di2), cr);
        Om[8] = mu(mu(m3, E.di2), cr);
        Om[9] = mu(mu(3.f, m2), cr);
        Om[10] = mu(m3, cr);
        Om[11] = mu(m2, cr);
        Om[12] = mu(mu(3.f, m3), cr);
        Om[13] = mu(mad<FUSE>(mu(m2, ux), c4, pd), cr);
        Om[14] = mu(mu(mu(m2, uy), c4), cr);
        Om[15] = mu(mad<FUSE>(mu(m3, uy), c4, pd), cr);
    }
#pragma unroll
    for (int k = 4; k < 16; k++) Om[k] = fm(-S[k], D[k - 4], Om[k]);
    if (E.a_hat) {
        Om[7] = ad(Om[7], mu(w8, A8));
        Om[8] = ad(Om[8], mu(w9, A9));
    }
    const float es2 = ad(Om[4], Om[6]), ea0 = ad(Om[4], -Om[6]), es3 = ad(Om[13], Om[15]), ea1 = ad(Om[13], -Om[15]);
#pragma unroll
    for (int r = 0; r < 4; r++) {
        z.es[r] = mu(K.Ies[4 * r + 2], es2);
        if (react) z.es[r] = fm(K.Ies[4 * r + 2], es2, mu(K.Ies[4 * r + 1], e1));
        z.es[r] = fm(K.Ies[4 * r + 3], es3, z.es[r]);
        z.ox[r] = fm(K.Iodd[4 * r + 3], Om[11], fm(K.Iodd[4 * r + 2], Om[9], mu(K.Iodd[4 * r + 1], Om[7])));
        z.oy[r] = fm(K.Iodd[4 * r + 3], Om[10], fm(K.Iodd[4 * r + 2], Om[12], mu(K.Iodd[4 * r + 1], Om[8])));
    }
#pragma unroll
    for (int r = 0; r < 2; r++) {
        z.ea[r] = fm(K.Iea[2 * r + 1], ea1, mu(K.Iea[2 * r], ea0));
        z.oo[r] = fm(K.Ioo[2 * r + 1], Om[14], mu(K.Ioo[2 * r], Om[5]));
    }
}
template <bool FUSE, typename R>
__device__ __forceinline__ void collide(const ModelConst<R>& K, const StepConst<R>& E, const R* S, const R* D, R m1,
                                        R m2, R m3, R ux, R uy, R u2, R T, R w8, R w9, R A8, R A9, bool react,
                                        R cr, R* W)
{
    Sectors<R> z;
    sectors<FUSE>(K, E, S, D, m1, m2, m3, ux, uy, u2, T, w8, w9, A8, A9, react, cr, z);
    const R *pes = z.es, *pea = z.ea, *px = z.ox, *py = z.oy, *po = z.oo;
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

// A_hat_8 and A_hat_9 (Eqs. (3)-(4)) as w8 A8 and w9 A9, from the differences of u between the right
// and left (..x) and, on a 2-D grid, the upper and lower (..y) neighbours. FP64: w8 = w9 = rho T
// (a_weight).
template <bool TWO_D>
__device__ __forceinline__ void a_hat(const StepConst<double>& E, double ux, double uy, double dxx, double dyx,
                                      double dxy, double dyy, double& A8, double& A9)
{
    const double gxx = mu(dxx, E.gx), u4 = mu(4.0, ux), v4 = mu(4.0, uy);
    if constexpr (TWO_D) {
        const double gyy = mu(dyy, E.gy), sh = mu(2.0, fm(dxy, E.gy, mu(dyx, E.gx)));
        const double th = mu(ad(gxx, gyy), E.inv_DI);
        A8 = mu(E.c8, fm(uy, sh, mu(u4, ad(gxx, -th))));
        A9 = mu(E.c9, fm(ux, sh, mu(v4, ad(gyy, -th))));
    } else {
        const double sh = mu(2.0, mu(dyx, E.gx)), th = mu(gxx, E.inv_DI);
        A8 = mu(E.c8, fm(uy, sh, mu(u4, ad(gxx, -th))));
        A9 = mu(E.c9, fm(ux, sh, mu(v4, -th)));
    }
}
template <bool TWO_D>
__device__ __forceinline__ void a_hat(const StepConst<float>& E, float ux, float uy, float dxx, float dyx, float dxy,
                                      float dyy, float& A8, float& A9)
{
    const float gxx = mu(dxx, E.gx), x4 = mu(4.f, ux), y4 = mu(4.f, uy);
    if constexpr (TWO_D) {
        const float gyy = mu(dyy, E.gy), sh = ad(mu(dyx, E.gx), mu(dxy, E.gy)), th = mu(ad(gxx, gyy), E.inv_DI);
        A8 = fm(x4, ad(gxx, -th), mu(mu(2.f, uy), sh));
        A9 = fm(y4, ad(gyy, -th), mu(mu(2.f, ux), sh));
    } else {
        const float sh = mu(dyx, E.gx), th = mu(gxx, E.inv_DI);
        A8 = fm(mu(2.f, uy), sh, mu(x4, fm(dxx, E.gx, -th)));
        A9 = fm(mu(2.f, ux), sh, mu(y4, -th));
    }
}
// w of a_hat; c: A8c or A9c
__device__ __forceinline__ double a_weight(double pT, double) { return pT; }
__device__ __forceinline__ float a_weight(float pT, float c) { return mu(pT, c); }

// The NND flux difference over c from three neighbouring differences around the upwind one:
// dc + (mm(dc, dr) - mm(dl, dc)) / 2 for v > 0, dc - (mm(dc, dr) - mm(dl, dc)) / 2 for v < 0
__device__ __forceinline__ double nnd3(double dl, double dc, double dr, bool neg)
{
    return fm(neg ? -0.5 : 0.5, ad(mm64(dc, dr), -mm64(dl, dc)), dc);
}
__device__ __forceinline__ float nnd3(float dl, float dc, float dr, bool neg)
{
    return fm(neg ? -0.5f : 0.5f, sgnmul(ad(mmag(dc, dr), -mmag(dl, dc)), dc), dc);
}

// ---- staging of a tile with its halo -----------------------------------------
// one element by an asynchronous copy
__device__ __forceinline__ void cp1(float* dst, const float* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp1(double* dst, const double* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Where a staged column (or row) at position j of an axis with n cells comes from: its index
// in the grid, or, beyond a Dirichlet side, -1 - side. Beyond a specular side: the mirror.
__device__ __forceinline__ int source(int j, int n, const int32_t* sbc, int side0, bool& mirrored)
{
    mirrored = false;
    if (j >= 0 && j < n) return j;
    const int s = side0 + (j < 0 ? 0 : 1), code = sbc[s];
    if (code == 3) return -1 - s;
    if (code == 4) {
        mirrored = true;
        j = j < 0 ? -j - 1 : 2 * n - 1 - j;
    }
    return map_index(j, n, code == 0 ? 0 : 1);
}

// Stages rows y0 .. y0 + SH - 1 and columns x0 .. x0 + 31 + EXTRA of all NPL planes, row r by
// warp r % TW: lane c copies the columns c and 32 + c. Sources that lie in the grid (all but
// Dirichlet ghosts) arrive asynchronously; `mirror(p)` is the plane whose v_y is reversed. A
// row without Dirichlet ghosts takes the branch-free loop.
template <int NPL, int SH, int SW, int TW, bool TWO_D, typename R, typename Mirror>
__device__ __forceinline__ void stage_tile(const R* __restrict__ in, R* sf, int x0, int y0, int nx, int ny,
                                           int pitch, int64_t plane, const int32_t* sides, const R (*sfeq)[NPL],
                                           Mirror mirror)
{
    constexpr int PS = SH * SW, EXTRA = SW - 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    bool m_;
    const int c0 = source(x0 + lane, nx, sides, 0, m_);
    const int c1 = lane < EXTRA ? source(x0 + 32 + lane, nx, sides, 0, m_) : 0;
    const bool inside = __all_sync(0xffffffffu, c0 >= 0 && c1 >= 0);
    for (int r = warp; r < SH; r += TW) {
        bool mir = false;
        const int gy = TWO_D ? source(y0 + r, ny, sides, 2, mir) : 0;
        R* dst = sf + r * SW + lane;
        const R* src = in + (int64_t)(gy < 0 ? 0 : gy) * pitch;
        if (inside && gy >= 0 && !mir) {
            const R *s0 = src + c0, *s1 = src + c1;
#pragma unroll
            for (int p = 0; p < NPL; p++) {
                cp1(dst + p * PS, s0);
                s0 += plane;
            }
            if (lane < EXTRA) {
#pragma unroll
                for (int p = 0; p < NPL; p++) {
                    cp1(dst + p * PS + 32, s1);
                    s1 += plane;
                }
            }
            continue;
        }
        const int g0 = gy < 0 ? gy : c0, g1 = gy < 0 ? gy : c1; // a Dirichlet row: all of it
#pragma unroll 1
        for (int p = 0; p < NPL; p++) {
            const R* sp = src + (mir ? mirror(p) : p) * plane;
            if (g0 >= 0) cp1(dst + p * PS, sp + g0);
            else dst[p * PS] = sfeq[-1 - g0][p];
            if (lane < EXTRA) {
                if (g1 >= 0) cp1(dst + p * PS + 32, sp + g1);
                else dst[p * PS + 32] = sfeq[-1 - g1][p];
            }
        }
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

// rho, u, T of one FP32 cell: exact conserved sums, then FP64 (REC = 0) or double-float (REC = 1
// normalised throughout, REC = 2 one correction per quotient); ig = T > T_ig in that precision,
// ok = rho, T > 0 and everything finite
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
        if constexpr (REC == 2) { // quotients of the sums with one correction, as recover_pair_df
            const float q = rcp_approx(m1.hi);
            auto quot = [&](S1 a) -> S1 {
                const float x = __fmul_rn(a.hi, q);
                float e = __fmaf_rn(-m1.hi, x, a.hi);
                e = __fadd_rn(e, __fmaf_rn(-m1.lo, x, a.lo));
                return s_norm({x, __fmul_rn(e, q)});
            };
            auto sqr = [](S1 a) -> S1 {
                const float p = __fmul_rn(a.hi, a.hi);
                return s_norm({p, __fmaf_rn(__fmul_rn(2.f, a.hi), a.lo, __fmaf_rn(a.hi, a.hi, -p))});
            };
            const S1 vx = quot(m2), vy = quot(m3), e = quot(m4);
            const S1 w = s_norm(s_add(sqr(vx), sqr(vy)));
            const S1 tt = s_norm(s_mul(s_norm(s_sub(e, w)), K.idh, K.idl));
            rho = m1.hi;
            ux = vx.hi;
            uy = vy.hi;
            T = tt.hi;
            ig = T > K.tigh || (T == K.tigh && tt.lo > K.tigl);
            ok = rho > 0.f && T > 0.f && T <= FLT_MAX && fabsf(ux) <= FLT_MAX && fabsf(uy) <= FLT_MAX;
            return;
        }
        double u, v, t;
        const double r = pair_to_f64(m1.hi, m1.lo);
        recover_one_f64_fast(m1.hi, m1.lo, r, pair_to_f64(m2.hi, m2.lo), pair_to_f64(m3.hi, m3.lo),
                             pair_to_f64(m4.hi, m4.lo), K.inv_DId, u, v, t);
        rho = m1.hi;
        ux = m2.hi == 0.f ? 0.f : d2f_fast(u); // (f2d_fast(0) is 2^-127)
        uy = m3.hi == 0.f ? 0.f : d2f_fast(v);
        T = d2f_fast(t);
        ig = dbits(t) > dbits(K.T_igd);
        ok = fabsf(m1.hi) <= FLT_MAX && fabsf(m2.hi) <= FLT_MAX && fabsf(m3.hi) <= FLT_MAX &&
             fabsf(m4.hi) <= FLT_MAX && m1.hi > 0.f && dbits(t) > 0 && dbits(t) <= dbits(DBL_MAX);
    }
}

// rho, u, T of one FP64 cell from its butterflies (Eqs. (5)-(7)); ok: rho, T > 0 and finite.
// AXIS_FIRST: the momenta of the axis orbits are added before the diagonal ones (the 2-D step), else
// in the orbits' order
template <bool AXIS_FIRST = false>
__device__ __forceinline__ void recover64(const ModelConst<double>& K, const Fly<double>& b, double& m1,
                                          double& m2, double& m3, double& ux, double& uy, double& ux2,
                                          double& uy2, double& u2, double& T, bool& ok)
{
    m1 = (b.P0 + b.P2) + (b.e1 + b.e3);
    constexpr int s = AXIS_FIRST ? 2 : 1, t = 3 - s; // the second and third orbit
    m2 = fm(K.cd[3], b.ax3, fm(K.cd[t], t == 1 ? b.ax1 : b.ax2, fm(K.cd[s], s == 1 ? b.ax1 : b.ax2, mu(K.cd[0], b.ax0))));
    m3 = fm(K.cd[3], b.ay3, fm(K.cd[t], t == 1 ? b.ay1 : b.ay2, fm(K.cd[s], s == 1 ? b.ay1 : b.ay2, mu(K.cd[0], b.ay0))));
    const double m4 = fm(K.wd[3], b.e3, fm(K.wd[1], b.e1, fm(K.wd[2], b.P2, mu(K.wd[0], b.P0))));
    const double q = recip64(m1);
    ux = mu(m2, q);
    uy = mu(m3, q);
    ux2 = mu(ux, ux);
    uy2 = mu(uy, uy);
    u2 = ad(ux2, uy2);
    T = mu(fm(m4, q, -u2), K.inv_DId);
    const long long tb = dbits(T), big = dbits(DBL_MAX);
    ok = dbits(m1) > 0 && dbits(m1) <= big && tb > 0 && tb <= big;
}

template <typename R>
inline void step_const(const ModelConst<R>& K, StepConst<R>* E)
{
    for (int j = 0; j < 4; j++) {
        E->h2[j] = R(0.5) * K.Bes[8 + j];
        E->h3[j] = R(0.5) * K.Bes[12 + j];
        E->ha[j] = R(0.5) * K.Bea[j];
        E->cdx[j] = K.c[j] * K.inv_dx;
        E->cdy[j] = K.c[j] * K.inv_dy;
    }
    E->c8 = K.A8c;
    E->c9 = K.A9c;
    E->gx = K.half_inv_dx;
    E->gy = K.half_inv_dy;
    E->inv_DI = K.inv_DI;
    E->dtdx = K.dt * K.inv_dx;
    E->dtdy = K.dt * K.inv_dy;
    E->di2 = K.DI + R(2);
    E->di4 = K.DI + R(4);
    E->a_hat = K.A8c != R(0) || K.A9c != R(0);
}

} // namespace lbk
