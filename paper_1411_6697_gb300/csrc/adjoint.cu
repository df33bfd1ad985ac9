// adjoint.cu -- discrete adjoint of the FP64 1-D step (reverse mode, hand-written).
//
// For one step (f, lambda)_n -> (f, lambda)_{n+1} of the fused kernel and adjoints
// (fb, lb)_{n+1} = dJ/d(state_{n+1}), these kernels produce (fb, lb)_n and add the
// step's contributions to dJ/dS_5..16, dJ/dQ, dJ/domega1, dJ/domega2. The forward
// values are recomputed from the stored FP64 state n (for an FP32 forward run, a state of
// the FP64 segment recomputed from the run's checkpoint, widened by adj_widen). Conventions at non-smooth points: the
// ignition switch T > T_ig is a hard switch (no derivative), minmod follows the
// branch the values select (a on a tie), the clamp of lambda passes the
// derivative when the unclamped value lies in [0, 1] (inclusive), the upwind
// choice for u.grad(lambda) by the sign of u has no derivative.
//
// adj_reverse runs several reverse steps per launch, one thread per cell; a launch replaces two
// kernels (and one that recovered the macroscopic fields) per step, whose FP64 unit did the
// stencils' transposes as products with stored coefficients, the branch tests, and a block
// reduction of 16 sums per step. Gradient of an 8192-cell detonation over 256 steps, checkpoints
// every 64: 40.5 -> 13.9 ms.
#include <float.h>
#include <math.h>

#include "adjoint.cuh"
#include "cellops.cuh"
#include "kernels.cuh"

namespace lbk {

namespace {

constexpr int ADJ_THREADS = 128;

// The increment of lambda over dt (Eq. (28), m = n = 1: the closed form of
// d lambda/dt = (1 - lambda)(a + b lambda), evaluated as the step evaluates it) and its
// partial derivatives with respect to lambda, a = omega1 p and b = omega2 p. With
// mu0 = 1 - lambda, k = a + b, e = exp(-k dt): mu = k mu0 e / (k - b mu0 (1 - e)) and
// dl = mu0 - mu; for b = 0, mu = mu0 e, whose derivative in b is the limit b -> 0.
__device__ __forceinline__ void reaction_partials(double lam, double a, double b, double dt,
                                                  double& dl, double& d_lam, double& d_a,
                                                  double& d_b)
{
    const double mu0 = 1.0 - lam;
    if (b == 0.0) {
        const double g = -expm1(-a * dt), e = 1.0 - g;
        const double ga = a > 0.0 ? g / a : dt; // (1 - e) / a
        dl = mu0 * g;
        d_lam = -g;
        d_a = mu0 * dt * e;
        d_b = mu0 * e * dt - mu0 * mu0 * e * ga;
        return;
    }
    const double k = a + b, e = exp(-k * dt), g = 1.0 - e;
    const double Dn = k - b * mu0 * g;
    const double mu = k * mu0 * e / Dn;
    const double mu_k = (mu0 * e * (1.0 - k * dt) - mu * (1.0 - b * mu0 * dt * e)) / Dn;
    const double mu_m0 = (k * e + mu * b * g) / Dn;
    dl = mu0 - mu;
    d_lam = mu_m0 - 1.0;
    d_a = -mu_k;
    d_b = -(mu_k + mu * mu0 * g / Dn);
}

// block sum of v in fixed order, added by thread 0 to acc[blockIdx.x]
__device__ void block_add(double v, double* acc, double* sred)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sred[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < ADJ_THREADS / 32; k++) s += sred[k];
        acc[blockIdx.x] += s;
    }
}

// ---- the reverse sweep ------------------------------------------------------------
constexpr int REV_THREADS = 128;  // most threads of a block
constexpr int NSLOT = 13;         // planes that move along x: six v_x > 0, six v_x < 0, lambda
// plane of a slot (16: lambda) and slot of a plane (-1: v_x = 0), as in the forward step
__host__ __device__ constexpr int slot_plane(int s)
{
    constexpr int t[NSLOT] = {0, 4, 7, 8, 12, 15, 2, 5, 6, 10, 13, 14, 16};
    return t[s];
}
__host__ __device__ constexpr int slot_of(int plane)
{
    constexpr int t[16] = {0, -1, 6, -1, 1, 7, 8, 2, 3, -1, 9, -1, 4, 10, 11, 5};
    return t[plane];
}

struct AdjConst {
    double ies[16], iea[4], iodd[16], ioo[4]; // dt M^-1 in blocks
    double half[4];                           // dt c / (2 dx) of each orbit
    double dtdx, gx;                          // dt / dx, 1 / (2 dx)
    double c8, c9, k8a, k8b, k9a, k9b;        // A8c, A9c; dA8c/dS_5, dA8c/dS_8, dA9c/dS_7, dA9c/dS_9
    double di2, di4, i1;                      // D + I + 2, D + I + 4, 1 / (D + I)
    double tw2;                               // 2 w_tne dx dt
};

// the branches of minmod(a, b): bit 0 the first argument is taken, bit 1 the second (the first
// on a tie, none unless the signs agree and neither vanishes)
__device__ __forceinline__ unsigned branch(double a, double b)
{
    const unsigned long long ia = (unsigned long long)dbits(a), ib = (unsigned long long)dbits(b);
    const unsigned long long m = 0x7fffffffffffffffull, ma = ia & m, mb = ib & m;
    if ((long long)(ia ^ ib) < 0 || ma == 0 || mb == 0) return 0u;
    return ma <= mb ? 1u : 2u;
}
// a small integer (|k| <= 4) as a double, without the conversion unit
__device__ __forceinline__ double small(int k)
{
    const int m = k < 0 ? -k : k;
    const unsigned hi16 = m == 4 ? 0x4010u : (unsigned)(0x400840003ff00000ull >> (16 * m)) & 0xffffu;
    return __hiloint2double((int)((hi16 << 16) | (k < 0 ? 0x80000000u : 0u)), 0);
}
// Twice the NND difference's derivative with respect to the value at offset o of its stencil:
// for v > 0 from the branches (a01, b01, a12, b12), for v < 0 from (a12, b12, a23, b23), packed
// as bits 0..3 of c. With P = 1 + (a12 - b01)/2 for v > 0 the weights at offsets -2..1 are a01/2,
// -P - a01/2, P - b12/2, b12/2; with P = 1 + (b12 - a23)/2 for v < 0 those at -1..2 are -a12/2,
// a12/2 - P, P + b23/2, -b23/2.
__device__ __forceinline__ int weight(unsigned c, bool neg, int o)
{
    const int a = c & 1, b = (c >> 1) & 1, e = (c >> 2) & 1, f = (c >> 3) & 1;
    if (!neg) {
        const int P = 2 + e - b;
        return o == -2 ? a : (o == -1 ? -P - a : (o == 0 ? P - f : (o == 1 ? f : 0)));
    }
    const int P = 2 + b - e;
    return o == -1 ? -a : (o == 0 ? a - P : (o == 1 ? P + f : (o == 2 ? -f : 0)));
}

// `steps` reverse steps in one launch. A block holds a window of cells, one per thread, with
// their adjoints (fb, lb) in registers; each step reads the stored state it reverses, forms
// everything local to a cell (the transposes of the back-transform, relaxation, A_hat, reaction,
// chemical term, equilibrium and lambda update), leaves its weighted stencil branches and the
// adjoints of the velocity gradients in shared memory for the neighbours to gather, and applies
// the transposes of the recovery and of M. A cell's new adjoint needs stencils two cells away,
// which need states four cells away: of the window all but 2 + 2 s cells at either end are right
// after s steps, and the block's own are those that still are after the launch. The parameter
// sums run in registers over the launch, so their block reductions cost one in `steps`.
//
// FP64 throughout and bound by its unit (cellops.cuh): branches travel as bits, a stencil's
// transpose is one FMA with a small integer per neighbour, and the reaction's part runs only in
// warps with an ignited cell.
__global__ void __launch_bounds__(REV_THREADS)
    adj_reverse(const __grid_constant__ ModelConst<double> K, const __grid_constant__ StepConst<double> E,
                const __grid_constant__ AdjConst A, const __grid_constant__ AdjReverse a, int kmax)
{
    extern __shared__ __align__(16) double sm[];
    const int n = blockDim.x, t = threadIdx.x, h = 2 * kmax + 2, own = n - 2 * h;
    double* pub = sm;                  // [NSLOT + 2][n]: moving planes, lambda, u_x, u_y
    double* dif = pub + 15 * n;        // [NSLOT][n]: differences to the right neighbour
    double* tw = dif + NSLOT * n;      // [NSLOT + 2][n]: stencil weights, adjoints of grad u
    double* fold = tw + 15 * n;        // [15][4]: what falls on ghost cells of zero-gradient ends
    double* red = fold + 60;           // [warps]
    unsigned* code = reinterpret_cast<unsigned*>(red + REV_THREADS / 32); // [2][n]: branches

    const int nx = K.nx;
    const int x0 = blockIdx.x * own - h, x = x0 + t;
    const bool per = K.bc_x == 0;
    const bool dom = per || (x >= 0 && x < nx);
    int gx = x;
    if (per) {
        gx = x % nx;
        gx = gx < 0 ? gx + nx : gx;
    } else {
        gx = x < 0 ? 0 : (x >= nx ? nx - 1 : x);
    }
    const bool mine = t >= h && t < h + own && x >= 0 && x < nx;
    const bool edge = !per && (x0 < 0 || x0 + n > nx); // block-uniform
    const int l1 = t >= 1 ? t - 1 : 0, l2 = t >= 2 ? t - 2 : 0;
    const int r1 = t + 1 < n ? t + 1 : n - 1, r2 = t + 2 < n ? t + 2 : n - 1;

    double fb[16], lb, pS[ADJ_NPAR], jt = 0.0;
#pragma unroll
    for (int i = 0; i < 16; i++) fb[i] = a.fb1[(size_t)i * nx + gx];
    lb = a.lb1[gx];
#pragma unroll
    for (int q = 0; q < ADJ_NPAR; q++) pS[q] = 0.0;

    for (int s = 0; s < a.steps; s++) {
        const double* st = a.state - s * a.stride + gx;
        double f[16];
#pragma unroll
        for (int i = 0; i < 16; i++) f[i] = st[i * K.plane];
        const double lam = st[16 * K.plane];
        const Fly<double> b = butterflies(f);
        double m1, m2, m3, ux, uy, ux2, uy2, u2, T;
        bool ok;
        recover64(K, b, m1, m2, m3, ux, uy, ux2, uy2, u2, T, ok);
#pragma unroll
        for (int k = 0; k < NSLOT; k++) pub[k * n + t] = slot_plane(k) == 16 ? lam : f[slot_plane(k) & 15];
        pub[13 * n + t] = ux;
        pub[14 * n + t] = uy;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < NSLOT; k++) dif[k * n + t] = pub[k * n + r1] - pub[k * n + t];
        const double gxx = mu(pub[13 * n + r1] - pub[13 * n + l1], A.gx);
        const double gyx = mu(pub[14 * n + r1] - pub[14 * n + l1], A.gx);
        const double pT = mu(m1, T), rinv = recip64(m1);
        double D[TNE_K];
        deltas<true>(K, E, b, m1, m2, m3, ux, uy, ux2, uy2, u2, T, pT, D);
        __syncthreads();

        // stencil weights: t = -(dt v / 2 dx) fb for f_i, the branches as bits
        unsigned c0 = 0u, c1 = 0u;
        const bool uneg = dbits(ux) < 0;
        double lsel;
#pragma unroll
        for (int k = 0; k < NSLOT; k++) {
            const double* d = dif + k * n;
            const bool neg = k < 12 ? k >= 6 : uneg;
            const double dl = d[neg ? l1 : l2], dc = d[neg ? t : l1], dr = d[neg ? r1 : t];
            const unsigned c = branch(dl, dc) | branch(dc, dr) << 2;
            if (k < 8) c0 |= c << (4 * k);
            else c1 |= c << (4 * (k - 8));
            if (k < 12) {
                const int p = slot_plane(k) & 15;
                tw[k * n + t] = dom ? mu(neg ? A.half[p >> 2] : -A.half[p >> 2], fb[p]) : 0.0;
            } else {
                lsel = (dbits(ux) << 1) == 0 ? 0.0 : nnd3(dl, dc, dr, neg);
            }
        }
        if (uneg) c1 |= 1u << 20;
        code[t] = c0;
        code[n + t] = c1;

        // the adjoint of Omega_hat: M^-T (dt fb) in block form
        double Om[16];
        {
            double pes[4], pea[2], px[4], py[4], po[2];
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const double pp = ad(fb[8 * q], fb[8 * q + 2]), pm = ad(fb[8 * q + 1], fb[8 * q + 3]);
                px[q] = ad(fb[8 * q], -fb[8 * q + 2]);
                py[q] = ad(fb[8 * q + 1], -fb[8 * q + 3]);
                pes[q] = ad(pp, pm);
                pea[q] = ad(pp, -pm);
                const double f0 = fb[4 + 8 * q], f1 = fb[5 + 8 * q], f2 = fb[6 + 8 * q], f3 = fb[7 + 8 * q];
                const double eo = ad(f0, f2), xp = ad(f0, -f2), em = ad(f1, f3), xm = ad(f3, -f1);
                pes[2 + q] = ad(eo, em);
                po[q] = ad(eo, -em);
                px[2 + q] = ad(xp, xm);
                py[2 + q] = ad(xp, -xm);
            }
            auto col = [](const double* B, int c, const double* v) {
                return fm(B[12 + c], v[3], fm(B[8 + c], v[2], fm(B[4 + c], v[1], mu(B[c], v[0]))));
            };
            const double e2 = col(A.ies, 2, pes), e3 = col(A.ies, 3, pes);
            const double a0 = fm(A.iea[2], pea[1], mu(A.iea[0], pea[0])), a1 = fm(A.iea[3], pea[1], mu(A.iea[1], pea[0]));
            Om[3] = col(A.ies, 1, pes);
            Om[4] = ad(e2, a0);
            Om[6] = ad(e2, -a0);
            Om[13] = ad(e3, a1);
            Om[15] = ad(e3, -a1);
            Om[7] = col(A.iodd, 1, px);
            Om[9] = col(A.iodd, 2, px);
            Om[11] = col(A.iodd, 3, px);
            Om[8] = col(A.iodd, 1, py);
            Om[12] = col(A.iodd, 2, py);
            Om[10] = col(A.iodd, 3, py);
            Om[5] = fm(A.ioo[2], po[1], mu(A.ioo[0], po[0]));
            Om[14] = fm(A.ioo[3], po[1], mu(A.ioo[1], po[0]));
        }
        // reaction over dt (Eq. (28)) and its derivatives, in warps with an ignited cell
        const bool ig = dbits(T) > dbits(K.T_igd), react = __any_sync(0xffffffffu, ig);
        double dl = 0.0, dl_lam = 0.0, dl_a = 0.0, dl_b = 0.0;
        if (react && ig) reaction_partials(lam, K.omega1 * pT, K.omega2 * pT, K.dt, dl, dl_lam, dl_a, dl_b);
        const double raw = ad(fm(mu(-A.dtdx, ux), lsel, dl), lam);
        const bool pass = (dbits(raw) >= 0 && dbits(raw) <= dbits(1.0)) || dbits(raw) == (long long)0x8000000000000000ull;
        const double lbc = pass ? lb : 0.0;
        tw[12 * n + t] = dom ? mu(mu(-0.5 * A.dtdx, ux), lbc) : 0.0;
        double rhob = 0.0, Tb = 0.0, lamb = lbc;
        double uxb = mu(mu(-A.dtdx, lsel), lbc), uyb = 0.0;
        if (react) {
            const double dA = fm(2.0 * A.di2, T, u2), xy = mu(ux, uy);
            // sum of d f_hat^eq / dT times the adjoint, over rho
            double cb = fm(K.DI, Om[3], ad(Om[4], Om[6]));
            cb = fm(ux, fm(A.di2, Om[7], fm(3.0, Om[9], Om[11])), cb);
            cb = fm(uy, fm(A.di2, Om[8], fm(3.0, Om[12], Om[10])), cb);
            cb = fm(fm(ux2, A.di4, dA), Om[13], cb);
            cb = fm(mu(xy, A.di4), Om[14], cb);
            cb = fm(fm(uy2, A.di4, dA), Om[15], cb);
            const double crb = mu(m1, cb), cr = mu(dl, K.chem), rc = mu(m1, cr);
            const double s2 = mu(2.0, ad(Om[13], Om[15]));
            rhob = mu(cr, cb);
            uxb = fm(rc, fm(A.di2, Om[7], fm(3.0, Om[9], ad(Om[11], fm(mu(uy, A.di4), Om[14],
                          fm(mu(mu(2.0, ux), A.di4), Om[13], mu(ux, s2)))))), uxb);
            uyb = mu(rc, fm(A.di2, Om[8], fm(3.0, Om[12], ad(Om[10], fm(mu(ux, A.di4), Om[14],
                          fm(mu(mu(2.0, uy), A.di4), Om[15], mu(uy, s2)))))));
            Tb = mu(mu(rc, s2), A.di2);
            const double dlb = fm(K.chem, crb, lbc), ab = mu(dl_a, dlb), bb = mu(dl_b, dlb);
            lamb = fm(dl_lam, dlb, lamb);
            const double pb = fm(K.omega1, ab, mu(K.omega2, bb));
            rhob = fm(T, pb, rhob);
            Tb = fm(m1, pb, Tb);
            if (mine) {
                pS[12] = fm(mu(dl, 2.0 / (K.DI * K.dt)), crb, pS[12]);
                pS[13] = fm(pT, ab, pS[13]);
                pS[14] = fm(pT, bb, pS[14]);
            }
        }
        // A_hat_8 = rho T A8c X8, A_hat_9 = rho T A9c X9 (Eqs. (3)-(4))
        double gxb, gyb;
        {
            const double p8 = mu(4.0 * (1.0 - A.i1), gxx), p9 = mu(-4.0 * A.i1, gxx), g2 = mu(2.0, gyx);
            const double X8 = fm(ux, p8, mu(uy, g2)), X9 = fm(uy, p9, mu(ux, g2));
            const double y8 = mu(X8, Om[7]), y9 = mu(X9, Om[8]);
            const double z = fm(A.c8, y8, mu(A.c9, y9));
            rhob = fm(T, z, rhob);
            Tb = fm(m1, z, Tb);
            if (mine) {
                const double q8 = mu(pT, y8), q9 = mu(pT, y9);
                pS[0] = fm(A.k8a, q8, pS[0]);
                pS[3] = fm(A.k8b, q8, pS[3]);
                pS[2] = fm(A.k9a, q9, pS[2]);
                pS[4] = fm(A.k9b, q9, pS[4]);
            }
            const double w8 = mu(mu(pT, A.c8), Om[7]), w9 = mu(mu(pT, A.c9), Om[8]);
            uxb = fm(p8, w8, fm(g2, w9, uxb));
            uyb = fm(g2, w8, fm(p9, w9, uyb));
            gxb = fm(mu(4.0 * (1.0 - A.i1), ux), w8, mu(mu(-4.0 * A.i1, uy), w9));
            gyb = mu(2.0, fm(uy, w8, mu(ux, w9)));
        }
        tw[13 * n + t] = dom ? mu(gxb, A.gx) : 0.0;
        tw[14 * n + t] = dom ? mu(gyb, A.gx) : 0.0;
        // relaxation: Delta's adjoint and dJ/dS, then f_hat^eq's part with r = -rho Delta_b
        double Db[TNE_K];
#pragma unroll
        for (int k = 0; k < TNE_K; k++) {
            Db[k] = fm(-K.S[k + 4], Om[k + 4], mu(A.tw2, D[k]));
            if (mine) {
                pS[k] = fm(-D[k], Om[k + 4], pS[k]);
                jt = fm(D[k], D[k], jt);
            }
        }
        {
            const double Ta = ad(T, ux2), Tc = ad(T, uy2), Aa = fm(A.di2, T, u2), B = fm(2.0, T, Aa);
            const double c3 = fm(2.0, T, Ta), c4 = fm(2.0, T, Tc), xy = mu(ux, uy), AT = mu(Aa, T);
            // over rho: the equilibrium is linear in it
            double e = fm(Db[0], Ta, fm(Db[1], xy, mu(Db[2], Tc)));
            e = fm(ux, fm(Db[3], Aa, fm(Db[5], c3, mu(Db[7], Tc))), e);
            e = fm(uy, fm(Db[4], Aa, fm(Db[6], Ta, mu(Db[8], c4))), e);
            e = fm(Db[9], fm(ux2, B, AT), fm(mu(xy, B), Db[10], fm(Db[11], fm(uy2, B, AT), e)));
            rhob = ad(rhob, -e);
            // the other arguments, each adjoint still over -rho
            const double v9 = mu(Db[5], ux), v12 = mu(Db[8], uy);
            const double tab = ad(Db[0], fm(Db[6], uy, v9)), tcb = ad(Db[2], fm(Db[7], ux, v12));
            const double d1315 = ad(Db[9], Db[11]);
            const double bbq = fm(Db[9], ux2, fm(Db[10], xy, mu(Db[11], uy2)));
            const double aab = ad(fm(Db[3], ux, fm(Db[4], uy, mu(d1315, T))), bbq);
            double xb = fm(Db[1], uy, fm(Db[3], Aa, fm(Db[5], c3, mu(Db[7], Tc))));
            double yb = fm(Db[1], ux, fm(Db[4], Aa, fm(Db[6], Ta, mu(Db[8], c4))));
            const double x2 = mu(2.0, ux), y2 = mu(2.0, uy);
            xb = fm(B, fm(Db[9], x2, mu(Db[10], uy)), xb);
            yb = fm(B, fm(Db[11], y2, mu(Db[10], ux)), yb);
            xb = fm(x2, ad(aab, tab), xb);
            yb = fm(y2, ad(aab, tcb), yb);
            double tb = fm(2.0, ad(ad(v9, v12), bbq), mu(d1315, Aa));
            tb = ad(fm(A.di2, aab, tb), ad(tab, tcb));
            uxb = fm(-m1, xb, uxb);
            uyb = fm(-m1, yb, uyb);
            Tb = fm(-m1, tb, Tb);
        }
        __syncthreads(); // weights, branches and gradient adjoints of every cell are there

        // the transposed stencils: what the cells around leave at this one
        double G[NSLOT], ugx, ugy;
        {
            const unsigned w0[5] = {code[l2], code[l1], code[t], code[r1], code[r2]};
            const unsigned w1[5] = {code[n + l2], code[n + l1], code[n + t], code[n + r1], code[n + r2]};
            const int at[5] = {l2, l1, t, r1, r2}; // the cell at distance q - 2 reads this one at 2 - q
#pragma unroll
            for (int k = 0; k < NSLOT; k++) {
                double g = 0.0;
#pragma unroll
                for (int q = 0; q < 5; q++) {
                    const int o = 2 - q;
                    if (k < 12 && (k >= 6 ? o == -2 : o == 2)) continue;
                    const unsigned w = k < 8 ? w0[q] >> (4 * k) : w1[q] >> (4 * (k - 8));
                    const bool neg = k < 12 ? k >= 6 : (w1[q] >> 20) & 1u;
                    g = fm(small(weight(w & 15u, neg, o)), tw[k * n + at[q]], g);
                }
                G[k] = g;
            }
            ugx = tw[13 * n + l1] - tw[13 * n + r1];
            ugy = tw[14 * n + l1] - tw[14 * n + r1];
        }
        if (edge) { // what fell on the ghost cells of a zero-gradient end goes to the end cell
            const int gl = x < 0 && x >= -2 ? -1 - x : (x >= nx && x < nx + 2 ? 2 + x - nx : -1);
            if (gl >= 0) {
#pragma unroll
                for (int k = 0; k < NSLOT; k++) fold[k * 4 + gl] = G[k];
                fold[13 * 4 + gl] = ugx;
                fold[14 * 4 + gl] = ugy;
            }
            __syncthreads();
            for (int side = 0; side < 2; side++) {
                if (x != (side ? nx - 1 : 0)) continue;
                const double* c = fold + 2 * side;
#pragma unroll
                for (int k = 0; k < NSLOT; k++) G[k] += c[k * 4] + c[k * 4 + 1];
                ugx += c[13 * 4] + c[13 * 4 + 1];
                ugy += c[14 * 4] + c[14 * 4 + 1];
            }
        }
        uxb = ad(uxb, ugx);
        uyb = ad(uyb, ugy);
        // rho, u, T from the conserved moments, and M^T
        const double Eb = mu(Tb, A.i1);
        uxb = fm(mu(-2.0, ux), Eb, uxb);
        uyb = fm(mu(-2.0, uy), Eb, uyb);
        const double M1 = mu(rinv, uxb), M2 = mu(rinv, uyb), M3 = mu(rinv, Eb);
        const double M0 = ad(rhob, -fm(ux, M1, fm(uy, M2, mu(fm(K.DI, T, u2), M3))));
        {
            const double p2 = ad(Db[0], Db[2]), p3 = ad(Db[9], Db[11]), q0 = ad(Db[0], -Db[2]), q1 = ad(Db[9], -Db[11]);
            double es[4], ea[2], xo[4], yo[4], oo[2];
#pragma unroll
            for (int c = 0; c < 4; c++) {
                es[c] = fm(E.h3[c], p3, fm(E.h2[c], p2, fm(K.Bes[4 + c], M3, mu(K.Bes[c], M0))));
                xo[c] = fm(K.Bodd[12 + c], Db[7], fm(K.Bodd[8 + c], Db[5], fm(K.Bodd[4 + c], Db[3], mu(K.Bodd[c], M1))));
                yo[c] = fm(K.Bodd[12 + c], Db[6], fm(K.Bodd[8 + c], Db[8], fm(K.Bodd[4 + c], Db[4], mu(K.Bodd[c], M2))));
            }
#pragma unroll
            for (int c = 0; c < 2; c++) {
                ea[c] = fm(E.ha[2 + c], q1, mu(E.ha[c], q0));
                oo[c] = fm(K.Boo[2 + c], Db[10], mu(K.Boo[c], Db[1]));
            }
            auto join = [&](int i, double m) {
                const int k = slot_of(i);
                fb[i] = k >= 0 ? ad(ad(fb[i], m), G[k]) : ad(fb[i], m);
            };
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const double sx = ad(es[q], ea[q]), sy = ad(es[q], -ea[q]);
                join(8 * q, ad(sx, xo[q]));
                join(8 * q + 2, ad(sx, -xo[q]));
                join(8 * q + 1, ad(sy, yo[q]));
                join(8 * q + 3, ad(sy, -yo[q]));
                const double e = es[2 + q], ax = xo[2 + q], ay = yo[2 + q], o = oo[q];
                const double s01 = ad(e, ay), s23 = ad(e, -ay), d01 = ad(ax, o), d23 = ad(o, -ax);
                join(4 + 8 * q, ad(s01, d01));
                join(5 + 8 * q, ad(s01, -d01));
                join(6 + 8 * q, ad(s23, d23));
                join(7 + 8 * q, ad(s23, -d23));
            }
        }
        lb = ad(lamb, G[12]);
    }
    if (mine) {
#pragma unroll
        for (int i = 0; i < 16; i++) a.fb0[(size_t)i * nx + x] = fb[i];
        a.lb0[x] = lb;
    }
    // the launch's sums, in a fixed order
    auto add = [&](double v, double* acc) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        __syncthreads();
        if ((t & 31) == 0) red[t >> 5] = v;
        __syncthreads();
        if (t == 0) {
            double s = 0.0;
            for (int k = 0; k < n / 32; k++) s += red[k];
            acc[blockIdx.x] += s;
        }
    };
    for (int q = 0; q < ADJ_NPAR; q++) add(pS[q], a.pacc + (size_t)q * gridDim.x);
    add(jt * a.jw, a.jacc);
}

// dJ/df of the final state from J_mis = w/2 sum_x (rho - rho*)^2 dx (rho = sum_i f_i)
__global__ void __launch_bounds__(ADJ_THREADS)
    adj_seed(const ModelConst<double> K, const AdjArgs a, const double* rho_t, double w)
{
    __shared__ double sred[ADJ_THREADS / 32];
    const int nx = K.nx;
    double jm = 0.0;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nx; j += gridDim.x * blockDim.x) {
        double rho = 0.0;
        for (int i = 0; i < 16; i++) rho += a.f[i * K.plane + j];
        const double d = rho - rho_t[j];
        jm += 0.5 * w * d * d * K.dx_;
        for (int i = 0; i < 16; i++) a.fb0[i * nx + j] = w * d * K.dx_;
        a.lb0[j] = 0.0;
    }
    block_add(jm, a.jacc, sred);
}

// dJ/drho0 of an equilibrium start f0 = M^-1 f_hat^eq(rho0, u0, T0): f_hat^eq is
// linear in rho0, so dJ/drho0 = sum_k (M^-T fb0)_k (M f0)_k / rho0.
__global__ void __launch_bounds__(ADJ_THREADS)
    adj_rho0(const ModelConst<double> K, const AdjArgs a, double* drho0)
{
    const int nx = K.nx;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nx; j += gridDim.x * blockDim.x) {
        double f[16], m[16], fb[16];
        for (int i = 0; i < 16; i++) f[i] = a.f[i * K.plane + j], fb[i] = a.fb1[i * nx + j];
        forward_moments(K, f, m);
        double qb[16];
        inverse_moments_t(K, fb, qb);
        double s = 0.0;
        for (int k = 0; k < 16; k++) s += qb[k] * m[k];
        drho0[j] = s / m[0];
    }
}

// the objective's TNE term of one state alone: w_tne dx dt sum_x sum_k Delta_k^2, each Delta_k formed
// as the reverse sweep forms it
__global__ void __launch_bounds__(ADJ_THREADS)
    adj_jtne(const __grid_constant__ ModelConst<double> K, const __grid_constant__ StepConst<double> E, const AdjArgs a)
{
    __shared__ double sred[ADJ_THREADS / 32];
    const int nx = K.nx;
    double jt = 0.0;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nx; j += gridDim.x * blockDim.x) {
        double f[16], m1, m2, m3, ux, uy, ux2, uy2, u2, T, D[TNE_K];
        bool ok;
        for (int i = 0; i < 16; i++) f[i] = a.f[i * K.plane + j];
        const Fly<double> b = butterflies(f);
        recover64(K, b, m1, m2, m3, ux, uy, ux2, uy2, u2, T, ok);
        deltas<true>(K, E, b, m1, m2, m3, ux, uy, ux2, uy2, u2, T, mu(m1, T), D);
        for (int k = 0; k < TNE_K; k++) jt = fm(D[k], D[k], jt);
    }
    block_add(jt * a.jw, a.jacc, sred);
}

// an FP32 checkpoint widened to FP64, element by element (exact)
__global__ void adj_widen(const float* __restrict__ in, double* __restrict__ out, size_t n)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        out[i] = (double)in[i];
}

} // namespace

int adj_grid(int nx)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int need = (nx + ADJ_THREADS - 1) / ADJ_THREADS;
    const int cap = sms * 4;
    return need < cap ? need : cap;
}

// The cut of the reverse sweep: blocks of `threads` cells, 4 steps + 4 of them overlap. A step
// takes 24 us with up to three warps an SM, 25.5 with four, then 6 us a warp (the FP64 unit), a
// launch 8 us beside its steps. Gradient over 256 steps, ms: 8192 cells, 96 threads x 8 steps
// 14.6, 128 x 16 15.0, 32 x 1 17.8, 96 x 16 17.2 (two blocks on most SMs); 300 cells 96 x 16
// 13.5, 64 x 1 16.6; 20000 cells 96 x 4 19.6, 128 x 16 26.5.
AdjPlan adj_plan(int nx)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 152;
    AdjPlan best = {128, 1, (nx + 119) / 120};
    double t_best = 1e300;
    for (int threads = 32; threads <= REV_THREADS; threads += 32)
        for (int steps = 1; steps <= 16; steps *= 2) {
            const int own = threads - 4 * steps - 4;
            if (own < 16) continue;
            const int grid = (nx + own - 1) / own;
            const double w = (double)((grid + sms - 1) / sms) * (threads / 32);
            const double t = (w > 4.25 ? 6.0 * w : (w > 3.25 ? 25.5 : 24.0)) + 8.0 / steps;
            if (t < t_best) t_best = t, best = {threads, steps, grid};
        }
    return best;
}

cudaError_t launch_adj_reverse(const ModelConst<double>& K, const AdjReverse& a, const AdjPlan& p, double tne_w,
                               cudaStream_t s)
{
    if (a.steps < 1 || a.steps > p.steps) return cudaErrorInvalidValue;
    StepConst<double> E;
    step_const(K, &E);
    AdjConst A;
    for (int k = 0; k < 16; k++) {
        A.ies[k] = K.dt * K.Ies[k];
        A.iodd[k] = K.dt * K.Iodd[k];
    }
    for (int k = 0; k < 4; k++) {
        A.iea[k] = K.dt * K.Iea[k];
        A.ioo[k] = K.dt * K.Ioo[k];
        A.half[k] = 0.5 * K.dt * K.c[k] * K.inv_dx;
    }
    A.dtdx = K.dt * K.inv_dx;
    A.gx = K.half_inv_dx;
    A.c8 = K.A8c;
    A.c9 = K.A9c;
    A.k8a = K.S[7] / (K.S[4] * K.S[4]);
    A.k8b = -1.0 / K.S[4];
    A.k9a = K.S[8] / (K.S[6] * K.S[6]);
    A.k9b = -1.0 / K.S[6];
    A.di2 = K.DI + 2.0;
    A.di4 = K.DI + 4.0;
    A.i1 = 1.0 / K.DI;
    A.tw2 = 2.0 * tne_w;
    const size_t bytes = sizeof(double) * ((size_t)(15 + NSLOT + 15) * p.threads + 60 + REV_THREADS / 32) +
                         sizeof(unsigned) * 2 * p.threads;
    static cudaError_t done = cudaFuncSetAttribute(
        adj_reverse, cudaFuncAttributeMaxDynamicSharedMemorySize,
        (int)(sizeof(double) * ((15 + NSLOT + 15) * REV_THREADS + 60 + REV_THREADS / 32) + sizeof(unsigned) * 2 * REV_THREADS));
    if (done != cudaSuccess) return done;
    adj_reverse<<<p.grid, p.threads, bytes, s>>>(K, E, A, a, p.steps);
    return cudaGetLastError();
}

cudaError_t launch_adj_seed(const ModelConst<double>& K, const AdjArgs& a, const double* rho_t,
                            double w, int grid, cudaStream_t s)
{
    adj_seed<<<grid, ADJ_THREADS, 0, s>>>(K, a, rho_t, w);
    return cudaGetLastError();
}

cudaError_t launch_adj_jtne(const ModelConst<double>& K, const AdjArgs& a, int grid, cudaStream_t s)
{
    StepConst<double> E;
    step_const(K, &E);
    adj_jtne<<<grid, ADJ_THREADS, 0, s>>>(K, E, a);
    return cudaGetLastError();
}

cudaError_t launch_adj_widen(const float* in, double* out, size_t n, int grid, cudaStream_t s)
{
    adj_widen<<<grid, ADJ_THREADS, 0, s>>>(in, out, n);
    return cudaGetLastError();
}

cudaError_t launch_adj_rho0(const ModelConst<double>& K, const AdjArgs& a, double* drho0,
                            int grid, cudaStream_t s)
{
    adj_rho0<<<grid, ADJ_THREADS, 0, s>>>(K, a, drho0);
    return cudaGetLastError();
}

} // namespace lbk
