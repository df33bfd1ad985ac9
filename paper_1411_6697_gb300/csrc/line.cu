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
// everything that can leave that unit does (cellops.cuh); each difference of neighbouring
// cells is formed once and exchanged: 298 FP64 instructions per warp and step (ncu, 16384-cell
// detonation). FP32: the latency of one warp's chain of about 900 instructions; the conserved
// sums are exact double-floats, which keeps all but 8 FP64 instructions off that unit.
//
// Measured per step, against one launch per step of a tile kernel with the plain formulas
// (every stencil's differences, FP64 minmod and FP64 sums of an FP32 state): Sod tube of 400
// cells FP64 29.8 -> 11.7 us (6.8 with four warps to a window, below); detonation of 16384 cells
// FP32 13.3 -> 2.0 us, FP64 with records at every step 58.9 -> 24.9 us.
//
// Boundaries: lanes past a zero-gradient end are read through the index of the end cell,
// lanes past a Dirichlet end hold the side's equilibrium, and on a periodic grid every lane
// stands for the cell its position wraps to.
#include <float.h>

#include "cellops.cuh"
#include "line.cuh"

namespace lbk {

namespace {

constexpr int NMOVE = 12;          // planes with v_x != 0
constexpr int NX = NMOVE + 1;      // and lambda: what neighbours read
constexpr int LINE_THREADS = 256; // threads of a block

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
    line_kernel(const __grid_constant__ ModelConst<R> K, const __grid_constant__ StepConst<R> E,
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
        R m1, m2, m3, ux, uy, T, A8 = R(0), A9 = R(0);
        bool hot; // the cell reacts; a burnt one adds nothing
        const Fly<R> b = butterflies(f);
        R* P = sizeof(R) == 4 && (s & 1) ? dif : pub; // what this step publishes
        R ux2, uy2, u2;
        if constexpr (sizeof(R) == 8) {
            bool ok;
            recover64(K, b, m1, m2, m3, ux, uy, ux2, uy2, u2, T, ok);
            if (mine && !ok) bad = 1;
            hot = dbits(T) > dbits(K.T_igd) && dbits(lam) != dbits(1.0);
        } else {
            bool ok;
            recover32<REC>(K, f, m1, ux, uy, T, hot, ok);
            if (mine && !ok) bad = 1;
            hot = hot && lam != 1.f;
            m2 = mu(m1, ux);
            m3 = mu(m1, uy);
            ux2 = mu(ux, ux);
            uy2 = mu(uy, uy);
            u2 = fm(ux, ux, uy2);
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
        if (E.a_hat)
            a_hat<false>(E, ux, uy, P[NX * n + jp1] - P[NX * n + jm1], P[(NX + 1) * n + jp1] - P[(NX + 1) * n + jm1],
                  R(0), R(0), A8, A9);
        R D[TNE_K], W[16];
        const R pT = mu(m1, T);
        deltas<true>(K, E, b, m1, m2, m3, ux, uy, ux2, uy2, u2, T, pT, D);
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
        collide<true>(K, E, K.S, D, m1, m2, m3, ux, uy, u2, T, a_weight(pT, E.c8), a_weight(pT, E.c9), A8, A9, react,
                mu(dlam, K.chem), W);
        // NND differences (v > 0 from d_{j-2}, d_{j-1}, d_j; v < 0 from d_{j-1}, d_j, d_{j+1};
        // d_j = q_{j+1} - q_j) and the Euler update; lambda's side by the sign of u_x
        if constexpr (sizeof(R) == 8) __syncthreads();
        auto nnd = [&](int k, R q, bool neg) -> R {
            if constexpr (sizeof(R) == 8) {
                const double* d = dif + k * n;
                return nnd3(d[neg ? dm1 : dm2], d[neg ? t : dm1], d[neg ? dp1 : t], neg);
            } else {
                const float* r = P + k * n;
                const float l = r[jm1], g = r[jp1];
                return neg ? nnd3(q - l, g - q, r[jp2] - g, true) : nnd3(l - r[jm2], q - l, g - q, false);
            }
        };
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const int k = slot_of(i);
            const R c = k >= 6 ? E.cdx[i >> 2] : -E.cdx[i >> 2];
            if (k >= 0) { // (FP32: the diagonal orbits' flux is rounded first, as with both axes)
                const R X = nnd(k, f[i], k >= 6);
                W[i] = sizeof(R) == 4 && (i >> 2 & 1) ? ad(W[i], mu(c, X)) : fm(c, X, W[i]);
            }
            nf[i] = fm(K.dt, W[i], f[i]);
        }
        const R X = nnd(12, lam, negative(ux));
        if constexpr (sizeof(R) == 8) nlam = ad(lam, fm(mu(-E.dtdx, ux), X, dlam));
        else nlam = ad(fm(-K.dt, mu(mu(ux, X), K.inv_dx), lam), dlam);
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

__device__ __forceinline__ void join_warps() // a barrier that the four warps reach from their own code
{
    asm volatile("bar.sync 1, 128;" ::: "memory");
}

// The FP64 step of a short grid: four warps of one SM share a window of 32 cells, warp r holding
// the velocities of orbit r and one sector of the moments, so each quarter of the SM runs about
// 110 FP64 instructions a step instead of 298 while the other three would idle. Butterflies and
// back-transformed sectors pass through shared memory, two barriers a step; what a cell's
// neighbours provide stays within the warp (shuffles). The operations and their order are those
// of line_kernel, so both give the same bits. Bound by that chain of FP64 instructions: Sod tube
// of 400 cells 11.7 -> 6.8 us per step.
template <int Q> // the orbit and sector of this warp: 0 ES + EA, 1 OX, 2 OY, 3 OO and lambda
__device__ __forceinline__ void split_steps(const ModelConst<double>& K, const StepConst<double>& E,
                                            const LineArgs& a, int kmax, double* bf, double* tr)
{
    constexpr bool DIAG = Q & 1;
    const unsigned all = 0xffffffffu;
    const int t = threadIdx.x & 31, n = 32, h = 2 * kmax, own = n - 2 * h;
    const int nx = K.nx, x0 = blockIdx.x * own - h, x = x0 + t;
    const int64_t plane = K.plane;
    const double* in = static_cast<const double*>(a.in);
    int gx = x, dir = -1;
    bool fixed = false;
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
    const int jm1 = at(t - 1), j0 = at(t), jp1 = at(t + 1);
    const int dm2 = t >= 2 ? t - 2 : 0, dm1 = t >= 1 ? t - 1 : 0, dp1 = t + 1 < n ? t + 1 : n - 1;
    const bool mine = t >= h && t < h + own && x < nx;

    double f[4], lam = dir >= 0 ? K.sfeq[dir][16] : in[16 * plane + gx];
#pragma unroll
    for (int j = 0; j < 4; j++) f[j] = dir >= 0 ? K.sfeq[dir][4 * Q + j] : in[(4 * Q + j) * plane + gx];
    int bad = 0;
    for (int s = 0; s < a.nsteps; s++) {
        // this orbit's butterflies
        if constexpr (!DIAG) {
            const double sx = f[0] + f[2], sy = f[1] + f[3];
            bf[(4 * Q + 0) * n + t] = sx + sy;
            bf[(4 * Q + 1) * n + t] = sx - sy;
            bf[(4 * Q + 2) * n + t] = f[0] - f[2];
            bf[(4 * Q + 3) * n + t] = f[1] - f[3];
        } else {
            const double s01 = f[0] + f[1], d01 = f[0] - f[1], s23 = f[2] + f[3], d23 = f[2] - f[3];
            bf[(4 * Q + 0) * n + t] = s01 + s23;
            bf[(4 * Q + 1) * n + t] = d01 + d23;
            bf[(4 * Q + 2) * n + t] = d01 - d23;
            bf[(4 * Q + 3) * n + t] = s01 - s23;
        }
        if constexpr (Q == 3) bf[16 * n + t] = lam;
        join_warps();
        Fly<double> b;
        {
            const double* c = bf + t;
            b.P0 = c[0], b.M0 = c[n], b.ax0 = c[2 * n], b.ay0 = c[3 * n];
            b.e1 = c[4 * n], b.o1 = c[5 * n], b.ax1 = c[6 * n], b.ay1 = c[7 * n];
            b.P2 = c[8 * n], b.M2 = c[9 * n], b.ax2 = c[10 * n], b.ay2 = c[11 * n];
            b.e3 = c[12 * n], b.o3 = c[13 * n], b.ax3 = c[14 * n], b.ay3 = c[15 * n];
            if constexpr (Q != 3) lam = c[16 * n];
        }
        double m1, m2, m3, ux, uy, ux2, uy2, u2, T;
        bool ok;
        recover64(K, b, m1, m2, m3, ux, uy, ux2, uy2, u2, T, ok);
        if (mine && !ok) bad = 1;
        const double pT = mu(m1, T);
        const bool hot = dbits(T) > dbits(K.T_igd) && dbits(lam) != dbits(1.0);
        const bool react = __any_sync(all, hot);
        double dlam = 0.0;
        if (react && hot) dlam = reaction_increment(lam, mu(K.omega1, pT), mu(K.omega2, pT), K.dt);
        const double cr = mu(dlam, K.chem);
        double A8 = 0.0, A9 = 0.0;
        if ((Q == 1 || Q == 2) && E.a_hat) {
            const double dux = __shfl_sync(all, ux, jp1) - __shfl_sync(all, ux, jm1);
            const double duy = __shfl_sync(all, uy, jp1) - __shfl_sync(all, uy, jm1);
            a_hat<false>(E, ux, uy, dux, duy, 0.0, 0.0, A8, A9);
        }
        // this sector's part of the collision (unused entries and rows fall away)
        double D[TNE_K];
        deltas<true>(K, E, b, m1, m2, m3, ux, uy, ux2, uy2, u2, T, pT, D);
        Sectors<double> z;
        sectors<true>(K, E, K.S, D, m1, m2, m3, ux, uy, u2, T, pT, pT, A8, A9, react, cr, z);
        if constexpr (Q == 0) {
#pragma unroll
            for (int r = 0; r < 4; r++) tr[r * n + t] = z.es[r];
            tr[4 * n + t] = z.ea[0];
            tr[5 * n + t] = z.ea[1];
        } else if constexpr (Q == 3) {
            tr[14 * n + t] = z.oo[0];
            tr[15 * n + t] = z.oo[1];
        } else {
#pragma unroll
            for (int r = 0; r < 4; r++) tr[((Q == 1 ? 6 : 10) + r) * n + t] = Q == 1 ? z.ox[r] : z.oy[r];
        }
        join_warps();
        // back to this orbit's velocities, NND differences and the Euler update
        double W[4];
        {
            const double* c = tr + t;
            constexpr int o = Q >> 1; // axis or diagonal orbit number
            const double px = c[(6 + (DIAG ? 2 : 0) + o) * n], py = c[(10 + (DIAG ? 2 : 0) + o) * n];
            if constexpr (!DIAG) {
                const double es = c[o * n], ea = c[(4 + o) * n];
                const double pp = ad(es, ea), pm = ad(es, -ea);
                W[0] = ad(pp, px);
                W[2] = ad(pp, -px);
                W[1] = ad(pm, py);
                W[3] = ad(pm, -py);
            } else {
                const double es = c[(2 + o) * n], oo = c[(14 + o) * n];
                const double eo = ad(es, oo), em = ad(es, -oo), xp = ad(px, py), xm = ad(px, -py);
                W[0] = ad(eo, xp);
                W[1] = ad(em, -xm);
                W[2] = ad(eo, -xp);
                W[3] = ad(em, xm);
            }
        }
        auto nnd = [&](double q, bool neg) { // d_j = q_{j+1} - q_j, exchanged within the warp
            const double d = __shfl_sync(all, q, jp1) - __shfl_sync(all, q, j0);
            const double l2 = __shfl_sync(all, d, dm2), l1 = __shfl_sync(all, d, dm1), r1 = __shfl_sync(all, d, dp1);
            return neg ? nnd3(l1, d, r1, true) : nnd3(l2, l1, d, false);
        };
        double nf[4], nlam = lam;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int k = slot_of(4 * Q + j);
            if (k >= 0) W[j] = fm(k >= 6 ? E.cdx[Q] : -E.cdx[Q], nnd(f[j], k >= 6), W[j]);
            nf[j] = fm(K.dt, W[j], f[j]);
        }
        if constexpr (Q == 3) {
            const double d = __shfl_sync(all, lam, jp1) - __shfl_sync(all, lam, j0);
            const double l2 = __shfl_sync(all, d, dm2), l1 = __shfl_sync(all, d, dm1), r1 = __shfl_sync(all, d, dp1);
            const bool neg = negative(ux);
            const double X = nnd3(neg ? l1 : l2, neg ? d : l1, neg ? r1 : d, neg);
            nlam = clamp01(ad(lam, fm(mu(-E.dtdx, ux), X, dlam)));
        }
        if (mine && (s == a.nsteps - 1 || a.out_stride > 0)) {
            double* out = static_cast<double*>(a.out) + (a.out_stride > 0 ? s * a.out_stride : 0) + x;
            const bool avg = a.stage >= 2;
            const double* prev = static_cast<const double*>(a.prev) + x;
            auto put = [&](int i, double v) {
                out[i * plane] = avg ? fm(a.wprev, prev[i * plane], mu(a.wnew, v)) : v;
            };
#pragma unroll
            for (int j = 0; j < 4; j++) put(4 * Q + j, nf[j]);
            if constexpr (Q == 3) put(16, nlam);
        }
        if (!fixed) {
#pragma unroll
            for (int j = 0; j < 4; j++) f[j] = nf[j];
            lam = nlam;
        }
    }
    if (Q == 0 && __any_sync(all, bad) && t == 0) atomicOr(&a.ctr->status, 1);
}

__global__ void __launch_bounds__(128)
    line_split_kernel(const __grid_constant__ ModelConst<double> K, const __grid_constant__ StepConst<double> E,
                      const __grid_constant__ LineArgs a, int kmax)
{
    __shared__ double bf[17 * 32], tr[16 * 32]; // butterflies and lambda; transformed sectors
    switch (threadIdx.x >> 5) {
    case 0: split_steps<0>(K, E, a, kmax, bf, tr); break;
    case 1: split_steps<1>(K, E, a, kmax, bf, tr); break;
    case 2: split_steps<2>(K, E, a, kmax, bf, tr); break;
    default: split_steps<3>(K, E, a, kmax, bf, tr); break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (a.stage < 2) a.ctr->tne_pending = 0;
        if (a.stage == 0 || a.stage == 2) a.ctr->step += a.nsteps;
    }
}

template <typename R, int REC, bool TNE>
cudaError_t line_launch_t(const ModelConst<R>& K, const LinePlan& p, const LineArgs& a, cudaStream_t s)
{
    const size_t bytes = line_smem<R>(p.threads, a.tne_every > 0);
    static cudaError_t done = cudaFuncSetAttribute(line_kernel<R, REC, TNE>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)line_smem<R>(LINE_THREADS, true));
    if (done != cudaSuccess) return done;
    StepConst<R> E;
    step_const(K, &E);
    line_kernel<R, REC, TNE><<<p.grid, p.threads, bytes, s>>>(K, E, a, p.steps);
    return cudaGetLastError();
}

} // namespace

// The cut of a 1-D grid: the (threads, steps) with the least time per step as measured over
// 19 cuts of seven lengths from 400 to 2^20 cells, modelled by the warps w an SM gets. FP64:
// an SM's FP64 units pass 3.0 us of warps one after another once its four quarters are busy
// (us per step: w = 3 12.8, 4 13.9, 5 16.3, 6 17.5, 8 24.1, 16 44.7) and a launch costs
// 1.5 us beside its steps. FP32: latency first, issue from about 20 warps on (w = 4 1.29,
// 6 1.63, 8 1.93, 16 2.95, 230 40.5), a launch 2.0 us. On 152 SMs that gives (threads x steps)
// FP64 grids of a few thousand cells 96 x 16, 16384 cells 128 x 4 (14.2 us per step measured; 128 x 8,
// whose 171 blocks no longer fit one per SM, 23.3), a million cells 192 x 1 (one step 622, four 683);
// FP32 400 cells 64 x 8 (3.3 with one step), 16384 cells 160 x 8 (2.0 measured; 128 x 4 1.8 to 2.0), a
// million cells 192 x 1.
LinePlan line_plan(int precision, int nx, bool tne)
{
    static int sms = -1;
    if (sms < 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 152;
    }
    LinePlan best = {128, 1, (nx + 123) / 124, false};
    double t_best = 1e300;
    for (int threads = 32; threads <= LINE_THREADS; threads += 32)
        for (int steps = 1; steps <= 16; steps *= 2) {
            const int own = threads - 4 * steps;
            if (own < 16) continue;
            const int grid = (nx + own - 1) / own;
            const double w = (double)((grid + sms - 1) / sms) * (threads / 32);
            const double t = precision == 0 ? (w > 4.25 ? 3.0 * w : 12.8) + 1.5 / steps
                                            : (w > 21.0 ? 0.17 * w : 0.85 + 0.131 * w) + 2.0 / steps;
            if (t < t_best) t_best = t, best = {threads, steps, grid, false};
        }
    // four warps to a window of 32 cells while an SM gets two windows at most (us per step, host
    // clock: 400 cells 7.2 against 11.7, 4200 cells 8.8; two windows, which share the FP64 unit:
    // 4864 cells 10.2 against 13.0, 8192 cells 11.7 against 14.2; a third would bring it to 14)
    for (int steps = 1; precision == 0 && !tne && steps <= 4; steps *= 2) {
        const int own = 32 - 4 * steps, grid = (nx + own - 1) / own;
        const double t = (grid <= sms ? 6.7 : 9.7) + 2.0 / steps;
        if (grid <= 2 * sms && t < t_best) t_best = t, best = {128, steps, grid, true};
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
        if (p.split) {
            if (b.tne_every > 0) return cudaErrorInvalidValue;
            StepConst<double> E;
            step_const(Kd, &E);
            line_split_kernel<<<p.grid, 128, 0, s>>>(Kd, E, b, p.steps);
            return cudaGetLastError();
        }
        return b.tne_every > 0 ? line_launch_t<double, 0, true>(Kd, p, b, s) : line_launch_t<double, 0, false>(Kd, p, b, s);
    }
    const ModelConst<float>& Kf = *static_cast<const ModelConst<float>*>(K);
    if (b.tne_every > 0)
        return recovery == 1 ? line_launch_t<float, 1, true>(Kf, p, b, s) : line_launch_t<float, 0, true>(Kf, p, b, s);
    return recovery == 1 ? line_launch_t<float, 1, false>(Kf, p, b, s) : line_launch_t<float, 0, false>(Kf, p, b, s);
}

} // namespace lbk
