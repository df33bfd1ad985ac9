// tile.cu -- the 2-D step in tiles of 32 x 8 (FP64) or 32 x 4 cells, one cell per thread: the
// FP64 form, and FP32 grids too small to fill the marching kernel (march.cu).
//
// Each block walks tiles (grid-stride loop, grid = SMs x resident blocks). Per tile it stages
// the 17 planes of the tile and a halo of two cells (element-wise asynchronous copies, ghost
// cells mapped once per row and column), recovers rho, u, T of its own cells and u of the
// one-cell rim (grad u), and updates the cells from registers and shared memory; each f_i is
// read once from HBM and written once. TNE statistics, when due, go through shared memory one
// quantity per lane (warp_tne) and stay in per-warp FP64 sums until the block has done all its
// tiles.
//
// What bounds it. FP64: the FP64 unit, 19 cycles of an SM per warp instruction (cellops.cuh),
// 83 % busy (ncu, 1024^2); a tile row takes 545 of them, against 698 adds, multiplies and FMAs
// and the compares of 28 limited differences with the plain formulas and the rim recovered in
// full (1024^2: 2.06 -> 1.14 ms per step). FP32: on small grids the
// latency of staging, recovery and update, a few us each, against about 20 us that a strip of
// the marching kernel takes from its first copy to its last store.
#include <float.h>

#include "cellops.cuh"
#include "tile.cuh"

namespace lbk {

namespace {

constexpr int TX = 32, SW = TX + 4, UW = TX + 2; // cells of a row, staged, with u

// FP64 takes eight rows (of the rim's 80 recoveries 3 warps' worth on 8 instead of 4), FP32
// four (more blocks on a small grid)
template <typename R>
struct Tile {
    static constexpr int TY = sizeof(R) == 8 ? 8 : 4, TT = TX * TY, TW = TY;
    static constexpr int SH = TY + 4, PS = SW * SH; // staged rows y0-2 .. y0+TY+1
    static constexpr int UH = TY + 2;               // u of the tile and its rim
    static constexpr size_t smem(bool tne)
    {
        return sizeof(R) * ((size_t)NPLANE * PS + 2 * UW * UH) +
               (tne ? sizeof(double) * (2 * TW * TNE_PART) + sizeof(R) * 14 * (TT + 1) : 0);
    }
};

// u of a cell of the rim from its 16 values at stride PS. FP64: by the formulas of the tile's own
// cells (what T takes falls away), so a velocity has the same bits in the tile and in its neighbours'
// rims and grad u of a uniform flow vanishes at tile edges too. FP32: plain FP32, as the marching
// kernel's strips have it at their sides; the exact sums take 3 % of a step (300 x 100).
__device__ __forceinline__ void rim_u(const ModelConst<double>& K, const double* s, double& ux, double& uy)
{
    double f[16], m1, m2, m3, ux2, uy2, u2, T;
    bool ok;
#pragma unroll
    for (int i = 0; i < 16; i++) f[i] = s[i * Tile<double>::PS];
    recover64<true>(K, butterflies(f), m1, m2, m3, ux, uy, ux2, uy2, u2, T, ok);
}
__device__ __forceinline__ void rim_u(const ModelConst<float>& K, const float* s, float& ux, float& uy)
{
    constexpr int PS = Tile<float>::PS;
    float f[16];
#pragma unroll
    for (int i = 0; i < 16; i++) f[i] = s[i * PS];
    velocity_f32(f, K, ux, uy);
}

template <typename R, int REC, bool TNE>
__global__ void __launch_bounds__(Tile<R>::TT, sizeof(R) == 8 ? 2 : 4)
    tile_kernel(const __grid_constant__ ModelConst<R> K, const __grid_constant__ StepConst<R> E,
                const __grid_constant__ StepLaunch a)
{
    constexpr int TY = Tile<R>::TY, TT = Tile<R>::TT, TW = Tile<R>::TW, SH = Tile<R>::SH, PS = Tile<R>::PS,
                  UH = Tile<R>::UH;
    extern __shared__ __align__(16) unsigned char smem[];
    R* sf = reinterpret_cast<R*>(smem);                       // [17][SH][SW]
    R* su = sf + NPLANE * PS;                                 // u_x, u_y  [2][UH][UW]
    double* acc = reinterpret_cast<double*>(su + 2 * UH * UW); // the launch's statistics [TW][TNE_PART]
    double* res = acc + TW * TNE_PART;                        // the tile's
    R* td = reinterpret_cast<R*>(res + TW * TNE_PART);        // [14][TT + 1]

    const int t = threadIdx.x, lx = t & 31, ly = t >> 5; // a warp is a row of the tile
    const int nx = K.nx, ny = K.ny, pitch = K.pitch;
    const int64_t plane = K.plane;
    const R* __restrict__ in = static_cast<const R*>(a.in);
    R* out = static_cast<R*>(a.out); // not restrict: prev may alias it
    const bool tne = TNE && a.tne_every > 0;
    const int64_t step = tne ? a.ctr->step : 0;
    const bool do_tne = tne && step % a.tne_every == 0;
    if (do_tne)
        for (int i = lx; i < TNE_PART; i += 32) {
            const int kind = tne_kind(i);
            acc[ly * TNE_PART + i] = kind == 0 ? 0.0 : (kind == 1 ? DBL_MAX : -DBL_MAX);
        }
    const bool avg = a.stage >= 2; // a later SSP Runge-Kutta stage: weighted with u^n
    const R* prev = static_cast<const R*>(a.prev);
    const R wp = (R)a.wprev, wn = (R)a.wnew;
    int bad = 0;

    const int tiles_x = (nx + TX - 1) / TX;
    const int ntiles = tiles_x * ((ny + TY - 1) / TY);
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int x0 = (tile % tiles_x) * TX, y0 = (tile / tiles_x) * TY;
        __syncthreads(); // the previous tile is done with shared memory
        stage_tile<NPLANE, SH, SW, TW, true>(in, sf, x0 - 2, y0 - 2, nx, ny, pitch, plane, K.sbc, K.sfeq,
                                             [](int p) { return mirror_plane(p); });
        cp_commit();
        cp_wait<0>();
        __syncthreads();
        // walls: the staged ghost rows hold copies of the edge fluid row (the index map
        // clamps); add the non-equilibrium-extrapolation correction
        if ((K.sbc[2] == 2 || K.sbc[3] == 2) && (y0 - 2 < 0 || y0 + TY + 2 > ny)) {
            for (int idx = t; idx < 2 * SW; idx += TT) {
                const int side = idx / SW, c = idx - side * SW;
                if (K.sbc[2 + side] != 2) continue;
                const int rs = (side == 0 ? 0 : ny - 1) - (y0 - 2); // fluid row
                if (rs < 0 || rs >= SH) continue;
                R fl[16], d[16];
#pragma unroll
                for (int i = 0; i < 16; i++) fl[i] = sf[i * PS + rs * SW + c];
                wall_correction(K, fl, side, d);
                for (int r = 0; r < SH; r++) {
                    const int gy = y0 - 2 + r;
                    if (side == 0 ? gy >= 0 : gy < ny) continue;
#pragma unroll
                    for (int i = 0; i < 16; i++) sf[i * PS + r * SW + c] += d[i];
                }
            }
            __syncthreads();
        }
        const int x = x0 + lx, y = y0 + ly;
        const bool active = x < nx && y < ny;
        const R* s0 = sf + (ly + 2) * SW + lx + 2;
        Fly<R> b;
        R f[16], lam = s0[16 * PS], m1, m2, m3, ux, uy, ux2, uy2, u2, T;
        bool hot = false, ok;
#pragma unroll
        for (int i = 0; i < 16; i++) f[i] = s0[i * PS];
        if (y < ny) { // whole warps past the last row have nothing to do
            b = butterflies(f);
            if constexpr (sizeof(R) == 8) {
                recover64<true>(K, b, m1, m2, m3, ux, uy, ux2, uy2, u2, T, ok);
                hot = dbits(T) > dbits(K.T_igd) && dbits(lam) != dbits(1.0);
            } else {
                recover32<REC>(K, f, m1, ux, uy, T, hot, ok);
                hot = hot && lam != 1.f;
                m2 = mu(m1, ux);
                m3 = mu(m1, uy);
                ux2 = mu(ux, ux);
                uy2 = mu(uy, uy);
                u2 = ad(ux2, uy2);
            }
            if (active && !ok) bad = 1;
            su[(ly + 1) * UW + lx + 1] = ux;
            su[(UH + ly + 1) * UW + lx + 1] = uy;
        }
        // the rim; with a ragged last row of tiles the row past the grid is one of the tile's
        for (int c = t; c < 2 * UW + 2 * TY || (y0 + TY > ny && c < 2 * UW + 2 * TY + TX); c += TT) {
            int rx, ry;
            if (c < 2 * UW) rx = c % UW, ry = c < UW ? 0 : UH - 1;
            else if (c < 2 * UW + 2 * TY) rx = (c & 1) ? UW - 1 : 0, ry = 1 + (c - 2 * UW) / 2;
            else rx = 1 + c - 2 * UW - 2 * TY, ry = ny - y0 + 1;
            rim_u(K, sf + (ry + 1) * SW + rx + 1, su[ry * UW + rx], su[(UH + ry) * UW + rx]);
        }
        __syncthreads();
        if (y >= ny) continue;

        const R pT = mu(m1, T);
        R D[TNE_K], W[16], A8 = R(0), A9 = R(0);
        deltas<false>(K, E, b, m1, m2, m3, ux, uy, ux2, uy2, u2, T, pT, D);
        if (do_tne) {
            R d2 = mu(D[0], D[0]);
            td[t] = D[0];
#pragma unroll
            for (int k = 1; k < TNE_K; k++) {
                td[k * (TT + 1) + t] = D[k];
                d2 = fm(D[k], D[k], d2);
            }
            td[12 * (TT + 1) + t] = sqrt(d2);
            td[13 * (TT + 1) + t] = d2;
            const unsigned mask = __ballot_sync(0xffffffffu, active);
            __syncwarp();
            double* rw = res + ly * TNE_PART;
            warp_tne(td + ly * 32, TT + 1, mask, rw);
            __syncwarp();
            for (int i = lx; i < TNE_PART; i += 32)
                acc[ly * TNE_PART + i] = tne_comb(tne_kind(i), acc[ly * TNE_PART + i], rw[i]);
        }
        const bool react = __any_sync(0xffffffffu, hot);
        R dlam = R(0);
        if (react && hot) dlam = reaction_increment(lam, mu(K.omega1, pT), mu(K.omega2, pT), K.dt);
        if (E.a_hat) {
            const R* u0 = su + (ly + 1) * UW + lx + 1;
            const R* v0 = u0 + UH * UW;
            a_hat<true>(E, ux, uy, u0[1] - u0[-1], v0[1] - v0[-1], u0[UW] - u0[-UW], v0[UW] - v0[-UW], A8, A9);
        }
        collide<false>(K, E, K.S, D, m1, m2, m3, ux, uy, u2, T, a_weight(pT, E.c8), a_weight(pT, E.c9), A8, A9, react,
                mu(dlam, K.chem), W);

        // NND flux differences of plane i along one axis (stride d), upwind side by `neg`
        auto nnd = [&](const R* q, R q0, int d, bool neg) -> R {
            const R l = q[-d], r = q[d];
            return neg ? nnd3(sub(q0, l), sub(r, q0), sub(q[2 * d], r), true)
                       : nnd3(sub(l, q[-2 * d]), sub(q0, l), sub(r, q0), false);
        };
        // the same with the side decided at run time: the operands are chosen, not the results
        auto nnd_by = [&](const R* q, R q0, int d, bool neg) -> R {
            const R* c = neg ? q + d : q;
            const R c0 = neg ? *c : q0, l = c[-d];
            return nnd3(sub(l, c[-2 * d]), sub(c0, l), sub(c[d], c0), neg);
        };
        const int64_t g = (int64_t)y * pitch + x;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const int o = i >> 2, j = i & 3;
            const int sx = (o & 1) ? (j == 0 || j == 3 ? 1 : -1) : (j == 0 ? 1 : (j == 2 ? -1 : 0));
            const int sy = (o & 1) ? (j < 2 ? 1 : -1) : (j == 1 ? 1 : (j == 3 ? -1 : 0));
            R w = W[i];
            if constexpr (sizeof(R) == 8) {
                if (sx != 0) w = fm(sx < 0 ? E.cdx[o] : -E.cdx[o], nnd(s0 + i * PS, f[i], 1, sx < 0), w);
                if (sy != 0) w = fm(sy < 0 ? E.cdy[o] : -E.cdy[o], nnd(s0 + i * PS, f[i], SW, sy < 0), w);
            } else { // v . grad f first
                const R X = sx != 0 ? nnd(s0 + i * PS, f[i], 1, sx < 0) : R(0);
                const R Y = sy != 0 ? nnd(s0 + i * PS, f[i], SW, sy < 0) : R(0);
                const R cx = sx < 0 ? -E.cdx[o] : E.cdx[o], cy = sy < 0 ? -E.cdy[o] : E.cdy[o];
                w = sub(w, sx == 0 ? mu(cy, Y) : sy == 0 ? mu(cx, X) : j == 1 ? fm(cy, Y, mu(cx, X)) : fm(cx, X, mu(cy, Y)));
            }
            const R v = fm(K.dt, w, f[i]);
            if (active) out[i * plane + g] = avg ? fm(wp, prev[i * plane + g], mu(wn, v)) : v;
        }
        const R lx_ = nnd_by(s0 + 16 * PS, lam, 1, negative(ux)), ly_ = nnd_by(s0 + 16 * PS, lam, SW, negative(uy));
        R ln;
        if constexpr (sizeof(R) == 8) ln = ad(lam, fm(mu(-E.dtdy, uy), ly_, fm(mu(-E.dtdx, ux), lx_, dlam)));
        else ln = ad(fm(-K.dt, fm(mu(ux, K.inv_dx), lx_, mu(mu(uy, K.inv_dy), ly_)), lam), dlam);
        ln = clamp01(ln);
        if (active) out[16 * plane + g] = avg ? fm(wp, prev[16 * plane + g], mu(wn, ln)) : ln;
    }

    // status, TNE partials, step counter: without TNE no block reads the counter, so block 0
    // moves it on; with TNE the last block to finish does
    if (__syncthreads_or(bad) && t == 0) atomicOr(&a.ctr->status, 1);
    if (do_tne && t < TNE_PART) {
        double v = acc[t];
        for (int w = 1; w < TW; w++) v = tne_comb(tne_kind(t), v, acc[w * TNE_PART + t]);
        a.partials[(size_t)t * gridDim.x + blockIdx.x] = v; // quantity-major
    }
    const bool counts = a.stage == 0 || a.stage == 2;
    if (!tne) {
        if (blockIdx.x == 0 && t == 0) {
            if (a.stage < 2) a.ctr->tne_pending = 0;
            if (counts) a.ctr->step += 1;
        }
    } else if (t == 0) {
        if (atomicAdd(&a.ctr->arrivals, 1u) == gridDim.x - 1) {
            if (do_tne) {
                a.ctr->hist_count += 1;
                a.ctr->tne_step = step;
            }
            a.ctr->tne_pending = do_tne ? 1 : 0;
            if (counts) a.ctr->step = step + 1;
            a.ctr->arrivals = 0u;
        }
    }
}

template <typename R, int REC, bool TNE>
cudaError_t tile_prepare()
{
    static cudaError_t done = cudaFuncSetAttribute(
        tile_kernel<R, REC, TNE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile<R>::smem(TNE));
    return done;
}

template <typename R, int REC, bool TNE>
int tile_resident()
{
    static int per_sm = -1;
    if (per_sm < 0) {
        if (tile_prepare<R, REC, TNE>() != cudaSuccess) return -1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, tile_kernel<R, REC, TNE>, Tile<R>::TT,
                                                          Tile<R>::smem(TNE)) != cudaSuccess)
            return -1;
        if (per_sm < 1) per_sm = 1;
    }
    return per_sm;
}

template <typename R, int REC, bool TNE>
cudaError_t tile_launch_t(const ModelConst<R>& K, const StepLaunch& a, cudaStream_t s)
{
    const cudaError_t e = tile_prepare<R, REC, TNE>();
    if (e != cudaSuccess) return e;
    StepConst<R> E;
    step_const(K, &E);
    tile_kernel<R, REC, TNE><<<a.grid, Tile<R>::TT, Tile<R>::smem(TNE), s>>>(K, E, a);
    return cudaGetLastError();
}

} // namespace

// FP32 grids of up to 1000 tiles (400 with the slower double-float recovery) step here: us per
// step here and in the marching kernel, 96^2 8.0 / 13.2, 300 x 100 per-side 9.9 / 21.9, 256^2
// 10.9 / 17.5, 300^2 17.8 / 22.2 (double-float 25.9 / 19.0), 30 x 3000 18.1 / 34.9, 512 x 300
// 20.0 / 20.3, 512^2 35.1 / 29.8.
bool tile_takes_f32(int recovery, int nx, int ny)
{
    const int64_t tiles = (int64_t)((nx + TX - 1) / TX) * ((ny + Tile<float>::TY - 1) / Tile<float>::TY);
    return tiles <= (recovery == 1 ? 400 : 1000);
}

int tile_grid(int precision, int recovery, int nx, int ny, bool tne)
{
    static int sms = -1;
    if (sms < 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
    }
    // the later stages of a Runge-Kutta step share the grid of the first, which keeps records
    const int per_sm = precision == 0 ? (tne ? tile_resident<double, 0, true>() : tile_resident<double, 0, false>())
                       : recovery == 1 ? (tne ? tile_resident<float, 1, true>() : tile_resident<float, 1, false>())
                                       : (tne ? tile_resident<float, 0, true>() : tile_resident<float, 0, false>());
    const int ty = precision == 0 ? Tile<double>::TY : Tile<float>::TY;
    const int64_t tiles = (int64_t)((nx + TX - 1) / TX) * ((ny + ty - 1) / ty), g = (int64_t)per_sm * sms;
    return per_sm < 1 ? -1 : (int)(tiles < g ? tiles : g);
}

cudaError_t launch_tile(int precision, int recovery, const void* K, const StepLaunch& a, cudaStream_t s)
{
    StepLaunch b = a;
    if (a.stage >= 2) b.tne_every = 0; // only u^n has records
    const bool tne = b.tne_every > 0;
    if (precision == 0) {
        const ModelConst<double>& Kd = *static_cast<const ModelConst<double>*>(K);
        return tne ? tile_launch_t<double, 0, true>(Kd, b, s) : tile_launch_t<double, 0, false>(Kd, b, s);
    }
    const ModelConst<float>& Kf = *static_cast<const ModelConst<float>*>(K);
    if (recovery == 1)
        return tne ? tile_launch_t<float, 1, true>(Kf, b, s) : tile_launch_t<float, 1, false>(Kf, b, s);
    return tne ? tile_launch_t<float, 0, true>(Kf, b, s) : tile_launch_t<float, 0, false>(Kf, b, s);
}

} // namespace lbk
