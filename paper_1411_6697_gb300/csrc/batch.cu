// batch.cu -- persistent driver for many 1-D instances of uneven length.
//
// The instances are concatenated into one flat grid (each starts on a 16-byte boundary: nx is a
// multiple of 4). Work items are (instance, segment). One launch runs `nsteps` time steps in
// phases of up to BATCH_STEPS: in a phase the blocks walk the item list (grid-stride), and a
// block carries a window of BT cells of its item, one per thread, through the phase's steps in
// registers, neighbours meeting in shared memory once per step; the middle BT - 4 BATCH_STEPS
// cells are the item's segment, the rest overlaps with the neighbour items' windows. Boundaries
// are zero-gradient per instance, S, Q and omega1 per instance. A grid barrier separates the
// phases; its wait is bounded in time and reports a timeout through the status word instead of
// hanging. The launch is cooperative, so all blocks are resident.
//
// What bounds it: instruction issue and the FP64 unit of the recovery (8 of its instructions a
// warp and step, 64 cycles each). Two steps per pass took half the state's traffic and half the
// barriers off; one cell per thread instead of a pair leaves registers for six blocks of 128 on
// an SM. 512 detonations, 7.95 M cells, ms per step: one step per pass and a pair of cells per
// thread 0.430; one cell and two steps 0.330 (four 0.361: the shared edges grow; five or eight
// blocks an SM 0.356, 0.333); with the pairs joined on the integer pipe (pair_to_f64) 0.315 (one
// step 0.367, three 0.329), with the even moments' equilibria rounded before they are subtracted
// (deltas, cellops.cuh) 0.322, and with pair_to_f64's one select before the rounding 0.314.
#include <float.h>
#include <stdint.h>

#include "cellops.cuh"
#include "kernels.cuh"

namespace lbk {

namespace {

constexpr int BATCH_STEPS = 2; // time steps between grid barriers
constexpr int BNX = 13;        // planes that neighbours read: those with v_x != 0, and lambda

// plane of a slot (v_x > 0 in the first six, v_x < 0 in the next six, then lambda) and the slot
// of a plane (-1: v_x = 0)
__host__ __device__ constexpr int slot_plane(int s)
{
    constexpr int t[BNX] = {0, 4, 7, 8, 12, 15, 2, 5, 6, 10, 13, 14, 16};
    return t[s];
}
__host__ __device__ constexpr int slot_of(int plane)
{
    constexpr int t[16] = {0, -1, 6, -1, 1, 7, 8, 2, 3, -1, 9, -1, 4, 10, 11, 5};
    return t[plane];
}

template <int BT>
struct BCfg {
    static constexpr int H = 2 * BATCH_STEPS, SEG = BT - 2 * H; // halo and own cells of an item
    static constexpr int PUB = (BNX + 2) * BT;                  // published planes, u_x, u_y
    static constexpr size_t SMEM = sizeof(float) * (2 * PUB + 32);
};

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// All blocks arrive; the last one advances the generation. A waiting block gives
// up after b.wait_ns nanoseconds, sets status bit 1 and reports false.
__device__ bool grid_barrier(const BatchLaunch& b, unsigned expected)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        volatile unsigned* gen = b.bar + 1;
        const unsigned g = *gen;
        __threadfence();
        const unsigned arrived = atomicAdd(b.bar, 1u) + 1u;
        if (arrived == expected) {
            b.bar[0] = 0u;
            __threadfence();
            atomicAdd(b.bar + 1, 1u);
        } else {
            const uint64_t t0 = global_ns();
            while (*gen == g) {
                if (global_ns() - t0 > (uint64_t)b.wait_ns) {
                    atomicOr(&b.ctr->status, 2);
                    ok = 0;
                    break;
                }
                __nanosleep(128);
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

template <int REC, int BT>
__global__ void __launch_bounds__(BT, 768 / BT)
    batch_kernel(const __grid_constant__ ModelConst<float> K, const __grid_constant__ StepConst<float> E,
                 const __grid_constant__ BatchLaunch b)
{
    using C = BCfg<BT>;
    extern __shared__ __align__(16) float sm[];
    float* par = sm + 2 * C::PUB; // S[16], A8c, A9c, chem, om1, om2
    const int t = threadIdx.x;
    const unsigned expected = gridDim.x + (unsigned)b.phantom_blocks;
    const int64_t plane = K.plane;

    int phase = 0;
    for (int done = 0; done < b.nsteps; phase++) {
        const int m = b.nsteps - done < BATCH_STEPS ? b.nsteps - done : BATCH_STEPS;
        const bool odd = (b.cur + phase) & 1;
        const float* __restrict__ in = static_cast<const float*>(odd ? b.buf[1] : b.buf[0]);
        float* __restrict__ out = static_cast<float*>(odd ? b.buf[0] : b.buf[1]);
        int bad = 0;
        for (int item = blockIdx.x; item < b.nitems; item += gridDim.x) {
            const BatchItem it = b.items[item];
            const InstParam& ip = b.inst[it.inst];
            const int w0 = it.x0 - C::H, x = w0 + t, nx = ip.nx;
            const int gx = x < 0 ? 0 : (x >= nx ? nx - 1 : x);
            const bool fixed = x != gx; // a ghost lane: read through the end cell, never updated
            const bool mine = t >= C::H && t < C::H + C::SEG && x < nx;
            const int lo = w0 < 0 ? -w0 : 0, hi = nx - 1 - w0 < BT - 1 ? nx - 1 - w0 : BT - 1;
            auto at = [&](int j) { return j < lo ? lo : (j > hi ? hi : j); };
            const int jm2 = at(t - 2), jm1 = at(t - 1), jp1 = at(t + 1), jp2 = at(t + 2);
            const float* src = in + ip.off + gx;
            float f[16], lam = src[16 * plane];
#pragma unroll
            for (int i = 0; i < 16; i++) f[i] = src[i * plane];
            __syncthreads(); // the previous item is done with shared memory
            if (t < 16) par[t] = ip.S[t];
            if (t == 16) par[16] = ip.A8c;
            if (t == 17) par[17] = ip.A9c;
            if (t == 18) par[18] = ip.chem;
            if (t == 19) par[19] = ip.om1;
            if (t == 20) par[20] = ip.om2;
            for (int s = 0; s < m; s++) {
                float* P = sm + (s & 1) * C::PUB;
                const Fly<float> fl = butterflies(f);
                float m1, ux, uy, T;
                bool hot, ok;
                recover32<REC>(K, f, m1, ux, uy, T, hot, ok);
                if (mine && !ok) bad = 1;
                hot = hot && lam != 1.f;
                const float m2 = mu(m1, ux), m3 = mu(m1, uy);
                const float ux2 = mu(ux, ux), uy2 = mu(uy, uy), u2 = fm(ux, ux, uy2), pT = mu(m1, T);
#pragma unroll
                for (int k = 0; k < BNX; k++) P[k * BT + t] = slot_plane(k) == 16 ? lam : f[slot_plane(k) & 15];
                P[BNX * BT + t] = ux;
                P[(BNX + 1) * BT + t] = uy;
                __syncthreads();
                float D[TNE_K], W[16], A8, A9;
                deltas<true>(K, E, fl, m1, m2, m3, ux, uy, ux2, uy2, u2, T, pT, D);
                a_hat<false>(E, ux, uy, P[BNX * BT + jp1] - P[BNX * BT + jm1],
                             P[(BNX + 1) * BT + jp1] - P[(BNX + 1) * BT + jm1], 0.f, 0.f, A8, A9);
                const bool react = __any_sync(0xffffffffu, hot);
                float dlam = 0.f;
                if (react && hot) dlam = reaction_increment(lam, mu(par[19], pT), mu(par[20], pT), K.dt);
                collide<true>(K, E, par, D, m1, m2, m3, ux, uy, u2, T, mu(pT, par[16]), mu(pT, par[17]), A8, A9, react,
                        mu(dlam, par[18]), W);
                auto nnd = [&](int k, float q, bool neg) -> float {
                    const float* r = P + k * BT;
                    const float l = r[jm1], g = r[jp1];
                    return neg ? nnd3(q - l, g - q, r[jp2] - g, true) : nnd3(l - r[jm2], q - l, g - q, false);
                };
#pragma unroll
                for (int i = 0; i < 16; i++) {
                    const int k = slot_of(i);
                    float w = W[i];
                    if (k >= 0) w = fm(k >= 6 ? E.cdx[i >> 2] : -E.cdx[i >> 2], nnd(k, f[i], k >= 6), w);
                    if (!fixed) f[i] = fm(K.dt, w, f[i]);
                }
                const float ln = clamp01(ad(lam, fm(mu(-E.dtdx, ux), nnd(12, lam, negative(ux)), dlam)));
                if (!fixed) lam = ln;
            }
            if (mine) {
                float* dst = out + ip.off + x;
#pragma unroll
                for (int i = 0; i < 16; i++) dst[i * plane] = f[i];
                dst[16 * plane] = lam;
            }
        }
        done += m;
        if (__syncthreads_or(bad) && t == 0) atomicOr(&b.ctr->status, 1);
        if (!grid_barrier(b, expected)) return;
        if (blockIdx.x == 0 && t == 0) b.ctr->step += m;
    }
}

template <int REC, int BT>
cudaError_t batch_prepare()
{
    static cudaError_t done = cudaFuncSetAttribute(
        batch_kernel<REC, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BCfg<BT>::SMEM);
    return done;
}

template <int REC, int BT>
int batch_max_blocks_per_sm()
{
    if (batch_prepare<REC, BT>() != cudaSuccess) return -1;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel<REC, BT>, BT,
                                                      BCfg<BT>::SMEM) != cudaSuccess)
        return -1;
    return per_sm;
}

template <int REC, int BT>
cudaError_t batch_launch_t(const ModelConst<float>& K, const BatchLaunch& b, int grid,
                           cudaStream_t s)
{
    cudaError_t e = batch_prepare<REC, BT>();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(BT);
    cfg.dynamicSmemBytes = BCfg<BT>::SMEM;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    StepConst<float> E;
    step_const(K, &E);
    E.c8 = E.c9 = 1.f; // A8c and A9c are the instances'
    E.a_hat = 1;
    return cudaLaunchKernelEx(&cfg, batch_kernel<REC, BT>, K, E, b);
}

constexpr int TI_THREADS = 256;

template <typename R>
__global__ void __launch_bounds__(TI_THREADS)
    tne_instances_kernel(const ModelConst<double> K, const R* state, const InstParam* inst,
                         TneRecord* out, double area)
{
    __shared__ double ssum[TI_THREADS / 32][2 * TNE_K + 2];
    __shared__ double smn[TI_THREADS / 32][TNE_K], smx[TI_THREADS / 32][TNE_K];
    const InstParam& ip = inst[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double acc[2 * TNE_K + 2], mn[TNE_K], mx[TNE_K];
    for (int q = 0; q < 2 * TNE_K + 2; q++) acc[q] = 0.0;
    for (int k = 0; k < TNE_K; k++) mn[k] = DBL_MAX, mx[k] = -DBL_MAX;
    for (int x = threadIdx.x; x < ip.nx; x += TI_THREADS) {
        const int64_t g = ip.off + x;
        double f[16], m[16], q[16];
        for (int i = 0; i < 16; i++) f[i] = (double)state[i * K.plane + g];
        forward_moments(K, f, m);
        const double r = m[0], u = m[1] / r, v = m[2] / r;
        const double t = (m[3] / r - (u * u + v * v)) * K.inv_DId;
        feq_moments(K.DI, r, u, v, t, q);
        double d2 = 0.0;
        for (int k = 4; k < 16; k++) {
            const double D = m[k] - q[k];
            acc[k - 4] += D;
            acc[TNE_K + k - 4] += fabs(D);
            mn[k - 4] = fmin(mn[k - 4], D);
            mx[k - 4] = fmax(mx[k - 4], D);
            d2 += D * D;
        }
        acc[2 * TNE_K] += sqrt(d2);
        acc[2 * TNE_K + 1] += d2;
    }
    for (int q = 0; q < 2 * TNE_K + 2; q++) {
        double v = acc[q];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) ssum[warp][q] = v;
    }
    for (int k = 0; k < TNE_K; k++) {
        double a = mn[k], c = mx[k];
        for (int o = 16; o > 0; o >>= 1) {
            a = fmin(a, __shfl_xor_sync(0xffffffffu, a, o));
            c = fmax(c, __shfl_xor_sync(0xffffffffu, c, o));
        }
        if (lane == 0) smn[warp][k] = a, smx[warp][k] = c;
    }
    __syncthreads();
    TneRecord* rec = out + blockIdx.x;
    const int k = threadIdx.x;
    if (k < 16) {
        double s0 = 0, s1 = 0, a = DBL_MAX, c = -DBL_MAX;
        if (k >= 4)
            for (int w = 0; w < TI_THREADS / 32; w++) {
                s0 += ssum[w][k - 4];
                s1 += ssum[w][TNE_K + k - 4];
                a = fmin(a, smn[w][k - 4]);
                c = fmax(c, smx[w][k - 4]);
            }
        rec->sum[k] = k < 4 ? 0.0 : s0 * area;
        rec->abs_sum[k] = k < 4 ? 0.0 : s1 * area;
        rec->min[k] = k < 4 ? 0.0 : a;
        rec->max[k] = k < 4 ? 0.0 : c;
    } else if (k == 32) {
        double d = 0, d2 = 0;
        for (int w = 0; w < TI_THREADS / 32; w++) d += ssum[w][2 * TNE_K], d2 += ssum[w][2 * TNE_K + 1];
        rec->d_sum = d * area;
        rec->d2_sum = d2 * area;
        rec->step = -1;
    }
}

} // namespace

cudaError_t launch_tne_instances(int precision, const ModelConst<double>& Kd, const void* state,
                                 const InstParam* inst, int n_inst, TneRecord* out,
                                 double area, cudaStream_t s)
{
    if (precision == 0)
        tne_instances_kernel<double><<<n_inst, TI_THREADS, 0, s>>>(
            Kd, static_cast<const double*>(state), inst, out, area);
    else
        tne_instances_kernel<float><<<n_inst, TI_THREADS, 0, s>>>(
            Kd, static_cast<const float*>(state), inst, out, area);
    return cudaGetLastError();
}

int batch_segment(int block_threads) { return block_threads - 4 * BATCH_STEPS; }
int batch_phases(int nsteps) { return (nsteps + BATCH_STEPS - 1) / BATCH_STEPS; }

int batch_max_blocks(int recovery, int block_threads)
{
    if (block_threads == 128)
        return recovery == 1 ? batch_max_blocks_per_sm<2, 128>() : batch_max_blocks_per_sm<0, 128>();
    if (block_threads == 64)
        return recovery == 1 ? batch_max_blocks_per_sm<2, 64>() : batch_max_blocks_per_sm<0, 64>();
    return -1;
}

cudaError_t launch_batch(int recovery, int block_threads, const ModelConst<float>& K,
                         const BatchLaunch& b, int grid, cudaStream_t s)
{
    if (block_threads == 128)
        return recovery == 1 ? batch_launch_t<2, 128>(K, b, grid, s) : batch_launch_t<0, 128>(K, b, grid, s);
    if (block_threads == 64)
        return recovery == 1 ? batch_launch_t<2, 64>(K, b, grid, s) : batch_launch_t<0, 64>(K, b, grid, s);
    return cudaErrorInvalidValue;
}

} // namespace lbk
