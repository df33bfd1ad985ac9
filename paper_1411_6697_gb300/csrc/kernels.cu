// kernels.cu -- the kernels around a step (equilibrium start, macroscopic fields, TNE of a
// state, the grid-wide TNE record of a step) and the choice of the 2-D step kernel: FP64 grids
// and small FP32 grids run tile_kernel (tile.cu), other FP32 grids march_kernel (march.cu);
// 1-D grids run line_kernel (line.cu).
#include <float.h>

#include "cell.cuh"
#include "kernels.cuh"
#include "line.cuh"
#include "reduce.cuh"
#include "tile.cuh"

namespace lbk {

namespace {

// ------------------------------------------------------------ init, macros, TNE
template <typename R>
__global__ void init_kernel(const ModelConst<double> K, const double* rho, const double* ux,
                            const double* uy, const double* T, const double* lam, R* state)
{
    const int64_t n = (int64_t)K.nx * K.ny;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n;
         c += (int64_t)gridDim.x * blockDim.x) {
        const int y = (int)(c / K.nx), x = (int)(c - (int64_t)y * K.nx);
        double q[16], f[16];
        feq_moments(K.DI, rho[c], ux[c], uy[c], T[c], q);
        inverse_moments(K, q, f);
        const int64_t g = (int64_t)y * K.pitch + x;
#pragma unroll
        for (int i = 0; i < 16; i++) state[i * K.plane + g] = (R)f[i];
        state[16 * K.plane + g] = (R)(lam ? lam[c] : 0.0);
    }
}

template <typename R>
__global__ void macros_kernel(const ModelConst<double> K, const R* state, double* rho,
                              double* ux, double* uy, double* T, double* p, double* lam)
{
    const int64_t n = (int64_t)K.nx * K.ny;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n;
         c += (int64_t)gridDim.x * blockDim.x) {
        const int y = (int)(c / K.nx), x = (int)(c - (int64_t)y * K.nx);
        const int64_t g = (int64_t)y * K.pitch + x;
        R f[16];
#pragma unroll
        for (int i = 0; i < 16; i++) f[i] = state[i * K.plane + g];
        double r, u, v, t;
        recover_f64(K.cd, K.wd, K.inv_DId, f, r, u, v, t);
        if (rho) rho[c] = r;
        if (ux) ux[c] = u;
        if (uy) uy[c] = v;
        if (T) T[c] = t;
        if (p) p[c] = r * t;
        if (lam) lam[c] = (double)state[16 * K.plane + g];
    }
}

constexpr int TNE_THREADS = 256;

template <typename R>
__global__ void __launch_bounds__(TNE_THREADS)
    tne_kernel(const ModelConst<double> K, const R* state, double* delta, double* partials,
               DevCounters* ctr, TneRecord* out, double area)
{
    __shared__ double ssum[TNE_THREADS / 32][NSUM];
    __shared__ double smm[TNE_THREADS / 32][NMM];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double acc[NSUM], mn[TNE_K], mx[TNE_K];
    for (int q = 0; q < NSUM; q++) acc[q] = 0.0;
    for (int k = 0; k < TNE_K; k++) mn[k] = DBL_MAX, mx[k] = -DBL_MAX;
    const int64_t n = (int64_t)K.nx * K.ny;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n;
         c += (int64_t)gridDim.x * blockDim.x) {
        const int y = (int)(c / K.nx), x = (int)(c - (int64_t)y * K.nx);
        const int64_t g = (int64_t)y * K.pitch + x;
        double f[16], m[16], q[16];
#pragma unroll
        for (int i = 0; i < 16; i++) f[i] = (double)state[i * K.plane + g];
        forward_moments(K, f, m);
        const double r = m[0], u = m[1] / r, v = m[2] / r;
        const double t = (m[3] / r - (u * u + v * v)) * K.inv_DId;
        feq_moments(K.DI, r, u, v, t, q);
        double d2 = 0.0;
        for (int k = 0; k < 16; k++) {
            double D = k < 4 ? 0.0 : m[k] - q[k];
            if (delta) delta[k * n + c] = D;
            if (k >= 4) {
                acc[k - 4] += D;
                acc[TNE_K + k - 4] += fabs(D);
                mn[k - 4] = fmin(mn[k - 4], D);
                mx[k - 4] = fmax(mx[k - 4], D);
                d2 += D * D;
            }
        }
        acc[2 * TNE_K] += sqrt(d2);
        acc[2 * TNE_K + 1] += d2;
    }
    for (int q = 0; q < NSUM; q++) {
        double s = warp_sum(acc[q]);
        if (lane == 0) ssum[warp][q] = s;
    }
    for (int k = 0; k < TNE_K; k++) {
        double a = warp_min(mn[k]), b = warp_max(mx[k]);
        if (lane == 0) smm[warp][k] = a, smm[warp][TNE_K + k] = b;
    }
    __syncthreads();
    double* part = partials + blockIdx.x; // quantity-major, stride gridDim.x
    const size_t ps = gridDim.x;
    if (threadIdx.x < NSUM) {
        double s = 0.0;
        for (int w = 0; w < TNE_THREADS / 32; w++) s += ssum[w][threadIdx.x];
        const int q = threadIdx.x;
        part[ps * (q < 2 * TNE_K ? q : 4 * TNE_K + (q - 2 * TNE_K))] = s;
    } else if (threadIdx.x >= 32 && threadIdx.x < 32 + NMM) {
        const int q = threadIdx.x - 32;
        double v = smm[0][q];
        for (int w = 1; w < TNE_THREADS / 32; w++)
            v = q < TNE_K ? fmin(v, smm[w][q]) : fmax(v, smm[w][q]);
        part[ps * (2 * TNE_K + q)] = v;
    }
    __threadfence();
    __syncthreads();
    __shared__ unsigned int s_last;
    if (threadIdx.x == 0) s_last = (atomicAdd(&ctr->arrivals, 1u) == gridDim.x - 1) ? 1u : 0u;
    __syncthreads();
    if (s_last) {
        __threadfence();
        finish_tne(partials, gridDim.x, out, ctr->step, area);
        __syncthreads();
        if (threadIdx.x == 0) ctr->arrivals = 0u;
    }
}

int sm_count()
{
    static int sms = -1;
    if (sms < 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    return sms;
}

int elementwise_grid(int64_t n, int threads)
{
    int64_t g = (n + threads - 1) / threads;
    int64_t cap = (int64_t)sm_count() * 16;
    return (int)(g < cap ? (g < 1 ? 1 : g) : cap);
}

} // namespace

static bool general_sides(const int sbc[4])
{
    return sbc[0] >= 2 || sbc[1] >= 2 || sbc[2] >= 2 || sbc[3] >= 2;
}

namespace {
constexpr int FIN_THREADS = 256;

// Block (q, slot) reduces quantity q of the partials of the launch's slot-th step
// (quantity-major: partials[(slot * TNE_PART + q) * nblocks + b]) in a fixed order --
// thread t takes blocks t, t + 256, ..., then the lanes in a shuffle tree and the warps in
// order -- and writes it into the step's record, if the step was due and its record is not
// already overwritten by a later one of the same launch.
__global__ void __launch_bounds__(FIN_THREADS)
    tne_finish_kernel(const double* __restrict__ partials, int nblocks, TneRecord* hist,
                      int hist_cap, int tne_every, const DevCounters* ctr, double area)
{
    const int slot = blockIdx.y, steps = ctr->tne_pending;
    if (slot >= steps) return;
    const int64_t step = ctr->tne_step + slot;
    if (step % tne_every) return;
    const int64_t after = (ctr->tne_step + steps - 1) / tne_every - step / tne_every; // later records
    if (after >= hist_cap) return;
    __shared__ double wsum[FIN_THREADS / 32];
    const int q = blockIdx.x, t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int kind = tne_kind(q);
    double acc = kind == 0 ? 0.0 : (kind == 1 ? DBL_MAX : -DBL_MAX);
    const double* pq = partials + ((size_t)slot * TNE_PART + q) * nblocks;
    for (int b = t; b < nblocks; b += FIN_THREADS) acc = tne_comb(kind, acc, __ldcg(pq + b));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc = tne_comb(kind, acc, __shfl_xor_sync(0xffffffffu, acc, o));
    if (lane == 0) wsum[w] = acc;
    __syncthreads();
    if (t != 0) return;
    for (int k = 1; k < FIN_THREADS / 32; k++) acc = tne_comb(kind, acc, wsum[k]);
    TneRecord* rec = hist + (ctr->hist_count - 1 - after) % hist_cap;
    if (q < TNE_K) rec->sum[q + 4] = acc * area;
    else if (q < 2 * TNE_K) rec->abs_sum[q - TNE_K + 4] = acc * area;
    else if (q < 3 * TNE_K) rec->min[q - 2 * TNE_K + 4] = acc;
    else if (q < 4 * TNE_K) rec->max[q - 3 * TNE_K + 4] = acc;
    else if (q == 4 * TNE_K) rec->d_sum = acc * area;
    else rec->d2_sum = acc * area;
    if (q == 0) {
        for (int k = 0; k < 4; k++) rec->sum[k] = rec->abs_sum[k] = rec->min[k] = rec->max[k] = 0.0;
        rec->step = step;
    }
}
} // namespace

cudaError_t launch_tne_finish_steps(const double* partials, int grid, int slots, TneRecord* hist,
                                    int hist_cap, int tne_every, const DevCounters* ctr, double area,
                                    cudaStream_t s)
{
    tne_finish_kernel<<<dim3(TNE_PART, slots), FIN_THREADS, 0, s>>>(partials, grid, hist, hist_cap,
                                                                    tne_every, ctr, area);
    return cudaGetLastError();
}

cudaError_t launch_tne_finish(const StepLaunch& a, cudaStream_t s)
{
    return launch_tne_finish_steps(a.partials, a.grid, 1, a.hist, a.hist_cap, a.tne_every, a.ctr,
                                   a.cell_area, s);
}

int step_grid(int precision, int recovery, int nx, int ny, const int sbc[4], bool tne)
{
    if (precision == 0 || tile_takes_f32(recovery, nx, ny)) return tile_grid(precision, recovery, nx, ny, tne);
    return march_grid(recovery | (general_sides(sbc) ? 2 : 0) | (tne ? 8 : 0), nx, ny);
}

cudaError_t launch_step(int precision, int recovery, const void* K, const StepLaunch& a,
                        cudaStream_t s)
{
    if (precision == 0) return launch_tile(0, 0, K, a, s);
    const ModelConst<float>& Kf = *static_cast<const ModelConst<float>*>(K);
    if (tile_takes_f32(recovery, Kf.nx, Kf.ny)) return launch_tile(1, recovery, K, a, s);
    return launch_march(recovery | (general_sides(Kf.sbc) ? 2 : 0) | (a.srt ? 4 : 0) |
                            (a.tne_every > 0 ? 8 : 0),
                        Kf, a, s);
}

cudaError_t launch_init(int precision, const ModelConst<double>& Kd, const double* rho,
                        const double* ux, const double* uy, const double* T, const double* lam,
                        void* state, cudaStream_t s)
{
    const int64_t n = (int64_t)Kd.nx * Kd.ny;
    const int g = elementwise_grid(n, 256);
    if (precision == 0)
        init_kernel<double><<<g, 256, 0, s>>>(Kd, rho, ux, uy, T, lam, (double*)state);
    else
        init_kernel<float><<<g, 256, 0, s>>>(Kd, rho, ux, uy, T, lam, (float*)state);
    return cudaGetLastError();
}

cudaError_t launch_macros(int precision, const ModelConst<double>& Kd, const void* state,
                          double* rho, double* ux, double* uy, double* T, double* p,
                          double* lam, cudaStream_t s)
{
    const int64_t n = (int64_t)Kd.nx * Kd.ny;
    const int g = elementwise_grid(n, 256);
    if (precision == 0)
        macros_kernel<double><<<g, 256, 0, s>>>(Kd, (const double*)state, rho, ux, uy, T, p, lam);
    else
        macros_kernel<float><<<g, 256, 0, s>>>(Kd, (const float*)state, rho, ux, uy, T, p, lam);
    return cudaGetLastError();
}

namespace {
// rows of `units` vectors of type V from pitched to packed storage; block (c, r) takes 1024 vectors
// of row r, r + gridDim.y, ... of all planes
template <typename V>
__global__ void __launch_bounds__(256)
    pack_kernel(const V* __restrict__ src, V* __restrict__ dst, int64_t plane, int pitch, int units, int ny,
                int64_t rows, unsigned* counter, unsigned lo, unsigned hi)
{
    const int x = blockIdx.x * 1024 + threadIdx.x;
    for (int64_t r = blockIdx.y; r < rows; r += gridDim.y) {
        const int64_t p = r / ny, y = r - p * ny;
        const V* in = src + p * plane + y * pitch;
        V* out = dst + r * units;
        V v[4];
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (x + 256 * k < units) v[k] = __ldcs(in + x + 256 * k);
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (x + 256 * k < units) out[x + 256 * k] = v[k];
    }
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        counter[0] = lo;
        counter[1] = hi;
    }
}
} // namespace

// One kernel instead of a 2-D copy per plane and one for the counter: 17 or 25 copies of a few us
// each (FP32 shock reflection, 300 x 100: 64 steps and a snapshot took 0.80 ms, now 0.71; a copy of
// its 2 MB, 8 us). 16-byte vectors where the row length and dst allow them (the pitch always
// does), elements otherwise.
// Whether launch_pack may write there: memory of the state's device, aligned to an element, that
// device being the current one (a kernel launches on the stream of no other). Memory of another
// device or of the host, or another current device, is left to the copies, which need no peer access.
bool can_pack(int elem, const void* state, const void* dst)
{
    cudaPointerAttributes to, from;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&to, dst) != cudaSuccess ||
        cudaPointerGetAttributes(&from, state) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return pack_there(elem, reinterpret_cast<uintptr_t>(dst), to.type == cudaMemoryTypeDevice, to.device, from.device,
                      dev);
}

cudaError_t launch_pack(int elem, int planes, const void* state, int64_t plane_elems, int pitch, int nx,
                        int ny, void* dst, int64_t step, cudaStream_t s)
{
    const int64_t bytes = (int64_t)planes * nx * ny * elem, rows = (int64_t)planes * ny;
    const bool wide = (int64_t)nx * elem % 16 == 0 && reinterpret_cast<uintptr_t>(dst) % 16 == 0;
    const int per = wide ? 16 / elem : 1, units = nx / per;
    const dim3 grid((units + 1023) / 1024, (unsigned)(rows < 32768 ? rows : 32768));
    unsigned* counter = reinterpret_cast<unsigned*>(static_cast<char*>(dst) + bytes);
    const unsigned lo = (unsigned)(uint64_t)step, hi = (unsigned)((uint64_t)step >> 32);
#define LBK_PACK(V, D)                                                                                        \
    pack_kernel<V><<<grid, 256, 0, s>>>(static_cast<const V*>(state), static_cast<V*>(dst), plane_elems / (D), \
                                        pitch / (D), units, ny, rows, counter, lo, hi)
    if (wide) LBK_PACK(float4, per);
    else if (elem == 8) LBK_PACK(double, 1);
    else LBK_PACK(float, 1);
#undef LBK_PACK
    return cudaGetLastError();
}

int tne_grid(int nx, int ny) { return elementwise_grid((int64_t)nx * ny, TNE_THREADS); }

cudaError_t launch_tne(int precision, const ModelConst<double>& Kd, const void* state,
                       double* delta, double* partials, int grid, DevCounters* ctr,
                       TneRecord* out, double area, cudaStream_t s)
{
    if (precision == 0)
        tne_kernel<double><<<grid, TNE_THREADS, 0, s>>>(Kd, (const double*)state, delta,
                                                        partials, ctr, out, area);
    else
        tne_kernel<float><<<grid, TNE_THREADS, 0, s>>>(Kd, (const float*)state, delta, partials,
                                                       ctr, out, area);
    return cudaGetLastError();
}

} // namespace lbk
