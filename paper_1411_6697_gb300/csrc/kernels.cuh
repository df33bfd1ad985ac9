// kernels.cuh -- launch interface between the C ABI and the CUDA kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "model.h"

namespace lbk {

// Device-side bookkeeping shared by the kernels of one handle.
struct DevCounters {
    int64_t step;          // steps taken (advanced by the last block of each step)
    int64_t hist_count;    // TNE records written so far
    unsigned int arrivals; // blocks of the current launch that finished (reset by the last)
    int status;            // bit 0: non-finite or non-positive rho or T seen
    int tne_pending;       // the launch just finished left TNE partials (set every step)
    int pad;
    int64_t tne_step;      // step index of those partials
};

// One on-the-fly TNE record, laid out like lbkm_tne_global.
struct TneRecord {
    double sum[16], abs_sum[16], min[16], max[16];
    double d_sum, d2_sum;
    int64_t step;
};

// An encoded TMA tensor map (the driver's opaque 128-byte CUtensorMap).
struct alignas(64) TmaDesc {
    unsigned long long w[16];
};

struct StepLaunch {
    const void* in;      // state at t_n  [17][ny][pitch]
    void* out;           // state at t_n+1
    // stage: 0 forward Euler step; 1 first stage of an SSP Runge-Kutta step (writes
    // E(u^n), reduces the TNE of u^n, does not advance the step counter); 2 last stage
    // (writes wprev * prev + wnew * E(in) with prev = u^n, no TNE, advances the
    // counter); 3 a middle stage (the same weighted write, no TNE, no counter)
    const void* prev;
    int stage;
    double wprev, wnew;
    double* partials;    // [grid][TNE_PART]
    DevCounters* ctr;
    TneRecord* hist;     // ring of hist_cap records
    int hist_cap;
    int tne_every;       // 0 = off
    int grid;            // blocks launched
    double cell_area;    // dx * dy
    const TmaDesc* tm_in;  // host copies of the tensor maps of in (loads) and out (stores),
    const TmaDesc* tm_out; // FP32 2-D grids only
    int srt;               // 1: single-relaxation-time collision (equal rates, no TNE)
};

// Grid-wide TNE record of the partials a step left (if its schedule reduced TNE): one
// block per quantity, each a fixed-order reduction over the step's blocks, written into
// history slot (hist_count - 1) % hist_cap. Launched after every full step.
cudaError_t launch_tne_finish(const StepLaunch& a, cudaStream_t s);

// precision: 0 = FP64, 1 = FP32; recovery: 0 = FP64, 1 = double-float (FP32 only)
// (2-D grids; 1-D grids: launch_line, line.cuh)
cudaError_t launch_step(int precision, int recovery, const void* K, const StepLaunch& a,
                        cudaStream_t s);
// Blocks to launch for a step on this grid (multiple of the SM count times the
// resident blocks per SM, capped by the number of tiles).
// sbc: the side conditions (walls, Dirichlet or specular sides select the general
// variant of the FP32 marching kernel); tne: the handle keeps TNE records
int step_grid(int precision, int recovery, int nx, int ny, const int sbc[4], bool tne);

cudaError_t launch_init(int precision, const ModelConst<double>& Kd, const double* rho,
                        const double* ux, const double* uy, const double* T, const double* lam,
                        void* state, cudaStream_t s);
cudaError_t launch_macros(int precision, const ModelConst<double>& Kd, const void* state,
                          double* rho, double* ux, double* uy, double* T, double* p,
                          double* lam, cudaStream_t s);
// A state snapshot on the device: `planes` planes of ny rows of nx elements (4 or 8 bytes) packed
// into dst, then the step counter; for the destinations that can_pack accepts.
bool can_pack(int elem, const void* state, const void* dst);
// the rule itself: devices of the state, of dst and the current one, and dst's alignment
inline bool pack_there(int elem, uintptr_t dst, bool device_memory, int dst_dev, int state_dev, int current)
{
    return dst % elem == 0 && device_memory && dst_dev == state_dev && current == state_dev;
}
cudaError_t launch_pack(int elem, int planes, const void* state, int64_t plane_elems, int pitch, int nx,
                        int ny, void* dst, int64_t step, cudaStream_t s);
// TNE fields (optional) and grid-wide record of a state, all FP64.
cudaError_t launch_tne(int precision, const ModelConst<double>& Kd, const void* state,
                       double* delta, double* partials, int grid, DevCounters* ctr,
                       TneRecord* out, double cell_area, cudaStream_t s);
int tne_grid(int nx, int ny);

// Batched 1-D instances (batch.cu): per-instance parameters, work items and the
// arguments of one persistent launch.
struct InstParam {
    float S[16];
    float A8c, A9c, chem, om1, om2; // (S5-S8)/S5, (S7-S9)/S7, 2Q/((D+I)dt), omega1, omega2
    int32_t nx;
    int64_t off; // first cell of the instance in the flat layout
};
struct BatchItem {
    int32_t inst, x0; // instance and first cell of the segment
};
struct BatchLaunch {
    void* buf[2];
    int cur;             // buffer holding the input of the first step
    const InstParam* inst;
    const BatchItem* items;
    int nitems;
    DevCounters* ctr;
    unsigned* bar;       // grid barrier: arrivals, generation
    int nsteps;
    int phantom_blocks;  // > 0 only to test the bounded barrier wait
    long long wait_ns;   // bound of each barrier wait
};
int batch_segment(int block_threads); // cells of a work item
int batch_phases(int nsteps);         // passes over the state (buffer swaps) of nsteps steps
int batch_max_blocks(int recovery, int block_threads);
cudaError_t launch_batch(int recovery, int block_threads, const ModelConst<float>& K,
                         const BatchLaunch& b, int grid, cudaStream_t s);
// grid-wide TNE record of every instance (one block per instance, FP64)
cudaError_t launch_tne_instances(int precision, const ModelConst<double>& Kd, const void* state,
                                 const InstParam* inst, int n_inst, TneRecord* out,
                                 double area, cudaStream_t s);

// FP32 2-D step: y-marching strips, two cells per thread (march.cu)
// mode = recovery | (general side conditions << 1) | (single relaxation time << 2) | (TNE << 3)
// Tensor maps of an FP32 state buffer for the step kernel's bulk tensor copies: loads of
// a box of BW + 8 columns x 2 rows x 17 planes, stores of BW x 2 x 17.
cudaError_t march_tensor_maps(const void* state, int nx, int ny, int pitch, int64_t plane,
                              TmaDesc* load, TmaDesc* store);
int march_grid(int mode, int nx, int ny);
// The strip height of least cost for nsx columns of strips on G resident blocks, at most `cap` (even)
// rows; `cost` of (strips, rows). Of the heights with the same number of strips the smallest is the
// cheapest, so only those are tried: about 2 sqrt(ny) of them (every even height up to ny took 1.7 ms
// a launch at a million rows).
template <typename Cost>
inline int march_rows(int ny, int cap, int nsx, Cost cost, int* tried = nullptr)
{
    int best_rows = 2, n = 0;
    double best = 1e300;
    for (int r = 2; r <= cap; n++) {
        const int k = (ny + r - 1) / r; // strips of a column
        const double t = cost((long)nsx * k, r);
        if (t <= best) best = t, best_rows = r;
        if (k == 1) break;
        const int next = ((ny + k - 2) / (k - 1) + 1) & ~1; // the least even height with fewer
        r = next > r ? next : r + 2;
    }
    if (tried) *tried = n + 1;
    return best_rows;
}
cudaError_t launch_march(int mode, const ModelConst<float>& K, const StepLaunch& a,
                         cudaStream_t s);

} // namespace lbk
