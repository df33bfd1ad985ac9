// line.cuh -- launch interface of the 1-D step (line.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.cuh"

namespace lbk {

// How a 1-D grid is cut: blocks of `threads` lanes, one cell each, of which the middle
// threads - 4 steps are the block's own; `steps` time steps run in one launch.
struct LinePlan {
    int threads, steps, grid;
    bool split; // FP64 without records on a short grid: the block's four warps share 32 cells
};
// precision: 0 = FP64, 1 = FP32; tne: launches may keep records
LinePlan line_plan(int precision, int nx, bool tne);

struct LineArgs {
    const void* in;        // state at t_n, 17 planes
    void* out;             // state at t_{n + nsteps}
    int64_t out_stride;    // > 0: every state is kept, t_{n+1+s} at out + s * out_stride (elements)
    int nsteps;            // 1 .. plan.steps
    // an SSP Runge-Kutta stage (nsteps = 1), as StepLaunch has it
    const void* prev;
    int stage;
    double wprev, wnew;
    double* partials;      // [plan.steps][TNE_PART][grid], null without TNE
    DevCounters* ctr;
    int tne_every;         // 0 = off
};

// TNE records of a launch that left the partials of `slots` steps (slot-major): a record
// for each due step, into the history ring.
cudaError_t launch_tne_finish_steps(const double* partials, int grid, int slots, TneRecord* hist,
                                    int hist_cap, int tne_every, const DevCounters* ctr, double area,
                                    cudaStream_t s);

cudaError_t launch_line(int precision, int recovery, const void* K, const LinePlan& p,
                        const LineArgs& a, cudaStream_t s);

} // namespace lbk
