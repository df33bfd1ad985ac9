// The discrete adjoint's reverse sweep and the objective without its derivative (adjoint.cu).
#pragma once
#include "kernels.cuh"

namespace lbk {

constexpr int ADJ_NPAR = 15; // dJ/dS_5..S_16, dJ/dQ, dJ/domega1, dJ/domega2
struct AdjArgs {
    const double* f;     // a state: 17 planes with the handle's pitch
    const double* fb1;   // dJ/df of it, [16][nx] (launch_adj_rho0)
    double *fb0, *lb0;   // dJ/df and dJ/dlambda of the final state (launch_adj_seed)
    double* jacc;        // [grid] per-block objective accumulators
    double jw;           // w_tne dx dt for the objective value
};
int adj_grid(int nx);
cudaError_t launch_adj_seed(const ModelConst<double>& K, const AdjArgs& a, const double* rho_t,
                            double w, int grid, cudaStream_t s);
cudaError_t launch_adj_rho0(const ModelConst<double>& K, const AdjArgs& a, double* drho0,
                            int grid, cudaStream_t s);
// n floats widened to doubles (an FP32 forward run's checkpoint, to restart a segment in FP64)
cudaError_t launch_adj_widen(const float* in, double* out, size_t n, int grid, cudaStream_t s);

// How the reverse sweep cuts a grid: blocks of `threads` cells, of which the middle
// threads - 4 steps - 4 are the block's own, `steps` reverse steps per launch.
struct AdjPlan {
    int threads, steps, grid;
};
AdjPlan adj_plan(int nx);

struct AdjReverse {
    const double* state; // the last state to reverse, 17 planes with the handle's pitch
    int64_t stride;      // elements from a state back to the one before
    int steps;           // states to reverse, 1 .. plan.steps
    const double *fb1, *lb1; // dJ/df [16][nx] and dJ/dlambda [nx] after the last step
    double *fb0, *lb0;       // the same before the first
    double* pacc;        // [ADJ_NPAR][plan.grid] per-block parameter accumulators
    double* jacc;        // [plan.grid] per-block objective accumulators
    double jw;           // w_tne dx dt for the objective value
};
// tne_w: w_tne dx dt, Delta_b += 2 tne_w Delta
cudaError_t launch_adj_reverse(const ModelConst<double>& K, const AdjReverse& a, const AdjPlan& p,
                               double tne_w, cudaStream_t s);

// Adds w_tne dx dt sum_x d^2 of the FP64 state a.f (d^2 = sum_{k=5..16} Delta_k^2,
// Sec. VI, Eq. (91); rho, u, T recovered in the kernel) to the per-block accumulators
// a.jacc[grid].
cudaError_t launch_adj_jtne(const ModelConst<double>& K, const AdjArgs& a, int grid,
                            cudaStream_t s);

} // namespace lbk
