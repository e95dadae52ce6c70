// The updates' marching forms, as the host code sees them (march.cuh).
#pragma once
#include "kernels.cuh"

namespace swept {

// Functions of one update's marching form (march_*.cu).
struct MarchTable {
    // the shape for these grids; -1 (unless `always`): the swept kernels do better
    int (*shape)(const int *nx, const int *ny, int count, bool always);
    int (*steps)(int shape);     // steps a phase
    MarchGrid (*cut)(int shape, int nx, int ny);
    // one grid (`g` its cut), or the tiles of a batch's table
    cudaError_t (*one)(int shape, const MarchGrid &g, const double *c, const void *src, void *b0,
                       void *b1, int *sched, long long steps, int *err, int first,
                       long long spin_limit, void **out, long long *launches, cudaStream_t);
    cudaError_t (*many)(int shape, const GridDesc *grids, const int2 *tiles, int NT,
                        const double *c, const void *src, void *b0, void *b1, int *sched,
                        long long steps, int *err, void **out, long long *launches, cudaStream_t);
    // one sub-step in place (Euler), as one launch: the naive path
    cudaError_t (*phase_one)(int shape, const MarchGrid &g, const double *c, void *state, int phase,
                             cudaStream_t);
    cudaError_t (*phase_many)(int shape, const GridDesc *grids, const int2 *tiles, int NT,
                              const double *c, void *state, int phase, cudaStream_t);
};

// Whether Euler's naive sub-steps, one launch each, are walks of the marching form
// (every point's fluxes formed once) rather than a thread a point, which forms its
// four neighbours' fluxes but has the shorter chain. Measured on the GB300, us a
// step in a graph, a thread a point / walks: binary64 64² 18.3 / 16.8, 200² 34.4 /
// 25.0, 2048² 1747 / 1260; binary32 64² 3.7 / 4.5, 400 x 300 6.1 / 6.1, 1009 x 757
// 24.5 / 18.6, 2048² 163 / 98.6; bfloat16 400 x 300 6.1 / 6.3, 2048² 141 / 66.
inline bool naive_walks(bool euler, bool euler_kahan, double points) {
    return euler || (euler_kahan && points >= 2e5);
}

const MarchTable *marchtable_heat();
const MarchTable *marchtable_heat_kahan_f32();
const MarchTable *marchtable_heat_kahan_bf16();
const MarchTable *marchtable_euler();
const MarchTable *marchtable_euler_kahan_f32();
const MarchTable *marchtable_euler_kahan_bf16();

}  // namespace swept
