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
};

const MarchTable *marchtable_heat();
const MarchTable *marchtable_heat_kahan_f32();
const MarchTable *marchtable_heat_kahan_bf16();
const MarchTable *marchtable_euler();
const MarchTable *marchtable_euler_kahan_f32();
const MarchTable *marchtable_euler_kahan_bf16();

}  // namespace swept
