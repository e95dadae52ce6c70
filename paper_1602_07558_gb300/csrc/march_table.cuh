// The updates' marching forms, as the host code sees them (march.cuh).
#pragma once
#include "kernels.cuh"

namespace swept {

// Functions of one update's marching form (march_*.cu).
struct MarchTable {
    // the shape for these grids; -1 where the swept kernels with these tile sides, in
    // the launch-per-phase or the persistent form, do better (without tile sides, a
    // shape in any case); c: the update's constants (heat's r)
    int (*shape)(const int *nx, const int *ny, const int *tile, int count, bool persistent,
                 const double *c);
    int (*steps)(int shape);     // steps a phase
    MarchGrid (*cut)(int shape, int nx, int ny);
    // ints of the counters that `one` needs, its own error word included
    long long (*words)(int shape, int nx, int ny);
    // whether an advance of so few sub-steps of one grid is quicker by naive launches
    // (made one by one or from a graph)
    bool (*is_short)(int shape, int nx, int ny, int tile, long long substeps, bool graph);
    // the shape whose walks (phase_one) are the quickest for the naive sub-steps of
    // one grid, -1 for a thread a point
    int (*naive_shape)(int nx, int ny, const double *c);
    // one grid (`g` its cut), or the tiles of a batch's table; without `err` (heat
    // alone) the result, which *out names beforehand, becomes NaN where a wait gives up
    cudaError_t (*one)(int shape, const MarchGrid &g, const double *c, const void *src, void *b0,
                       void *b1, int *sched, long long steps, int *err, int first,
                       long long spin_limit, void **out, long long *launches, cudaStream_t);
    cudaError_t (*many)(int shape, const GridDesc *grids, const int2 *tiles, int NT,
                        const double *c, const void *src, void *b0, void *b1, int *sched,
                        long long steps, int *err, void **out, long long *launches, cudaStream_t);
    // one sub-step by walks as one launch, the naive path: `g` the grid's naive_cut;
    // Euler in place (dst == src)
    MarchGrid (*naive_cut)(int shape, int nx, int ny);
    cudaError_t (*phase_one)(int shape, const MarchGrid &g, const double *c, const void *src,
                             void *dst, int phase, cudaStream_t);
    cudaError_t (*phase_many)(int shape, const GridDesc *grids, const int2 *tiles, int NT,
                              const double *c, void *state, int phase, cudaStream_t);
};

// Whether a batch's naive sub-steps are walks (phase_many) rather than a thread a
// point. Measured on the GB300, us a step in a graph, a thread a point / walks:
// binary64 64 grids of 16..48 53 / 42, 256 of 32..96 470 / 469, 256 of 32..512 7498 /
// 5478; binary32 64 of 16..48 8.2 / 8.6, 40 of 64..160 20.6 / 18.7, 256 of 32..96 48 /
// 33, 256 of 32..512 808 / 420.
inline bool batch_naive_walks(bool euler, bool euler_kahan, double points) {
    return euler || (euler_kahan && points >= 2e5);
}

const MarchTable *marchtable_heat();
const MarchTable *marchtable_heat_kahan_f32();
const MarchTable *marchtable_heat_kahan_bf16();
const MarchTable *marchtable_euler();
const MarchTable *marchtable_euler_kahan_f32();
const MarchTable *marchtable_euler_kahan_bf16();

}  // namespace swept
