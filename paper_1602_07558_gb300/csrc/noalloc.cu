// Allocation-free swept advance of the heat equation (FP64).
//
// Who needs this: callers that must not allocate device memory at the point
// where they advance a grid -- for example a host application that owns every
// device allocation through its own fixed pool and forbids cudaMalloc outside
// it, a plugin running under such an application, or a latency-critical loop
// where cudaMalloc/cudaFree would add their implicit device-wide
// synchronisation. They pass their own input and output buffers; the only
// other device memory this path touches is the file-scope array below, which
// the CUDA runtime sets up when it loads this library's device code.
//
// The marching form of swept2d_advance (march.cuh) on the caller's buffers, or, where
// the diffusion number keeps that off the integer units, the swept kernels (Up, then
// per half cycle the x/y Bridge launch and the Octahedron, a final Down, naive tail),
// so the result is bit for bit that of a handle created with op SWEPT2D_OP_HEAT and
// advanced with SWEPT2D_SWEPT from the same input. The call has returned before a
// wait of the marching form could give up, and its caller has no handle to ask: the
// block then overwrites u_out with NaN.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>

#include "../../include/swept2d.h"
#include "launch.cuh"
#include "march_table.cuh"

namespace {

constexpr size_t kScratchBytes = SWEPT2D_STATIC_SCRATCH_BYTES;

// Shared by every call on a device and kept until the process exits. Holds the
// second state buffer and the counters of the marching form, or the swept kernels'
// panels. Nothing in it has
// to start at zero: every element a call reads was written earlier in that same
// call.
static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

void set_err(char *err, int errlen, const char *msg) {
    if (err && errlen > 0) {
        strncpy(err, msg, (size_t)errlen - 1);
        err[errlen - 1] = '\0';
    }
}

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// Device address of g_scratch on the current device. In host code the name
// g_scratch is only a host-side stand-in, so the address is looked up on every
// call, with the caller's device current: a cached address would outlive a
// cudaDeviceReset or a switch to another context on the same device, after
// which the module is loaded again at another address.
int scratch_address(void **out, char *err, int errlen) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess || !p) {
        set_err(err, errlen, e != cudaSuccess ? cudaGetErrorString(e)
                                              : "cudaGetSymbolAddress returned NULL");
        return SWEPT2D_ECUDA;
    }
    *out = p;
    return SWEPT2D_OK;
}

// The swept schedule on the caller's buffers and two panel sets, then the tail, whose
// last sub-step lands in u_out (`tmp`: one state copy, where there is a tail).
cudaError_t advance_swept(const swept::Geom &G, const double *consts, const double *u_in,
                          double *u_out, void *up, void *br, double *tmp, long long nsteps,
                          cudaStream_t st) {
    const swept::OpTable *t = swept::optable_heat();
    const swept::Tuning tn;   // 256 threads, per-level prefetch (the handle path's heat default)
    const int half = G.n / 2;
    const long long H = nsteps / half, rem = nsteps - H * half;
    const double *src = u_in;
    cudaError_t e = cudaSuccess;
    if (H > 0) {
        double *to = rem % 2 == 1 ? tmp : u_out;
        e = t->up(G, consts, u_in, up, 0, 0, st);
        for (long long j = 0; j < H && e == cudaSuccess; ++j) {
            const u64 g0 = (u64)j * half;
            const int o = (j & 1) ? half : 0;
            e = t->bridge(G, consts, up, br, g0, nullptr, tn, st);
            if (e == cudaSuccess)
                e = j + 1 < H ? t->octahedron(G, consts, br, up, o, g0, nullptr, tn, st)
                              : t->down(G, consts, br, to, o, g0, nullptr, tn, st);
        }
        src = to;
    }
    for (long long i = 0; i < rem && e == cudaSuccess; ++i) {
        double *to = (rem - 1 - i) % 2 == 0 ? u_out : tmp;
        e = t->naive(G, consts, src, to, (u64)(H * half + i), st);
        src = to;
    }
    return e;
}

// The advance; `skip` (the wait-timeout self-test): its first phase is skipped.
int advance_static(const double *u_in, double *u_out, int nx, int ny, int tile, double r,
                   long long nsteps, bool skip, long long spin_limit, void *stream, char *err,
                   int errlen) {
    set_err(err, errlen, "");
    if (!u_in || !u_out) {
        set_err(err, errlen, "u_in and u_out must be device pointers");
        return SWEPT2D_EINVAL;
    }
    if (nx < 1 || ny < 1 || nsteps < 0) {
        set_err(err, errlen, "need nx, ny >= 1 and nsteps >= 0");
        return SWEPT2D_EINVAL;
    }
    if (tile < 4 || (tile & 1) || nx % tile || ny % tile) {
        set_err(err, errlen, "tile must be even, >= 4 and divide nx and ny");
        return SWEPT2D_EINVAL;
    }
    const size_t state_bytes = (size_t)nx * ny * sizeof(double);
    const char *in_b = (const char *)u_in, *out_b = (const char *)u_out;
    if (in_b < out_b + state_bytes && out_b < in_b + state_bytes) {
        set_err(err, errlen, "u_in and u_out must not overlap");
        return SWEPT2D_EINVAL;
    }
    const size_t smem = swept::optable_heat()->smem_for(tile, false);
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        optin = 227 * 1024;
    if (smem > (size_t)optin) {
        set_err(err, errlen, "tile too large for shared memory");
        return SWEPT2D_EINVAL;
    }
    swept::Geom G;
    G.nx = nx; G.ny = ny; G.n = tile;
    G.T = nx / tile; G.Q = ny / tile;
    G.PS = swept::panel_stride(tile);
    const size_t panel_bytes = (size_t)G.T * G.Q * 4 * G.PS * sizeof(double);
    const int half = tile / 2;
    const long long H = nsteps / half, rem = nsteps - H * half;
    const size_t need = 2 * align256(panel_bytes) + (rem > 0 ? align256(state_bytes) : 0);
    if (need > kScratchBytes) {
        char msg[200];
        snprintf(msg, sizeof msg,
                 "grid needs %zu bytes of scratch; the static scratch holds %zu bytes",
                 need, kScratchBytes);
        set_err(err, errlen, msg);
        return SWEPT2D_EINVAL;
    }
    void *base = nullptr;
    int rc = scratch_address(&base, err, errlen);
    if (rc != SWEPT2D_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    if (nsteps == 0) {
        const cudaError_t e = cudaMemcpyAsync(u_out, u_in, state_bytes, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) set_err(err, errlen, cudaGetErrorString(e));
        return e == cudaSuccess ? SWEPT2D_OK : SWEPT2D_ECUDA;
    }
    // the scratch holds the second state buffer, an error word and the marching
    // form's counters; two panel sets hold more than four times the state, so they
    // fit wherever the check above passed
    const swept::MarchTable *mt = swept::marchtable_heat();
    const double consts[8] = {r, 0, 0, 0, 0, 0, 0, 0};
    const int shape = mt->shape(&nx, &ny, nullptr, 1, false, consts);
    const swept::MarchGrid cut = mt->cut(shape, nx, ny);
    const int tiles = cut.bx * cut.by;
    void *tmp = base;
    cudaError_t e = cudaSuccess;
    if (!skip && swept::heat_ratio(r) == 0 &&
        mt->shape(&nx, &ny, &tile, 1, false, consts) < 0) {
        char *const sb = (char *)base;
        e = advance_swept(G, consts, u_in, u_out, sb, sb + align256(panel_bytes),
                          (double *)(sb + 2 * align256(panel_bytes)), nsteps, st);
        if (e != cudaSuccess) set_err(err, errlen, cudaGetErrorString(e));
        return e == cudaSuccess ? SWEPT2D_OK : SWEPT2D_ECUDA;
    }
    if (!skip && mt->is_short(shape, nx, ny, tile, nsteps, false)) {
        // naive launches, the last of which lands in u_out
        const void *src = u_in;
        for (long long i = 0; i < nsteps && e == cudaSuccess; ++i) {
            void *dst = (nsteps - 1 - i) % 2 == 0 ? (void *)u_out : tmp;
            e = swept::optable_heat()->naive(G, consts, src, dst, (unsigned long long)i, st);
            src = dst;
        }
        if (e != cudaSuccess) set_err(err, errlen, cudaGetErrorString(e));
        return e == cudaSuccess ? SWEPT2D_OK : SWEPT2D_ECUDA;
    }
    int *sched = (int *)((char *)base + align256(state_bytes));
    // the buffers alternate phase by phase; the last phase writes u_out
    if (skip) nsteps = 2LL * mt->steps(shape);
    const long long phases = (nsteps + mt->steps(shape) - 1) / mt->steps(shape);
    void *b0 = (phases & 1) ? (void *)u_out : tmp, *b1 = (phases & 1) ? tmp : (void *)u_out;
    void *out = u_out;
    long long made = 0;
    e = mt->one(shape, cut, consts, u_in, b0, b1, sched, nsteps, nullptr,
                skip ? tiles : 0, spin_limit, &out, &made, st);
    if (e != cudaSuccess) {
        char msg[200];
        snprintf(msg, sizeof msg, "marching kernel: %s", cudaGetErrorString(e));
        set_err(err, errlen, msg);
        return SWEPT2D_ECUDA;
    }
    return SWEPT2D_OK;
}

}  // namespace

extern "C" {

int swept2d_heat_advance_static(const double *u_in, double *u_out, int nx, int ny, int tile,
                                double r, long long nsteps, void *stream, char *err, int errlen) {
    return advance_static(u_in, u_out, nx, ny, tile, r, nsteps, false, swept::kPersistSpinLimit,
                          stream, err, errlen);
}

int swept2d_selftest_static_timeout(const double *u_in, double *u_out, int nx, int ny, int tile,
                                    double r, long long spin_limit, void *stream, char *err,
                                    int errlen) {
    if (spin_limit < 1) {
        set_err(err, errlen, "selftest: spin_limit < 1");
        return SWEPT2D_EINVAL;
    }
    return advance_static(u_in, u_out, nx, ny, tile, r, 1, true, spin_limit, stream, err, errlen);
}

}  // extern "C"
