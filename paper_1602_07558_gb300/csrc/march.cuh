// The marching form of an advance: one launch runs every step of one or many
// grids. The steps are cut into phases of up to K; in a phase each tile (a
// rectangle of the grid, unrelated to the caller's tile side) is read with a
// ring of K points around it, advanced K steps by one block with its values in
// registers, and written to the other state buffer. The ring is computed
// redundantly, which the swept rule avoids; in exchange a point's values stay
// in registers for the whole phase and only the warps' edge rows and columns
// pass through shared memory.
//
// Items (phase, tile) are taken in order from an atomic counter. An item of
// phase j starts once its periodic 3 x 3 tile neighbourhood has finished phase
// j - 1: those tiles hold every point its ring reads (a tile is at least K
// points wide when the grid has more than one along that side), and they are
// the only readers of the buffer it overwrites. A dependency has a smaller
// index, so the lowest unfinished item can always run, whatever number of
// blocks is resident. Waits are bounded, as in the persistent form.
#pragma once
#include <climits>
#include <cmath>
#include <type_traits>

#include "exact64.cuh"
#include "kernels.cuh"
#include "launch.cuh"
#include "march_table.cuh"

namespace swept {

// One tile of a phase.
struct MarchTile {
    MarchGrid g;
    int x0, y0, w, h;         // the tile
    int I, J, base;           // its place, and its grid's first index among the counters
    long long soff;           // first element of the grid's state in the pooled state
    const double *c;          // the grid's own update constants (nullptr: the launch's)
    // first column of tile i of a row of tiles: even, but for the grid's end
    __device__ __forceinline__ int column(int i) const {
        return i == g.bx ? g.nx : (int)((long long)i * g.nx / g.bx) & ~1;
    }
    __device__ __forceinline__ void place(int t) {
        J = t / g.bx;
        I = t - J * g.bx;
        x0 = column(I);
        y0 = (int)((long long)J * g.ny / g.by);
        w = column(I + 1) - x0;
        h = (int)((long long)(J + 1) * g.ny / g.by) - y0;
    }
};

struct OneMarch {
    MarchGrid g;
    __device__ __forceinline__ MarchTile operator()(int t) const {
        MarchTile m;
        m.g = g;
        m.base = 0;
        m.soff = 0;
        m.c = nullptr;
        m.place(t);
        return m;
    }
};

// A launch's share of an advance: `phases` phases of K steps (the last one of
// `last` steps), reading `src` in the first and then the buffer the phase
// before wrote; phase j writes buf[j & 1].
template <class S>
struct MarchRun {
    const S *src;
    S *buf[2];
    int *done, *queue, *err;   // per-tile phase counts, item counter (zeroed), error word
    int NT, phases, K, last, first;
    long long spin_limit;
};

// A ring of K columns, rounded up so that it starts at an even column.
__host__ __device__ constexpr int even_ring(int k) { return (k + 1) & ~1; }

__device__ __forceinline__ int wrap_index(int i, int n) {
    i %= n;
    return i < 0 ? i + n : i;
}

// Waits until the 3 x 3 neighbourhood of the tile has finished `need` phases.
// Returns false (the same for the whole block) when the wait gave up.
__device__ __forceinline__ bool march_wait(const MarchTile &m, const int *done, int need, int *err,
                                           long long spin_limit) {
    bool bad = false;
    if (need > 0 && threadIdx.x < 9) {
        const int dj = (int)threadIdx.x / 3 - 1, di = (int)threadIdx.x % 3 - 1;
        const int J = wrap_index(m.J + dj, m.g.by), I = wrap_index(m.I + di, m.g.bx);
        const int *flag = done + m.base + J * m.g.bx + I;
        long long it = 0;
        while (ld_acquire(flag) < need) {
            if (++it > spin_limit || ((it & 255) == 0 && ld_relaxed(err) != 0)) {
                bad = true;
                break;
            }
            __nanosleep(32);
        }
        if (bad) atomicExch(err, 2);
    }
    return __syncthreads_or(bad) == 0;
}

// The items of a run, taken until none is left; false if a wait gave up.
template <class Body, class Op, class Loc>
__device__ __forceinline__ bool march_items(const Op &op, const Loc &at,
                                            const MarchRun<typename Op::S> &run,
                                            typename Body::Smem &sm, int &s_item) {
    typedef typename Op::S S;
    const int nitems = run.NT * run.phases;
    for (;;) {
        if (threadIdx.x == 0) {
            const int it = atomicAdd(run.queue, 1) + run.first;
            s_item = ld_relaxed(run.err) ? nitems : it;
        }
        __syncthreads();
        const int item = s_item;
        if (item >= nitems) return true;
        const int j = item / run.NT, t = item - j * run.NT;
        const MarchTile m = at(t);
        if (!march_wait(m, run.done, j, run.err, run.spin_limit)) return false;
        const S *src = (j == 0 ? run.src : run.buf[(j - 1) & 1]) + m.soff;
        Body::run(m.c ? Op(m.c) : op, m, src, run.buf[j & 1] + m.soff, run.K,
                  j + 1 == run.phases ? run.last : run.K, j, sm);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) add_release(run.done + t, 1);
    }
}

// AFTER: launched without a gap to the launch before (launch_after).
template <class Body, class Op, class Loc, bool AFTER>
__global__ void __launch_bounds__(Body::kThreads, Body::kMinBlocks)
march_kernel(Op op, Loc at, MarchRun<typename Op::S> run) {
    __shared__ typename Body::Smem sm;
    __shared__ int s_item;
    if constexpr (AFTER) after_previous_launch();
    march_items<Body>(op, at, run, sm, s_item);
}

// The same for a caller that cannot ask for the error word: a block whose wait gives
// up overwrites the `points` values of the result with NaN. (Its own tile stays so,
// as no phase of it follows; blocks in the middle of theirs may still write those.)
template <class Body, class Op, class Loc, bool AFTER>
__global__ void __launch_bounds__(Body::kThreads, Body::kMinBlocks)
march_or_spoil_kernel(Op op, Loc at, MarchRun<double> run, double *result, size_t points) {
    __shared__ typename Body::Smem sm;
    __shared__ int s_item;
    if constexpr (AFTER) after_previous_launch();
    if (march_items<Body>(op, at, run, sm, s_item)) return;
    for (size_t i = threadIdx.x; i < points; i += Body::kThreads)
        result[i] = __longlong_as_double(0x7ff8000000000000LL);
}

// One phase, one tile a block: the naive path's launch per sub-step (Euler in place,
// dst == src).
template <class Body, class Op, class Loc>
__global__ void __launch_bounds__(Body::kThreads, Body::kMinBlocks)
march_phase_kernel(Op op, Loc at, const typename Op::S *src, typename Op::S *dst, int phase) {
    __shared__ typename Body::Smem sm;
    const MarchTile m = at(blockIdx.x);
    const Op own = m.c ? Op(m.c) : op;
    after_previous_launch();
    Body::run(own, m, src + m.soff, dst + m.soff, Body::K, Body::K, phase, sm);
}

// ------------------------------------------------------------------- heat
// Two values of one plane in adjacent columns. Binary32 pairs go through the
// packed instructions (one issue slot for two results; each result rounded as
// by the scalar instruction).
struct F2 {
    unsigned long long v;
    __device__ __forceinline__ float lo() const { return __uint_as_float((unsigned)v); }
    __device__ __forceinline__ float hi() const { return __uint_as_float((unsigned)(v >> 32)); }
};
struct D2 {
    double l, h;
    __device__ __forceinline__ double lo() const { return l; }
    __device__ __forceinline__ double hi() const { return h; }
};
struct L2 {
    long long l, h;
    __device__ __forceinline__ long long lo() const { return l; }
    __device__ __forceinline__ long long hi() const { return h; }
};
__device__ __forceinline__ F2 two(float l, float h) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(l), "f"(h));
    return r;
}
__device__ __forceinline__ D2 two(double l, double h) { return D2{l, h}; }
__device__ __forceinline__ L2 two(long long l, long long h) { return L2{l, h}; }
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
// a - b (the product by -1 is exact)
__device__ __forceinline__ F2 sub2(F2 a, F2 b) { return fma2(b, two(-1.0f, -1.0f), a); }
// a + b where one of them comes from two registers that are no pair yet (two
// scalar additions instead of two moves and a packed one, whose half of the FMA
// pipe is the busier: 2048² binary32, 2000 steps, 8.23 to 7.77 ms)
__device__ __forceinline__ F2 add_mixed(F2 a, F2 b) {
    return two(__fadd_rn(a.lo(), b.lo()), __fadd_rn(a.hi(), b.hi()));
}

// Two adjacent columns' east values (the second's comes from the next lane), and
// a row's pair sums E + S moved one column to the right, which makes them the
// W + N sums of the row below.
// SEG: lanes that hold one run of columns (a warp may hold several).
template <int SEG = 32>
__device__ __forceinline__ unsigned seg_lanes() {
    return SEG == 32 ? 0xffffffffu : ((1u << (SEG & 31)) - 1u) << (threadIdx.x & 31 & ~(SEG - 1));
}
template <int SEG = 32, class V2>
__device__ __forceinline__ V2 east_of(V2 v) {
    return two(v.hi(), __shfl_down_sync(seg_lanes<SEG>(), v.lo(), 1, SEG));
}
template <int SEG = 32, class V2>
__device__ __forceinline__ V2 moved_right(V2 v) {
    return two(__shfl_up_sync(seg_lanes<SEG>(), v.hi(), 1, SEG), v.lo());
}

// The values a thread keeps for two points, and their update.
template <class Op>
struct HeatCell;
template <>
struct HeatCell<HeatOp> {
    typedef double V;
    typedef D2 V2;
    static constexpr bool kComp = false;
    double r;
    __device__ __forceinline__ explicit HeatCell(const HeatOp &op) : r(op.r) {}
    __device__ static __forceinline__ V ld(double v) { return v; }
    __device__ static __forceinline__ double st(V v) { return v; }
    __device__ __forceinline__ V2 pair(V2 a, V2 b) const {
        return two(__dadd_rn(a.l, b.l), __dadd_rn(a.h, b.h));
    }
    __device__ __forceinline__ void next(V2 &u, V2 &, V2 pe, V2 pw) const {
        u = two(__fma_rn(r, __fma_rn(-4.0, u.l, __dadd_rn(pe.l, pw.l)), u.l),
                __fma_rn(r, __fma_rn(-4.0, u.h, __dadd_rn(pe.h, pw.h)), u.h));
    }
};
// The heat update in a block's fixed-point unit (exact64.cuh).
struct FixedCell {
    typedef L2 V2;
    static constexpr bool kComp = false;
    FixedHeat f;
    __device__ __forceinline__ V2 pair(V2 a, V2 b) const {
        return two(f.sum(a.l, b.l), f.sum(a.h, b.h));
    }
    __device__ __forceinline__ void next(V2 &u, V2 &, V2 pe, V2 pw) {
        u = two(f.next(u.l, pe.l, pw.l), f.next(u.h, pe.h, pw.h));
    }
};
// The storage rounding of a pair.
__device__ __forceinline__ F2 stored2(F2 a, const float *) { return a; }
__device__ __forceinline__ F2 stored2(F2 a, const __nv_bfloat16 *) {
    unsigned p;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p) : "f"(a.hi()), "f"(a.lo()));
    return two(__uint_as_float(p << 16), __uint_as_float(p & 0xffff0000u));
}
template <class SS>
struct HeatCell<HeatKahanOp<SS>> {
    typedef float V;
    typedef F2 V2;
    static constexpr bool kComp = true;
    F2 r;
    __device__ __forceinline__ explicit HeatCell(const HeatKahanOp<SS> &op) : r(two(op.r, op.r)) {}
    __device__ static __forceinline__ V ld(SS v) { return Store<SS>::ld(v); }
    __device__ static __forceinline__ SS st(V v) { return Store<SS>::st(v); }
    __device__ __forceinline__ V2 pair(V2 a, V2 b) const { return add_mixed(a, b); }
    __device__ __forceinline__ void next(V2 &u, V2 &c, V2 pe, V2 pw) const {
        const SS *s = nullptr;
        const F2 d = fma2(two(-4.0f, -4.0f), u, add_mixed(pe, pw));
        const F2 y = sub2(mul2(r, d), c);
        const F2 un = stored2(add2(u, y), s);
        c = stored2(sub2(sub2(un, u), y), s);
        u = un;
    }
};

// A block is WY warps over a region of 64 columns and R WY rows: a thread holds
// R rows of two adjacent columns. A step: the warps' first and last rows go to
// shared memory (two buffers in turn, one barrier a step), then each thread
// walks down its rows. The outermost columns and rows of the region go wrong by
// one more each step, which the ring covers; warps whose rows no later step
// needs rest. Against the swept kernels: 2048², 2,000 steps, binary32 20.1 -> 7.8 ms,
// bfloat16 15.7 -> 8.8 (the heavy half of the FMA pipe 70% busy).
template <class Op, int R_, int WY_, int MINB_, int K_>
struct HeatMarch {
    typedef typename Op::S S;
    typedef HeatCell<Op> Cell;
    typedef typename Cell::V V;
    typedef typename Cell::V2 V2;
    static constexpr int R = R_, WY = WY_, K = K_;   // K: steps a phase
    static constexpr int kThreads = 32 * WY, kMinBlocks = MINB_;
    static constexpr bool kInPlace = false;
    static constexpr int kRows = R * WY;     // the region's, of 64 columns, ring included
    static constexpr int kTileCols = 64 - 2 * even_ring(K), kTileRows = kRows - 2 * K;
    static_assert(kTileCols >= 2 * K + 4 && kTileRows >= 2 * K, "a tile is at least K points wide");
    static constexpr bool kFixed = std::is_same<Op, HeatOp>::value;
    struct Smem {
        V2 row[2][WY][2][32];    // a warp's first and last row
        int high[WY], low[WY];   // its extremes (FP64)
    };
    struct alignas(2 * sizeof(S)) Two {
        S a, b;
    };
    // Calls f(row, element of the thread's first column) for the thread's rows.
    template <class F>
    __device__ static __forceinline__ void each_row(const MarchTile &m, int gx, int gy, F &&f) {
        const size_t nx = m.g.nx, back = nx - nx * m.g.ny;   // to the next row, to the first one
        size_t at = (size_t)gy * nx + gx;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            f(j, at);
            const bool last = ++gy == m.g.ny;
            gy = last ? 0 : gy;
            at += last ? back : nx;
        }
    }

    // `steps` steps of the region's values.
    template <class C, class T, int N>
    __device__ static __forceinline__ void march(C &cell, T (&u)[R], T (&comp)[N], int rows, int r0,
                                                 int lane, int wy, int steps, T (*edge)[WY][2][32]) {
#pragma unroll 1
        for (int s = 0; s < steps; ++s) {
            T (*row)[2][32] = edge[s & 1];
            row[wy][0][lane] = u[0];
            row[wy][1][lane] = u[R - 1];
            __syncthreads();
            if (r0 + R <= s + 1 || r0 >= rows - 1 - s) continue;
            const T above = wy > 0 ? row[wy > 0 ? wy - 1 : 0][1][lane] : u[0];
            const T below = wy + 1 < WY && r0 + R < rows ? row[wy + 1 < WY ? wy + 1 : 0][0][lane]
                                                         : u[R - 1];
            T pp = cell.pair(east_of(above), u[0]);       // the row above's pair sums
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const T pe = cell.pair(east_of(u[j]), j + 1 < R ? u[j + 1 < R ? j + 1 : 0] : below);
                cell.next(u[j], comp[N > 1 ? j : 0], pe, moved_right(pp));
                pp = pe;
            }
        }
    }

    __device__ static __forceinline__ void run(const Op &op, const MarchTile &m, const S *src,
                                               S *dst, int ring, int steps, int, Smem &sm) {
        Cell cell(op);
        const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
        const int c = 2 * lane, r0 = wy * R;
        const int ring_x = even_ring(ring);
        const int cols = m.w + 2 * ring_x, rows = m.h + 2 * ring;
        const size_t plane = (size_t)m.g.nx * m.g.ny;
        // (lanes and rows beyond the region repeat its last ones: values of the
        // field's own size)
        const int gx = wrap_index(m.x0 - ring_x + min(c, (cols - 1) & ~1), m.g.nx);
        const int gy = wrap_index(m.y0 - ring + r0, m.g.ny);
        // (tiles start at even columns, so with an even nx a thread's two columns
        // are one aligned pair of an aligned plane)
        const ptrdiff_t east = gx + 1 == m.g.nx ? 1 - m.g.nx : 1;
        const bool pairs = (m.g.nx & 1) == 0 &&
                           (((size_t)src | (size_t)dst) & (2 * sizeof(S) - 1)) == 0;
        V2 u[R], comp[Cell::kComp ? R : 1];
        const auto load = [&](auto &&get) {
            each_row(m, gx, gy, [&](int j, size_t at) {
                if (j == 0 || r0 + j < rows) {
                    u[j] = get(src + at);
                    if (Cell::kComp) comp[j] = get(src + plane + at);
                } else {
                    u[j] = u[j > 0 ? j - 1 : 0];
                    if (Cell::kComp) comp[j] = comp[j > 0 ? j - 1 : 0];
                }
            });
        };
        const auto read = [&] {
            if (pairs)
                load([&](const S *p) {
                    const Two t = *reinterpret_cast<const Two *>(p);
                    return two(Cell::ld(t.a), Cell::ld(t.b));
                });
            else
                load([&](const S *p) { return two(Cell::ld(p[0]), Cell::ld(p[east])); });
        };
        read();
        bool done = false;
        if constexpr (kFixed) {
            // the block's extremes decide on the unit
            int high = INT_MIN, low = INT_MAX;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const int l = __double2hiint(u[j].l), h = __double2hiint(u[j].h);
                high = max(high, max(l, h));
                low = min(low, min(l, h));
            }
            high = __reduce_max_sync(0xffffffffu, high);
            low = __reduce_min_sync(0xffffffffu, low);
            if (lane == 0) {
                sm.high[wy] = high;
                sm.low[wy] = low;
            }
            __syncthreads();
#pragma unroll
            for (int w = 0; w < WY; ++w) {
                high = max(high, sm.high[w]);
                low = min(low, sm.low[w]);
            }
            FixedCell fixed;
            // (with one row a thread, which latency bounds, the ratio formed here is 2-5%
            // quicker than the kernel's parameter: 1770 x 30 3.42 / 3.58 ms; otherwise 1-5%
            // slower: 768² 576 / 623 us)
            if (fixed.f.fits(R == 1 ? heat_ratio(op.r) : op.R, high, low)) {
                L2 v[R], none[1];
#pragma unroll
                for (int j = 0; j < R; ++j) v[j] = two(fixed.f.from(u[j].l), fixed.f.from(u[j].h));
                march(fixed, v, none, rows, r0, lane, wy, steps,
                      reinterpret_cast<L2 (*)[WY][2][32]>(sm.row));
                done = __syncthreads_or(fixed.f.failed()) == 0;
                if (done) {
#pragma unroll
                    for (int j = 0; j < R; ++j) u[j] = two(fixed.f.to(v[j].l), fixed.f.to(v[j].h));
                } else {
                    read();
                }
            }
        }
        if (!done) march(cell, u, comp, rows, r0, lane, wy, steps, sm.row);
        const bool one = c >= ring_x && c < ring_x + m.w;
        const bool both = c + 1 >= ring_x && c + 1 < ring_x + m.w;
        const int first = ring - r0, end = ring + m.h - r0;
        if (pairs) {
            if (one)
                each_row(m, gx, gy, [&](int j, size_t at) {
                    if (j >= first && j < end) {
                        Two *p = reinterpret_cast<Two *>(dst + at);
                        *p = Two{Cell::st(u[j].lo()), Cell::st(u[j].hi())};
                        if (Cell::kComp)
                            *reinterpret_cast<Two *>(dst + plane + at) =
                                Two{Cell::st(comp[j].lo()), Cell::st(comp[j].hi())};
                    }
                });
        } else {
            each_row(m, gx, gy, [&](int j, size_t at) {
                if (j < first || j >= end) return;
                S *p = dst + at;
                if (one) p[0] = Cell::st(u[j].lo());
                if (both) p[east] = Cell::st(u[j].hi());
                if (Cell::kComp && one) p[plane] = Cell::st(comp[j].lo());
                if (Cell::kComp && both) p[(ptrdiff_t)plane + east] = Cell::st(comp[j].hi());
            });
        }
    }
};

// FP64 heat by the FP64 operations, a step a phase, for fields that the integer
// units cannot take: with no ring of K the pipe, which bounds it, does 1.03 times the
// work of the points kept (HeatMarch 1.31 and more), as much as the swept kernels. A
// warp walks down 64 columns, two a lane, of which the outermost only supply
// neighbours, with the rows above and at the current one in registers; its walks share
// nothing. 4096², mixed-sign noise, 100 steps, ms: 13.4 (swept 13.5, HeatMarch 17.5);
// 2048²: 3.44 (3.89, 4.46); 1024 x 512: 0.66 (0.60, 0.75).
struct HeatWalkOp : HeatOp {
    __host__ __device__ explicit HeatWalkOp(const double *c) : HeatOp(c) {}
};
template <int HR_, int WY_, int MINB_>
struct HeatWalk {
    typedef double S;
    static constexpr int HR = HR_, WY = WY_, K = 1;
    static constexpr int kThreads = 32 * WY, kMinBlocks = MINB_;
    static constexpr bool kInPlace = false;
    static constexpr int kTileCols = 62, kTileRows = HR * WY;
    struct Smem {};
    // `steps` is 1, or 0 for a copy (a phase that only moves the state to the other buffer).
    __device__ static __forceinline__ void run(const HeatOp &op, const MarchTile &m, const S *src,
                                               S *dst, int, int steps, int, Smem &) {
        const HeatCell<HeatOp> cell(op);
        const int wy = threadIdx.x >> 5, c = 2 * (int)(threadIdx.x & 31) - 1;
        const int y = wy * m.h / WY, n = (wy + 1) * m.h / WY - y;
        if (n == 0) return;
        const int gx = wrap_index(m.x0 + c, m.g.nx), ny = m.g.ny;
        const ptrdiff_t east = gx + 1 == m.g.nx ? 1 - m.g.nx : 1;
        const bool one = c >= 0 && c < m.w, both = c + 1 < m.w;
        const size_t nx = m.g.nx, plane = nx * ny;
        int gy = m.y0 + y == 0 ? ny - 1 : m.y0 + y - 1;      // the row that is read next
        const S *p = src + (size_t)gy * nx + gx;
        const auto fetch = [&] {
            const D2 v = two(p[0], p[east]);
            const bool last = ++gy == ny;
            gy = last ? 0 : gy;
            p += last ? nx - plane : nx;
            return v;
        };
        S *o = dst + (size_t)(m.y0 + y) * nx + gx;
        const D2 up = fetch();
        if (steps == 0) {
            for (int i = 0; i < n; ++i, o += nx) {
                const D2 u = fetch();
                if (one) o[0] = u.l;
                if (both) o[east] = u.h;
            }
            return;
        }
        D2 at = fetch(), ahead = fetch(), none;
        D2 pp = cell.pair(east_of(up), at);
        for (int i = 0; i < n; ++i, o += nx) {
            const D2 dn = ahead;
            if (i + 1 < n) ahead = fetch();
            const D2 pe = cell.pair(east_of(at), dn);
            D2 u = at;
            cell.next(u, none, pe, moved_right(pp));
            if (one) o[0] = u.l;
            if (both) o[east] = u.h;
            pp = pe;
            at = dn;
        }
    }
};

// ------------------------------------------------------------------- Euler
// Packed arithmetic on two columns, in the update's arithmetic type.
__device__ __forceinline__ D2 add2(D2 a, D2 b) { return two(__dadd_rn(a.l, b.l), __dadd_rn(a.h, b.h)); }
__device__ __forceinline__ D2 sub2(D2 a, D2 b) { return two(__dsub_rn(a.l, b.l), __dsub_rn(a.h, b.h)); }
__device__ __forceinline__ D2 mul2(D2 a, D2 b) { return two(__dmul_rn(a.l, b.l), __dmul_rn(a.h, b.h)); }
__device__ __forceinline__ D2 fma2(D2 a, D2 b, D2 c) {
    return two(__fma_rn(a.l, b.l, c.l), __fma_rn(a.h, b.h, c.h));
}
// 1 / a, correctly rounded (the bits of the division)
__device__ __forceinline__ D2 rcp2(D2 a) { return two(__drcp_rn(a.l), __drcp_rn(a.h)); }
__device__ __forceinline__ F2 rcp2(F2 a) { return two(__frcp_rn(a.lo()), __frcp_rn(a.hi())); }
template <int SEG, class V2>
__device__ __forceinline__ V2 west_of(V2 v) { return moved_right<SEG>(v); }

// One row of the stage's stencil values in a thread: W, and F1-F3, G1-G3 of the
// two points (F0 = m and G0 = q are W's).
template <class V2>
struct EulerRow {
    V2 w[4], F[3], G[3];
};

// One stage of the midpoint scheme per phase, in place: stage 0 reads U with its
// neighbours and writes U*, stage 1 reads U* with its neighbours and writes U
// (and C) at the point alone. SEG lanes walk down 2 SEG columns, two a thread,
// with the rows above, at and below the current one in registers: every point's
// primitives and fluxes are formed once and serve its four neighbours, the east
// and west ones by shuffle. The outermost columns only supply neighbours. The
// walks of a block take HR rows each and share nothing. Binary64 is bound by the
// FP64 pipe (0.93 of its rate), binary32 by DRAM (28 planes a step, 4.7 TB/s) and,
// with bfloat16, by the loads' latency. 2048² against the swept kernels: binary64 50
// steps 66.4 -> 56.7 ms, binary32 200 steps 31.3 -> 19.5, bfloat16 30.4 -> 14.1.
template <class Op, int SEG_, int HR_, int WY_, int MINB_>
struct EulerMarch {
    typedef typename Op::S S;
    static constexpr bool kWide = std::is_same<Op, EulerOp>::value;   // binary64, not compensated
    typedef typename std::conditional<kWide, D2, F2>::type V2;
    typedef typename std::conditional<kWide, double, float>::type V;
    static constexpr int SEG = SEG_, HR = HR_, WY = WY_, K = 1;
    static constexpr int kThreads = 32 * WY, kMinBlocks = MINB_;
    static constexpr int kWalks = kThreads / SEG;
    static constexpr bool kInPlace = true;
    static constexpr int kRing = kWide ? 1 : 2;    // (aligned pairs for the narrow types)
    static constexpr int kTileCols = 2 * SEG - 2 * kRing, kTileRows = HR * kWalks;
    struct Smem {};
    struct alignas(2 * sizeof(S)) Two {
        S a, b;
    };
    __device__ static __forceinline__ V ld(S v) {
        if constexpr (kWide) return v; else return Store<S>::ld(v);
    }
    __device__ static __forceinline__ V2 stored(V2 v) {
        if constexpr (kWide) return v; else return stored2(v, (const S *)nullptr);
    }
    __device__ static __forceinline__ S st(V v) {
        if constexpr (kWide) return v; else return Store<S>::st(v);
    }

    // The thread's two columns of a plane: aligned pairs (PAIRS), or the two
    // elements, the second `east` of the first.
    template <bool PAIRS>
    struct Columns {
        ptrdiff_t east;
        bool one, both;     // this thread stores its first, its second column
        __device__ __forceinline__ V2 get(const S *p) const {
            if constexpr (PAIRS) {
                const Two t = *reinterpret_cast<const Two *>(p);
                return two(ld(t.a), ld(t.b));
            }
            return two(ld(p[0]), ld(p[east]));
        }
        __device__ __forceinline__ void put(S *p, V2 v) const {
            if constexpr (PAIRS) {
                if (one) *reinterpret_cast<Two *>(p) = Two{st(v.lo()), st(v.hi())};
            } else {
                if (one) p[0] = st(v.lo());
                if (both) p[east] = st(v.hi());
            }
        }
    };

    __device__ static __forceinline__ V2 all(V c) { return two(c, c); }

    __device__ static __forceinline__ void fluxes(const Op &op, EulerRow<V2> &r) {
        const V2 m = r.w[1], q = r.w[2];
        const V2 iv = rcp2(r.w[0]);
        const V2 u = mul2(m, iv), v = mul2(q, iv);
        const V2 ke = mul2(all(V(0.5)), fma2(m, u, mul2(q, v)));
        const V2 pr = mul2(all(op.gm1), sub2(r.w[3], ke));
        const V2 Ep = add2(r.w[3], pr);
        r.F[0] = fma2(m, u, pr);
        r.F[1] = mul2(q, u);
        r.F[2] = mul2(Ep, u);
        r.G[0] = mul2(m, v);
        r.G[1] = fma2(q, v, pr);
        r.G[2] = mul2(Ep, v);
    }

    // L of the conserved variable c at row `at` between rows `up` and `dn`.
    template <int c>
    __device__ static __forceinline__ V2 rate(const Op &op, const EulerRow<V2> &up,
                                              const EulerRow<V2> &at, const EulerRow<V2> &dn) {
        const V2 wE = east_of<SEG>(at.w[c]), wW = west_of<SEG>(at.w[c]);
        const V2 f = c == 0 ? at.w[1] : at.F[c > 0 ? c - 1 : 0];
        const V2 dF = sub2(east_of<SEG>(f), west_of<SEG>(f));
        const V2 dG = c == 0 ? sub2(dn.w[2], up.w[2])
                             : sub2(dn.G[c > 0 ? c - 1 : 0], up.G[c > 0 ? c - 1 : 0]);
        const V2 lx = fma2(all(V(-2)), at.w[c], add2(wE, wW));
        const V2 ly = fma2(all(V(-2)), at.w[c], add2(dn.w[c], up.w[c]));
        const V2 diss = fma2(all(op.kax), lx, mul2(all(op.kay), ly));
        const V2 flux = fma2(all(op.cx), dF, mul2(all(op.cy), dG));
        return sub2(diss, flux);
    }

    // Stage `ST` of the rows [y, y + n) of the warp's columns.
    template <int ST, bool PAIRS>
    __device__ static __forceinline__ void walk(const Op &op, const MarchTile &m, S *state, int gx,
                                                int c, int y, int n) {
        const Columns<PAIRS> col{gx + 1 == m.g.nx ? 1 - m.g.nx : 1, c >= 0 && c < m.w,
                                 c + 1 >= 0 && c + 1 < m.w};
        const size_t nx = m.g.nx, plane = nx * m.g.ny;
        const int ny = m.g.ny;
        int gy = y == 0 ? ny - 1 : y - 1;            // the row that is read next
        const S *p = state + (ST == 0 ? 0 : 4 * plane) + (size_t)gy * nx + gx;
        V2 ahead[4];                                 // W of that row, read one row early
        const auto fetch = [&] {
#pragma unroll
            for (int c = 0; c < 4; ++c) ahead[c] = col.get(p + c * plane);
            const bool last = ++gy == ny;
            gy = last ? 0 : gy;
            p += last ? nx - plane : nx;
        };
        const auto next_row = [&](EulerRow<V2> &r) {
#pragma unroll
            for (int c = 0; c < 4; ++c) r.w[c] = ahead[c];
        };
        S *o = state + (size_t)y * nx + gx;          // the centre row's U
        EulerRow<V2> A, B, C;
        fetch();
        next_row(A);
        fetch();
        fluxes(op, A);
        next_row(B);
        fetch();
        fluxes(op, B);
        const auto step = [&](const EulerRow<V2> &up, const EulerRow<V2> &at, EulerRow<V2> &dn,
                              bool more) {
            V2 U[4], Cc[4];
            if constexpr (ST == 1) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    U[c] = col.get(o + c * plane);
                    if constexpr (!kWide) Cc[c] = col.get(o + (8 + c) * plane);
                }
            }
            next_row(dn);
            if (more) fetch();
            fluxes(op, dn);
            const auto finish = [&](int c, V2 L) {
                if constexpr (ST == 0) {
                    col.put(o + (4 + c) * plane, stored(fma2(all(op.tau0), L, at.w[c])));
                } else if constexpr (kWide) {
                    col.put(o + c * plane, fma2(all(op.tau1), L, U[c]));
                } else {
                    const V2 yy = sub2(mul2(all(op.tau1), L), Cc[c]);
                    const V2 un = stored(add2(U[c], yy));
                    col.put(o + c * plane, un);
                    col.put(o + (8 + c) * plane, sub2(sub2(un, U[c]), yy));
                }
            };
            finish(0, rate<0>(op, up, at, dn));
            finish(1, rate<1>(op, up, at, dn));
            finish(2, rate<2>(op, up, at, dn));
            finish(3, rate<3>(op, up, at, dn));
            o += nx;
        };
        // (the row after the last one is read, but not the one after that)
        for (int i = 0; i < n; i += 3) {
            step(A, B, C, i + 1 < n);
            if (i + 1 >= n) break;
            step(B, C, A, i + 2 < n);
            if (i + 2 >= n) break;
            step(C, A, B, i + 3 < n);
        }
    }

    __device__ static __forceinline__ void run(const Op &op, const MarchTile &m, const S *,
                                               S *state, int, int, int phase, Smem &) {
        const int walk_at = threadIdx.x / SEG;
        const int c = 2 * (int)(threadIdx.x % SEG) - kRing;   // first column, from the tile's
        const int nx = m.g.nx;
        const int gx = wrap_index(m.x0 + c, nx);
        const bool pairs = !kWide && (nx & 1) == 0 && ((size_t)state & (2 * sizeof(S) - 1)) == 0;
        // the tile's rows, shared evenly
        const int y = walk_at * m.h / kWalks, n = (walk_at + 1) * m.h / kWalks - y;
        if (n == 0) return;
        const auto stage = [&](auto st) {
            constexpr int ST = decltype(st)::value;
            if (!kWide && pairs)
                walk<ST, !kWide>(op, m, state, gx, c, m.y0 + y, n);
            else
                walk<ST, false>(op, m, state, gx, c, m.y0 + y, n);
        };
        if ((phase & 1) == 0)
            stage(std::integral_constant<int, 0>());
        else
            stage(std::integral_constant<int, 1>());
    }
};

// The shapes an update's tiles come in, largest first.
//
// Heat: rows a thread, warps, blocks an SM and steps a phase. Rows in registers and the region's
// size save redundant work, steps a phase save passes over memory and waits,
// and both cost warps an SM, which hide the shuffles' and the integer chains'
// latency. Measured on the GB300 (ms for the whole advance):
//   binary64, 4096², 500 steps: (8, 8, 3, 4) 36.4, (8, 4, 5, 4) 40.1,
//     (4, 8, 4, 4) 40.4, (8, 8, 2, 4) 45.4, (8, 16, 1, 4) 52.6
//   binary64, 768², 403 steps: (2, 8, 4, 3) 2.0, (4, 8, 4, 4) 2.2, (8, 4, 5, 4) 2.9
//   binary64, 64², 512 steps: (1, 8, 4, 2) 0.68, (2, 8, 4, 3) 0.72, (1, 16, 2, 3) 0.73
//   binary32, 2048², 2000 steps (all additions packed): (16, 4, 4, 8) 8.2, (8, 8, 4, 6) 8.9,
//     (16, 8, 2, 12) 8.7; 1,024 grids of {32..512}²: 25.7, 27.6, 28.0
//
// FP64 heat's walks: rows a walk, warps, blocks an SM; ms for 100 steps of mixed-sign noise:
//   4096² 13.3, 13.6, 14.3, 18.5; 2048² 3.72, 3.44, 3.53, 4.35; 1280² 2.31, 1.77, 1.40,
//   1.64; 1024² 1.80, 1.50, 1.08, 1.10; 768² 1.37, 1.14, 0.95, 0.68
//
// Euler: lanes and rows a walk, warps, blocks an SM. More rows form fewer fluxes
// twice; more blocks hide the loads' latency, as far as the three rows of values
// stay in registers (binary64, at the FP64 pipe's rate, needs few); fewer lanes
// waste less on narrow tiles and spread a small grid over more SMs.
//   binary64, 32 stages, us, for the four shapes: 1024² 7567, 5049, 5779, 7536;
//     512² 2720, 2669, 1481, 1924; 128 x 128 2714, 1416, 457, 336; 2048², 50 steps:
//     56.7, 61.0 ms
//   binary32, 2048², 200 steps, ms: (32, 32, 4, 4) 19.5, (32, 16, 4, 5) 19.5,
//     (32, 16, 4, 6) 21.0, (32, 8, 4, 4) 21.4, (32, 32, 4, 3) 25.0; bfloat16: 14.2,
//     16.0, 16.4, 16.8, 21.7; 256 grids binary32, 50 steps: 23.8, 24.7, 25.8, 27.9,
//     30.1; 64 stages, us, for the five shapes: 1024² 1321, 614, 795, 1160, 1938;
//     512² 1190, 466, 385, 307, 491; 128 x 128 1169, 411, 276, 216, 187
template <class Op>
struct MarchShapes;
template <>
struct MarchShapes<HeatOp> {
    static constexpr int kCount = 4;
    template <int I>
    using Body = std::conditional_t<
        I == 0, HeatMarch<HeatOp, 8, 8, 3, 4>,
        std::conditional_t<I == 1, HeatMarch<HeatOp, 4, 8, 4, 4>,
                           std::conditional_t<I == 2, HeatMarch<HeatOp, 2, 8, 4, 3>,
                                              HeatMarch<HeatOp, 1, 8, 4, 2>>>>;
};
template <>
struct MarchShapes<HeatWalkOp> {
    static constexpr int kCount = 4;
    template <int I>
    using Body = std::conditional_t<
        I == 0, HeatWalk<16, 4, 8>,
        std::conditional_t<I == 1, HeatWalk<8, 4, 8>,
                           std::conditional_t<I == 2, HeatWalk<4, 4, 8>, HeatWalk<2, 4, 8>>>>;
};
template <>
struct MarchShapes<EulerOp> {
    static constexpr int kCount = 4;
    template <int I>
    using Body = std::conditional_t<
        I == 0, EulerMarch<EulerOp, 32, 16, 4, 3>,
        std::conditional_t<I == 1, EulerMarch<EulerOp, 16, 8, 4, 3>,
                           std::conditional_t<I == 2, EulerMarch<EulerOp, 16, 2, 4, 3>,
                                              EulerMarch<EulerOp, 8, 1, 2, 6>>>>;
};
template <class SS>
struct MarchShapes<EulerKahanOp<SS>> {
    typedef EulerKahanOp<SS> Op;
    static constexpr int kCount = 5;
    template <int I>
    using Body = std::conditional_t<
        I == 0, EulerMarch<Op, 32, 32, 4, 4>,
        std::conditional_t<
            I == 1, EulerMarch<Op, 32, 8, 4, 4>,
            std::conditional_t<I == 2, EulerMarch<Op, 32, 4, 4, 4>,
                               std::conditional_t<I == 3, EulerMarch<Op, 32, 2, 4, 4>,
                                                  EulerMarch<Op, 32, 1, 4, 4>>>>>;
};
template <class SS>
struct MarchShapes<HeatKahanOp<SS>> {
    typedef HeatKahanOp<SS> Op;
    static constexpr int kCount = 3;
    template <int I>
    using Body = std::conditional_t<
        I == 0, HeatMarch<Op, 16, 4, 4, 8>,
        std::conditional_t<I == 1, HeatMarch<Op, 8, 4, 4, 6>, HeatMarch<Op, 2, 8, 4, 4>>>;
};

// Tiles of many grids: the table lists each grid's tiles consecutively.
struct ManyMarch {
    const GridDesc *grids;
    const int2 *tiles;           // (grid, tile within the grid)
    __device__ __forceinline__ MarchTile operator()(int t) const {
        const int2 e = tiles[t];
        const GridDesc *gd = grids + e.x;
        MarchTile m;
        m.g = gd->m;
        m.base = t - e.y;
        m.soff = gd->state_off;
        m.c = gd->c;
        m.place(e.y);
        return m;
    }
};

// ----------------------------------------------------------- host side
// Calls f with the body type of shape i.
template <class Op, int I = 0, class F>
inline cudaError_t with_march_shape(int i, F &&f) {
    if constexpr (I < MarchShapes<Op>::kCount) {
        if (i == I) return f((typename MarchShapes<Op>::template Body<I> *)nullptr);
        return with_march_shape<Op, I + 1>(i, f);
    } else {
        return cudaErrorInvalidValue;
    }
}

// How one grid is cut for a shape.
template <class Op>
inline MarchGrid march_cut(int shape, int nx, int ny) {
    MarchGrid g{nx, ny, 0, 0};
    with_march_shape<Op>(shape, [&](auto *body) {
        typedef typename std::remove_pointer<decltype(body)>::type B;
        // (even first columns: a tile may be one column wider than its share)
        g.bx = nx <= B::kTileCols ? 1 : (nx + B::kTileCols - 2) / (B::kTileCols - 1);
        g.by = (ny + B::kTileRows - 1) / B::kTileRows;
        return cudaSuccess;
    });
    return g;
}

template <class Op>
inline int march_steps(int shape) {
    int k = 1;
    with_march_shape<Op>(shape, [&](auto *body) {
        k = std::remove_pointer<decltype(body)>::type::K;
        return cudaSuccess;
    });
    return k;
}

// All grids' tiles in a shape.
template <class Op>
inline long long march_tiles(int shape, const int *nx, const int *ny, int count) {
    long long tiles = 0;
    for (int i = 0; i < count; ++i) {
        const MarchGrid g = march_cut<Op>(shape, nx[i], ny[i]);
        tiles += (long long)g.bx * g.by;
    }
    return tiles;
}

// Binary64 Euler: the µs of a step (two stages). A step of one tile alone takes
// `alone`; with more than about 76 tiles blocks share an SM's FP64 pipe, up to 2.7
// times that, and many tiles take `each`, where a walk of a grid of few rows is
// shorter (a row more forms fluxes at either end). Measured on the GB300, tiles: µs -
//   shape 0: 20: 170, 85: 255, 136: 319, 475: 523, 1088: 1142
//   shape 1: 72: 89, 96: 142, 170: 200, 288: 249, 576: 323, 2272: 1218
//   shape 2: 60: 28.8, 96: 45, 168: 61, 336: 75, 576: 92, 1152: 185, 2304: 365
//   shape 3: 96: 19.0, 260: 28, 512: 42, 1000: 49, 1440: 68, 2560: 120
inline double euler_march_cost(int shape, const int *nx, const int *ny, int count) {
    double tiles = 0, full = 0;
    with_march_shape<EulerOp>(shape, [&](auto *body) {
        typedef typename std::remove_pointer<decltype(body)>::type B;
        for (int i = 0; i < count; ++i) {
            const MarchGrid g = march_cut<EulerOp>(shape, nx[i], ny[i]);
            const double rows = (double)ny[i] / g.by / B::kWalks;
            tiles += (double)g.bx * g.by;
            full += (double)g.bx * g.by * ((rows < 1 ? 1 : rows) + 2) / (B::HR + 2);
        }
        return cudaSuccess;
    });
    static const double alone[] = {169.6, 88.6, 28.5, 17.4}, each[] = {1.05, 0.537, 0.1585, 0.047},
                        shared[] = {1.42, 1.42, 1.42, 1}, spread[] = {150, 150, 150, 306};
    double crowd = tiles <= 76 ? 1.0 : shared[shape] + (tiles - 76) / spread[shape];
    if (crowd > 2.7) crowd = 2.7;
    const double one = alone[shape] * crowd, all = each[shape] * full;
    return one > all ? one : all;
}
// The same of the swept kernels, whose launches are per tile side n (0: the naive
// ones): n = 8: 64 tiles 18.4, 400: 33, 1024: 81, 4096: 282; n = 16: 144: 22, 256: 36,
// 576: 71, 1024: 119; n = 32: 64: 47, 144: 53, 256: 99, 400: 149, 576: 196, 1024: 342;
// n = 40: 64: 67, 144: 82, 256: 164, 400: 245, 576: 327 (whole waves of the SMs, as the
// tiles grow). One persistent launch takes more where the tiles about fill the SMs:
// n = 16: 144: 29, n = 32: 64: 57, 144: 82, 256: 94, 576: 191.
inline double euler_swept_cost(int n, double tiles, bool persistent) {
    if (n == 0) return 18.7 + 16.3 / 152 * tiles;
    double t = 17.3 + 0.00442 * std::pow((double)n, 2.6);
    const double wave = n >= 20 ? 0.6 + 0.01 * n : 0.38 + 0.0225 * n;   // of each after the first
    if (persistent && tiles > 200)                // (13 µs a wave at n = 8, 17.5, 47.5 at n = 32)
        return (t - 5.3) * (n >= 20 ? std::ceil(tiles / 152) - 0.15 : tiles / 152 + 0.2);
    const double more = (double)(((long long)tiles - 1) / 152);
    if (n >= 20)
        t *= tiles <= 100 ? 0.88 : 1.0 + wave * (more == 1 ? 0.93 : more);
    else if (more > 0)
        t *= more == 1 ? 1.16 + 0.028 * n : more == 2 ? 1.25 + 0.067 * n : 1.0 + wave * more;
    if (!persistent || tiles <= 48) return t;
    if (n >= 36) return 1.05 * t;
    return t * (tiles > 100 ? 1.0 + (n < 25 ? 0.02 * n : 0.5) : n < 20 ? 1.06 : 1.25);
}
inline double euler_swept_cost(const int *nx, const int *ny, const int *tile, int count,
                               bool persistent) {
    double t = 0;
    for (int i = 0; i < count; ++i) {
        const int n = tile[i];
        bool seen = false;
        for (int k = 0; k < i && !seen; ++k) seen = tile[k] == n;
        if (seen) continue;
        double tiles = 0;
        for (int k = i; k < count; ++k)
            if (tile[k] == n)
                tiles += n ? (double)(nx[k] / n) * (ny[k] / n)
                           : (double)((nx[k] + 31) / 32) * ((ny[k] + 7) / 8);
        t += euler_swept_cost(n, tiles, persistent);
    }
    return t;
}

// The shape for these grids (all together) with the callers' tile sides, -1 where
// the swept kernels (as a persistent launch or not) do better; without tile sides, a
// shape in any case.
//  - The largest shape that gives the GPU's 152 SMs three tiles each, else the
//    smallest one. Binary64 heat, whose redundant points may cost FP64 time, stays
//    with the swept kernels when its tiles fill less than 0.78 of their 64 columns
//    and the grid is too large to be bound by latency (fields with a zero crossing in
//    every tile, 96 steps, us, swept / marching: 64 x 2048 292 / 437, 192 x 384 241 /
//    281, but 48 x 512 221 / 181, 256 x 256 241 / 232, 1024 x 1024 1469 / 706), and so
//    it does where r keeps it off the integer units altogether (r = 1/4, 100 steps, us:
//    256² 306 / 290, 512² 413 / 492, 1024² 1122 / 1370, 4096² 13505 / 17470).
//  - Binary64 Euler, bound by the FP64 pipe in either form: the least of the costs
//    above (us a step, swept at the tile given / marching: 64 x 2048, 32, 54 / 61;
//    384 x 384, 32, 54 / 68; 48 x 512, 16, 22 / 27; 128 x 512, 32, 47 / 43; 256 grids
//    of 32..96 460 / 385, by the largest shape that fills the SMs 450).
template <class Op>
inline int march_shape(const int *nx, const int *ny, const int *tile, int count, bool persistent,
                       const double *c) {
    if constexpr (std::is_same<Op, EulerOp>::value) {
        int best = 0;
        double least = 0;
        for (int s = 0; s < MarchShapes<Op>::kCount; ++s) {
            const double t = euler_march_cost(s, nx, ny, count);
            if (s == 0 || t < least) {
                least = t;
                best = s;
            }
        }
        return tile && euler_swept_cost(nx, ny, tile, count, persistent) < least ? -1 : best;
    }
    int shape = 0;
    while (march_tiles<Op>(shape, nx, ny, count) < 3 * 152 && shape + 1 < MarchShapes<Op>::kCount)
        ++shape;
    if (tile && std::is_same<Op, HeatOp>::value) {
        double points = 0, columns = 0;
        for (int i = 0; i < count; ++i) {
            points += (double)nx[i] * ny[i];
            columns += 64.0 * march_cut<Op>(shape, nx[i], ny[i]).bx * ny[i];
        }
        if (points > 28000 && (points < 0.78 * columns || heat_ratio(c[0]) == 0)) return -1;
    }
    return shape;
}

// The shape of FP64 heat's walks: the most rows that still give every resident block a tile.
inline int heat_walk_shape(int nx, int ny) {
    int shape = 0;
    while (march_tiles<HeatWalkOp>(shape, &nx, &ny, 1) < 8 * 152 &&
           shape + 1 < MarchShapes<HeatWalkOp>::kCount)
        ++shape;
    return shape;
}

// ---------------------------------------------- the naive path's walks (Euler)
// What a step (two launches) of the naive path takes, in µs: `more` for each wave of
// blocks that run at once beside `base`. In binary64 a block has an SM for itself,
// as the FP64 pipe is the bound, and the waves are whole; otherwise the resident
// blocks of an SM end at different times, and the second wave alone costs an extra.
struct WaveCost {
    double base, more;
    int wave;
    double least;               // however few the blocks
    bool whole;
    double operator()(long long blocks) const {
        double w = (double)((blocks + wave - 1) / wave);
        if (!whole && w > 1) {
            w = (double)blocks / wave + 0.1;
            if (w < 1.65) w = 1.65;
        }
        const double t = base + more * w;
        return t > least ? t : least;
    }
};
// By shape; last: a thread a point, in blocks of 32 x 8 points, which forms
// its four neighbours' fluxes, too, but has the shorter chain. Measured on the
// GB300, us a step in a graph, walks by shape 0, 1, ... / a thread a point:
//   binary64: 64 x 64 166, 88, 28.0, 17.2 / 18.6; 64 x 512 167, 88, 28.2, 25.3 / 18.8;
//     256 x 256 167, 88, 28.5, 40.2 / 34.6; 384 x 384 167, 88, 75, 74.7 / 67;
//     1024 x 65 -, -, 51, 40 / 35; 512 x 512 167, 88, 99, 131 / 116;
//     1024 x 1024 320, 332, 383, 483 / 441; 2048 x 2048 1260, 1218, 1420, 1885 / 1748
//   binary32: 400 x 300 36, 13, 8.9, 7.3, 8.7 / 6.1; 128 x 2048 37, 13.6, 10.0, 12.4, 14.5
//     / 9.8; 272 x 1056 35, 13.8, 10.0, 11.9, 13.9 / 10.8; 512 x 512 38, 13.2, 9.8, 8.1,
//     11.2 / 9.6; 1024 x 1024 39, 19.6, 22.5, 26.6, 38.6 / 39.1; 2048 x 2048 98, 102, 112,
//     120, 167 / 164; bfloat16: 272 x 1056 44, 15.9, 11.1, 13.0, 14.5 / 11.0; 1024 x 1024
//     47, 20.2, 23.2, 28.1, 39.2 / 31.3; 2048 x 2048 67, 77, 88, 106, 152 / 142
template <class Op>
inline const WaveCost *naive_costs() {
    return nullptr;
}
template <>
inline const WaveCost *naive_costs<EulerOp>() {
    static const WaveCost c[] = {{6, 157, 152, 0, true},
                                 {8, 79.5, 152, 0, true},
                                 {4.5, 23.7, 152, 0, true},
                                 {2.5, 7.5, 152, 17.2, true},
                                 {2.4, 16.3, 152, 0, true}};
    return c;
}
template <>
inline const WaveCost *naive_costs<EulerKahanOp<float>>() {
    static const WaveCost c[] = {{-15, 55, 608, 0, false},   {-4, 20, 608, 0, false},
                                 {-2.1, 12.5, 608, 0, false}, {2, 6.2, 608, 0, false},
                                 {1.8, 4.6, 608, 0, false},   {1, 5, 608, 0, false}};
    return c;
}
template <>
inline const WaveCost *naive_costs<EulerKahanOp<__nv_bfloat16>>() {
    static const WaveCost c[] = {{-12, 57, 608, 0, false},   {-4, 20, 608, 0, false},
                                 {-1.0, 12.5, 608, 0, false}, {2.4, 6.3, 608, 0, false},
                                 {2.1, 4.7, 608, 0, false},   {1, 5, 608, 0, false}};
    return c;
}

template <class Op>
inline int naive_shape(int nx, int ny, const double *c) {
    // FP64 heat: its walks where no warp could take the integer units (r) and the pipe
    // is the bound (us a step, naive_heat_kernel / walks: 4096² 147 / 136)
    if constexpr (std::is_same<Op, HeatOp>::value)
        return heat_ratio(c[0]) == 0 && (double)nx * ny >= 5e5 ? heat_walk_shape(nx, ny) : -1;
    const WaveCost *cost = naive_costs<Op>();
    if (!cost) return -1;
    int best = -1;
    double least = cost[MarchShapes<Op>::kCount](((nx + 31LL) / 32) * ((ny + 7) / 8));
    for (int s = 0; s < MarchShapes<Op>::kCount; ++s) {
        const MarchGrid g = march_cut<Op>(s, nx, ny);
        const double t = cost[s]((long long)g.bx * g.by);
        if (t < least) {
            least = t;
            best = s;
        }
    }
    return best;
}

// Whether an advance of one grid by `substeps` sub-steps is quicker as so many naive
// launches than as one launch in the marching form, whose ring and first phase it
// then has alone (a batch's naive launches take a thread a point: it marches). Measured on the GB300, us by the stream, naive launches / marching:
//   heat binary64: 256 x 256, 2 steps 10.9 / 12.9, 4: 19.1 / 19.0; 768 x 768, 2: 22 / 27,
//     4: 43 / 40 (with the survey 47, mixed signs 45 / 46); 2048 x 2048, 2: 46 / 74, 6: 140 / 157 (mixed signs 251 / 290), 16: 370 /
//     371; 4096 x 4096, 6: 510 / 514 (mixed signs 836 / 1090); in a graph (uniform noise) 64 x
//     384, 7: 59 / 65 with the state's copies
//   heat binary32: 256 x 256, 1 step 5.4 / 10.3, 2: 9.8 / 9.9, 3: 14.4 / 9.8; 2048 x 2048, 1:
//     15.9 / 33, 2: 28 / 33, 3: 41 / 33
//   Euler binary32: 256 x 256, 1 step 11.9 / 15.8, 2: 20.3 / 22.2, 3: 28.6 / 28.8; in a
//     graph every step of what fills no half cycle: 512 x 512 8.1 / 9.9, 128 x 2048 9.8 /
//     12.5, 1024 x 1024 19.6 / 20.8, 2048 x 2048 98.2 / 96.2
//   Euler binary64 (by both forms' costs; never more than the caller's half cycle, which
//     the swept form would not fill either): 80 x 320, 3 steps 76 / 104; 384 x 192, 3: 126 /
//     147; 64 x 64, 1: 24 / 21
template <class Op>
inline bool march_short(int shape, int nx, int ny, int tile, long long substeps, bool graph) {
    if constexpr (std::is_same<Op, HeatOp>::value) {
        const double points = (double)nx * ny;
        if (graph && substeps <= 12 && substeps < tile / 2 && points < 1e6) return true;
        return substeps <= 3 || (substeps <= 5 && points >= 5e5) || (substeps <= 6 && points >= 2e6);
    } else if constexpr (std::is_same<Op, EulerOp>::value) {
        if (substeps >= tile / 2) return false;
        const int s = naive_shape<Op>(nx, ny, nullptr);
        const WaveCost cost = naive_costs<Op>()[s < 0 ? MarchShapes<Op>::kCount : s];
        const double naive = cost(s < 0 ? ((nx + 31LL) / 32) * ((ny + 7) / 8)
                                        : march_tiles<Op>(s, &nx, &ny, 1));
        return 0.5 * (double)substeps * (naive - euler_march_cost(shape, &nx, &ny, 1)) < 6;
    } else if constexpr (Op::NST == 2) {
        return substeps <= 4 || substeps < tile / 2;
    } else {
        return substeps <= 2;
    }
}

// One launch of a run whose counters are set; with `spoil`, the advance's result, that
// becomes NaN where a wait gives up.
template <class B, bool AFTER, class Op, class Loc>
inline cudaError_t march_launch(const Op &op, const Loc &at, const MarchRun<typename Op::S> &run,
                                void *spoil, size_t points, cudaStream_t st) {
    const auto launch = [&](auto *kern, auto... more) {
        int per_sm = 0, dev = 0, nsm = 0;
        const cudaError_t e =
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, B::kThreads, 0);
        if (e != cudaSuccess) return e;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        long long grid = (long long)(per_sm > 0 ? per_sm : 1) * nsm;
        if (grid > 2LL * run.NT) grid = 2LL * run.NT;
        if (grid > (long long)run.NT * run.phases) grid = (long long)run.NT * run.phases;
        if constexpr (AFTER)
            return launch_after(kern, dim3((unsigned)grid), B::kThreads, 0, st, op, at, run, more...);
        kern<<<(int)grid, B::kThreads, 0, st>>>(op, at, run, more...);
        return cudaGetLastError();
    };
    if constexpr (std::is_base_of<HeatOp, Op>::value && std::is_same<Loc, OneMarch>::value)
        if (spoil)
            return launch(&march_or_spoil_kernel<B, Op, Loc, AFTER>, (double *)spoil, points);
    return launch(&march_kernel<B, Op, Loc, AFTER>);
}

// Queues `steps` steps over NT tiles: reads `src`, writes b0, b1, b0, ... phase
// by phase (src may be b1). sched: NT counters and the item counter; without `err`
// (one heat grid) the word before them is the error word and is cleared with them,
// and the result, which `*out` then names beforehand, becomes NaN where a wait gives
// up. `launches` is raised by the launches made, `*out` set to the buffer with the
// result.
template <class Op, class Loc>
inline cudaError_t march_advance(int shape, const Op &op, const Loc &at, int NT, const void *src,
                                 void *b0, void *b1, int *sched, long long steps, int *err,
                                 int first, long long spin_limit, void **out, long long *launches,
                                 cudaStream_t st, size_t points = 0) {
    typedef typename Op::S S;
    return with_march_shape<Op>(shape, [&](auto *body) {
        typedef typename std::remove_pointer<decltype(body)>::type B;
        constexpr int K = B::K;
        if (B::kInPlace) b0 = b1 = const_cast<void *>(src);
        // items of one launch count in an int
        // (an even number of phases: the stages of Euler alternate)
        const long long most = (((1LL << 30) - 1) / NT + 2) & ~1LL;
        int *clear = sched;
        void *const spoil = err ? nullptr : *out;
        if (!err) err = sched++;
        while (steps > 0) {
            const long long left = (steps + K - 1) / K;
            MarchRun<S> run;
            run.src = (const S *)src;
            run.buf[0] = (S *)b0;
            run.buf[1] = (S *)b1;
            run.done = sched;
            run.queue = sched + NT;
            run.err = err;
            run.NT = NT;
            run.phases = (int)(left < most ? left : most);
            run.K = K;
            run.last = run.phases < left ? K : (int)(steps - (left - 1) * K);
            run.first = first;
            run.spin_limit = spin_limit;
            cudaError_t e = cudaMemsetAsync(clear, 0, (sched + NT + 1 - clear) * sizeof(int), st);
            if (e != cudaSuccess) return e;
            clear = sched;
            if ((e = march_launch<B, false>(op, at, run, spoil, points, st)) != cudaSuccess)
                return e;
            *launches += 1;
            steps -= (long long)(run.phases - 1) * K + run.last;
            *out = run.buf[(run.phases - 1) & 1];
            src = *out;
            if (*out == b0) {
                b0 = b1;
                b1 = *out;
            }
        }
        return cudaSuccess;
    });
}

// ----------------------------------------------------- FP64 heat by its field
// Whether large FP64 heat grids march on the integer units or by the walks of the
// FP64 operations depends on the field, which only the device has: a survey of up to
// 304 tiles counts those that the integer units could not take, and leaves the item
// counter of the form that does not run behind its last item; both are launched. A
// tile of which more than 60% are unfit is quicker by the walks (2048², us a step,
// integer / FP64 tiles / walks: 20.6 / 44.6 / 34.7). Measured on the GB300, the survey
// and the launch that finds nothing to do: 5 to 8 us an advance.
constexpr int kEitherSteps = 264;        // steps a survey decides on: whole phase pairs of K = 2, 3, 4

template <class Op>
__global__ void __launch_bounds__(256) heat_survey_kernel(Op op, MarchGrid g, const double *u,
                                                          bool soon, unsigned *count, int *march_queue,
                                                          int march_items, int *walk_queue,
                                                          int walk_items) {
    __shared__ int extreme[4][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const MarchTile m = OneMarch{g}((int)((long long)blockIdx.x * (g.bx * g.by) / gridDim.x));
    // 32 rows of the tile (the last repeated), 8 values a thread
    int high = INT_MIN, low = INT_MAX;
    double sum = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const size_t y = m.y0 + min(4 * warp + j, m.h - 1);
            const double v = u[y * g.nx + m.x0 + min(2 * lane + i, m.w - 1)];
            high = max(high, __double2hiint(v));
            low = min(low, __double2hiint(v));
            sum += v;
        }
    // sums of 8 x 4 points: what some ten steps leave of a field that is only rough
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    const int s = __double2hiint(sum);
    high = __reduce_max_sync(0xffffffffu, high);
    low = __reduce_min_sync(0xffffffffu, low);
    const int shigh = __reduce_max_sync(0xffffffffu, s), slow = __reduce_min_sync(0xffffffffu, s);
    if (lane == 0) {
        extreme[0][warp] = high;
        extreme[1][warp] = low;
        extreme[2][warp] = shigh;
        extreme[3][warp] = slow;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    int e[4] = {extreme[0][0], extreme[1][0], extreme[2][0], extreme[3][0]};
    for (int w = 1; w < 8; ++w) {
        e[0] = max(e[0], extreme[0][w]);
        e[1] = min(e[1], extreme[1][w]);
        e[2] = max(e[2], extreme[2][w]);
        e[3] = min(e[3], extreme[3][w]);
    }
    FixedHeat f;
    const unsigned unfit = !f.fits(op.R, e[0], e[1]) && !(soon && f.fits(op.R, e[2], e[3]));
    // (blocks that have counted in the lower half, unfit tiles in the upper)
    const unsigned before = atomicAdd(count, (unfit << 16) + 1);
    if ((before & 0xffff) + 1 < gridDim.x) return;
    if (5 * ((before >> 16) + unfit) > 3 * gridDim.x)
        *march_queue = march_items;
    else
        *walk_queue = walk_items;
}

// Counters of the two forms, with the survey's and the error word's.
template <class Op>
inline long long march_words(int shape, int nx, int ny) {
    long long words = march_tiles<Op>(shape, &nx, &ny, 1) + 2;
    if constexpr (std::is_same<Op, HeatOp>::value)
        words += march_tiles<HeatWalkOp>(heat_walk_shape(nx, ny), &nx, &ny, 1) + 2;
    return words;
}

// Whether a grid takes either: where the walks are the quicker ones on a field that
// the integer units cannot take (us a step of mixed-sign noise, HeatMarch / walks:
// 640 x 640 6.17 / 6.49, 1024 x 512 7.46 / 6.57, 768 x 768 8.17 / 6.77).
template <class Op>
inline bool march_either(const double *c, int nx, int ny) {
    if constexpr (std::is_same<Op, HeatOp>::value)
        return heat_ratio(c[0]) != 0 && (double)nx * ny >= 5e5 &&
               march_tiles<HeatWalkOp>(heat_walk_shape(nx, ny), &nx, &ny, 1) *
                       (kEitherSteps + 1LL) < (1LL << 30);
    return false;
}

// As march_advance for one grid.
inline cudaError_t heat_either_advance(int shape, const MarchGrid &g, const HeatOp &op,
                                       const HeatWalkOp &walk, const void *src, void *b0, void *b1,
                                       int *sched, long long steps, int *err,
                                       long long spin_limit, void **out, long long *launches,
                                       cudaStream_t st) {
    const int ws = heat_walk_shape(g.nx, g.ny);
    const MarchGrid wg = march_cut<HeatWalkOp>(ws, g.nx, g.ny);
    const int NT = g.bx * g.by, WT = wg.bx * wg.by, K = march_steps<HeatOp>(shape);
    int *clear = sched;
    void *const spoil = err ? nullptr : *out;
    const size_t points = (size_t)g.nx * g.ny;
    if (!err) err = sched++;
    int *const walk_sched = sched + NT + 1, *const count = walk_sched + WT + 1;
    while (steps > 0) {
        const int n = steps < kEitherSteps ? (int)steps : kEitherSteps;
        MarchRun<double> run;
        run.src = (const double *)src;
        run.buf[0] = (double *)b0;
        run.buf[1] = (double *)b1;
        run.err = err;
        run.first = 0;
        run.spin_limit = spin_limit;
        run.done = sched;
        run.queue = sched + NT;
        run.NT = NT;
        run.K = K;
        run.phases = (n + K - 1) / K;
        run.last = n - (run.phases - 1) * K;
        MarchRun<double> walked = run;
        walked.done = walk_sched;
        walked.queue = walk_sched + WT;
        walked.NT = WT;
        walked.K = 1;
        walked.phases = n + ((n ^ run.phases) & 1);     // (both end in the same buffer)
        walked.last = n + 1 - walked.phases;
        cudaError_t e = cudaMemsetAsync(clear, 0, (count + 1 - clear) * sizeof(int), st);
        if (e != cudaSuccess) return e;
        clear = sched;
        heat_survey_kernel<HeatOp><<<NT < 304 ? NT : 304, 256, 0, st>>>(
            op, g, run.src, n >= 8, (unsigned *)count, run.queue, NT * run.phases, walked.queue,
            WT * walked.phases);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        e = with_march_shape<HeatOp>(shape, [&](auto *body) {
            return march_launch<typename std::remove_pointer<decltype(body)>::type, true>(
                op, OneMarch{g}, run, spoil, points, st);
        });
        if (e != cudaSuccess) return e;
        e = with_march_shape<HeatWalkOp>(ws, [&](auto *body) {
            return march_launch<typename std::remove_pointer<decltype(body)>::type, true>(
                walk, OneMarch{wg}, walked, spoil, points, st);
        });
        if (e != cudaSuccess) return e;
        *launches += 3;
        steps -= n;
        src = *out = run.buf[(run.phases - 1) & 1];
    }
    return cudaSuccess;
}

// One phase of one step over NT tiles.
template <class Op, class Loc>
inline cudaError_t march_phase(int shape, const Op &op, const Loc &at, int NT, const void *src,
                               void *dst, int phase, cudaStream_t st) {
    typedef typename Op::S S;
    return with_march_shape<Op>(shape, [&](auto *body) {
        typedef typename std::remove_pointer<decltype(body)>::type B;
        if constexpr (B::K == 1)
            return launch_after(march_phase_kernel<B, Op, Loc>, dim3(NT), B::kThreads, 0, st, op, at,
                                (const S *)src, (S *)dst, phase);
        else
            return cudaErrorInvalidValue;
    });
}

template <class Op>
struct March {
    static MarchGrid naive_cut(int shape, int nx, int ny) {
        if constexpr (std::is_same<Op, HeatOp>::value)
            return march_cut<HeatWalkOp>(shape, nx, ny);
        else
            return march_cut<Op>(shape, nx, ny);
    }
    static cudaError_t phase_one(int shape, const MarchGrid &g, const double *c, const void *src,
                                 void *dst, int phase, cudaStream_t st) {
        if constexpr (std::is_same<Op, HeatOp>::value)      // (by its walks)
            return march_phase(shape, HeatWalkOp(c), OneMarch{g}, g.bx * g.by, src, dst, phase, st);
        else
            return march_phase(shape, Op(c), OneMarch{g}, g.bx * g.by, src, dst, phase, st);
    }
    static cudaError_t phase_many(int shape, const GridDesc *grids, const int2 *tiles, int NT,
                                  const double *c, void *state, int phase, cudaStream_t st) {
        return march_phase(shape, Op(c), ManyMarch{grids, tiles}, NT, state, state, phase, st);
    }
    static cudaError_t one(int shape, const MarchGrid &g, const double *c, const void *src,
                           void *b0, void *b1, int *sched, long long steps, int *err, int first,
                           long long spin_limit, void **out, long long *launches,
                           cudaStream_t st) {
        if constexpr (std::is_same<Op, HeatOp>::value)
            if (first == 0 && march_either<Op>(c, g.nx, g.ny))
                return heat_either_advance(shape, g, Op(c), HeatWalkOp(c), src, b0, b1, sched,
                                           steps, err, spin_limit, out, launches, st);
        return march_advance(shape, Op(c), OneMarch{g}, g.bx * g.by, src, b0, b1, sched, steps,
                             err, first, spin_limit, out, launches, st, (size_t)g.nx * g.ny);
    }
    static cudaError_t many(int shape, const GridDesc *grids, const int2 *tiles, int NT,
                            const double *c, const void *src, void *b0, void *b1, int *sched,
                            long long steps, int *err, void **out, long long *launches,
                            cudaStream_t st) {
        return march_advance(shape, Op(c), ManyMarch{grids, tiles}, NT, src, b0, b1, sched, steps,
                             err, 0, kPersistSpinLimit, out, launches, st);
    }
    static const MarchTable *table() {
        static const MarchTable t = {&march_shape<Op>, &march_steps<Op>, &march_cut<Op>,
                                     &march_words<Op>,
                                     &march_short<Op>, &naive_shape<Op>, &one, &many,
                                     &naive_cut, &phase_one, &phase_many};
        return &t;
    }
};

}  // namespace swept
