// The FP64 heat update on the integer units, with the bits of the FP64 one.
//
// The FP64 pipe takes 19 clocks of an SM for one warp instruction, in which the
// SM can issue 76 others; the heat update has four FP64 operations, p = a + b
// (the pair sum, shared by two points), s = p1 + p2, d = fma(-4, c, s) and
// u' = fma(r, d, c). Here the magnitudes of a block whose values have one sign
// are 64-bit integers in one unit, a quarter of the last place of the lowest one's
// binade e0, which represents the normal numbers of the binades e0 .. e0 + 5 exactly:
//  - a sum is an integer addition and a rounding, to nearest even, to the 53
//    leading bits (the position of the first bit gives the rounding's);
//  - K = s / 4 - c is a multiple of 4, and d = 4 K is exact while |K| < 2^55, twice
//    the lowest value of binade e0: always, if the values differ by less;
//  - r d = 4 r K = R K 2^-64 with a 64-bit integer R, a multiple of 8, for r in
//    [2^-11, 1/4), a 128-bit product whose lower half only tells whether something
//    lies below the unit; the unit's two bits below a last place are enough for the
//    same rounding of c + r d.
// A new value is a rounded mean of old ones with weights 1 - 4r and r, so it
// stays within the block's extremes, hence in the six binades. A K that is too
// large is recorded, and the caller repeats the block's steps by the FP64
// operations; blocks on a zero crossing, or with values more than a factor of 32
// to 64 apart, take them from the start. Measured on the GB300: 4096², 500 steps,
// 35.4 ms with this (the integer ALU 68% busy), 67.4 by the FP64 operations of the
// swept kernels (their pipe 95% busy). On the host the same functions serve to compare
// them with the FP64 operations.
#pragma once
#include <cuda_runtime.h>

#include <cstring>

namespace swept {

// 4 r as R 2^-64, R a multiple of 8; 0 when r is not in [2^-11, 1/4).
__host__ __device__ inline unsigned long long heat_ratio(double r) {
    if (!(r >= 0.00048828125 && r < 0.25)) return 0;
    unsigned long long bits;
    memcpy(&bits, &r, 8);
    const int below = 1020 - (int)(bits >> 52);          // binades below [1/8, 1/4): 0 .. 8
    return ((bits & 0xfffffffffffffULL) | 0x10000000000000ULL) << (11 - below);
}

constexpr int kFixedBinades = 6;

// Position of the first set bit of a positive value's upper word.
__host__ __device__ __forceinline__ int first_bit(long long v) {
#ifdef __CUDA_ARCH__
    int p;
    asm("bfind.u32 %0, %1;" : "=r"(p) : "r"((unsigned)(v >> 32)));
    return p;
#else
    return 31 - __builtin_clz((unsigned)(v >> 32));
#endif
}

// v rounded to its 53 leading bits, to nearest even (2^53 < v < 2^63).
__host__ __device__ __forceinline__ long long leading_53(long long v) {
    const int at = first_bit(v) - 20;            // the last of the 53 bits
    unsigned below;
#ifdef __CUDA_ARCH__
    asm("bmsk.clamp.b32 %0, 0, %1;" : "=r"(below) : "r"(at));
#else
    below = (1u << at) - 1u;
#endif
    return (v + ((below >> 1) + (((unsigned)v >> at) & 1u))) & ~(long long)below;
}

// A block's unit: e0 the exponent field of its lowest binade; and its sign.
struct FixedHeat {
    unsigned long long R;        // heat_ratio(r)
    int e0;
    unsigned sign;               // 0 or 0x80000000
    unsigned wide;               // largest K seen, as the upper word of K + 2^55

    // Sets the unit for values whose upper words lie in [low, high] as signed
    // integers (of negative values, too, the larger word is the larger magnitude);
    // false unless they are normal, of one sign and within the binades, r has a
    // ratio (heat_ratio(r)), and sums stay finite.
    __host__ __device__ __forceinline__ bool fits(unsigned long long ratio, int high, int low) {
        const int top = (high >> 20) & 0x7ff;
        R = ratio;
        e0 = (low >> 20) & 0x7ff;
        sign = (unsigned)high & 0x80000000u;
        wide = 0;
        return R != 0 && (high ^ low) >= 0 && top - e0 < kFixedBinades && e0 > 0 && top < 2040;
    }
    __host__ __device__ __forceinline__ long long from(double v) const {
        long long b;
        memcpy(&b, &v, 8);
        const int e = (int)(b >> 52) & 0x7ff;
        return ((b & 0xfffffffffffffLL) | 0x10000000000000LL) << (e - e0 + 2);
    }
    __host__ __device__ __forceinline__ double to(long long v) const {
        const int up = first_bit(v) - 22;        // the binade above e0
        const long long b = ((long long)(e0 + up) << 52) | ((v >> (up + 2)) & 0xfffffffffffffLL);
        const unsigned long long bits = (unsigned long long)b | ((unsigned long long)sign << 32);
        double v64;
        memcpy(&v64, &bits, 8);
        return v64;
    }
    // some result is not the FP64 one
    __host__ __device__ __forceinline__ bool failed() const { return (wide >> 24) != 0; }
    __host__ __device__ __forceinline__ long long sum(long long a, long long b) const {
        return leading_53(a + b);
    }
    __host__ __device__ __forceinline__ long long next(long long c, long long pe, long long pw) {
        const long long K = (sum(pe, pw) >> 2) - c;
        wide = max(wide, (unsigned)(K >> 32) + (1u << 23));
        const unsigned long long Kb = (unsigned long long)(K + (1LL << 61));   // 2^61 R 2^-64 = R / 8
        const unsigned k0 = (unsigned)Kb, k1 = (unsigned)(Kb >> 32);
        const unsigned r0 = (unsigned)R, r1 = (unsigned)(R >> 32);
        const unsigned long long m0 = (unsigned long long)k0 * r0;
        const unsigned long long m1 = (unsigned long long)k0 * r1 + (m0 >> 32);
        const unsigned long long m2 = (unsigned long long)k1 * r0 + (unsigned)m1;
        const unsigned long long m3 = (unsigned long long)k1 * r1 + (m1 >> 32) + (m2 >> 32);
        const unsigned below = min((unsigned)m0 | (unsigned)m2, 1u);
        return leading_53((c - (long long)(R >> 3) + (long long)m3) | below);
    }
};

}  // namespace swept
