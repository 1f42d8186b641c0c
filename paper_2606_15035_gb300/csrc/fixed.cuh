// 64-bit fixed point for bounded quantities of the orbit integrals, on the integer pipe (sm_103a).
//
// The FP64 pipe issues one warp instruction in 64 clocks per scheduler; a 64-bit multiply-add takes
// about ten integer instructions at one or two clocks each.  Coordinates, piece lengths and moments are
// at most one, so 62 fractional bits hold them (2^-62 absolute, where FP64 rounds at 2^-53 of each);
// fields and velocities carry a common power of two (the largest exponent of what they are summed
// with), kept beside them.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace pic {

// x times 2^s truncated to an integer, |x| 2^s < 2^63: `drop` is how far the exponent of x is below
// the one whose mantissa is shifted left by `up`.
__device__ __forceinline__ long long fixed_of(double x, int top, int up) {
    const int hi = __double2hiint(x);
    const int drop = min(max(top - ((hi >> 20) & 0x7ff), 0), 63);
    const unsigned long long mant =
        ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x);
    const long long r = (long long)((mant << up) >> drop);
    return hi < 0 ? -r : r;
}

// A factor: its signed high word and the upper 31 bits of its low word.
struct Fx {
    int h, l;
};

__device__ __forceinline__ Fx fx_split(long long v) { return Fx{(int)(v >> 32), (int)((unsigned)v >> 1)}; }

// a b 2^-62 from three 32 x 32 products; the constant stands for the mean of the dropped low product
// and rounds (errors within about 2 units, mean below a quarter).
__device__ __forceinline__ long long fx_mul(Fx a, Fx b) {
    const long long u = (long long)a.h * b.l + ((long long)a.l * b.h + 912680550LL);   // 1.7 x 2^29
    return (((long long)a.h * b.h) << 2) + (u >> 29);
}

constexpr long long FX_ONE = 1LL << 62;

// A factor of a sum of products: its signed high word and the upper 29 bits of its low word, so that
// eight products' cross terms stay in 63 bits.
struct Fs {
    int h, l;
};

__device__ __forceinline__ Fs fs_of(long long v) { return Fs{(int)(v >> 32), (int)((unsigned)v >> 3)}; }

// A sum of products 2^-62 (sum) a b: the high products and the cross terms are summed apart, two and
// one 32 x 32 multiply-adds a product, and shifted together once.  (A sum of separate fx_mul took about
// 25 instructions a product as compiled; this takes 3 and some 8 per sum.)  The start of u stands for
// the mean of what a product drops.
struct FxSum {
    long long t, u;
    __device__ __forceinline__ FxSum() : t(0), u(0) {}
    __device__ __forceinline__ void add(Fs a, Fs b) {
        t += (long long)a.h * b.h;
        u += (long long)a.h * b.l;
        u += (long long)a.l * b.h;
    }
    __device__ __forceinline__ void add_one(Fs a) {   // a times one
        t += (long long)a.h << 30;
        u += (long long)a.l << 30;
    }
    __device__ __forceinline__ long long value() const { return (t << 2) + ((u + (1LL << 29)) >> 27); }
    __device__ __forceinline__ Fs factor() const { return fs_of(value()); }
};

__device__ __forceinline__ FxSum fx_sum(Fs a, Fs b) {
    FxSum s;
    s.add(a, b);
    return s;
}
__device__ __forceinline__ FxSum fx_sum(Fs a, Fs b, Fs c, Fs d) {
    FxSum s = fx_sum(a, b);
    s.add(c, d);
    return s;
}

// The biased exponent of x, and the power of two of a biased exponent (0 below the normal range).
__device__ __forceinline__ int exponent_of(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ double pow2_biased(int e) { return e < 1 ? 0.0 : __hiloint2double(min(e, 2047) << 20, 0); }

}  // namespace pic
