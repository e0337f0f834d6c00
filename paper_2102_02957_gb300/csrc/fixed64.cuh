// Block fixed-point arithmetic for complex128 gates on the integer pipe.
//
// Measured on GB300, per clock and SM: 2.0 FP64 FMAs, 57 to 61 32-bit integer multiply-adds into a
// 64-bit accumulator (mad.wide.s32), 63 shifts or logic operations, 125 32-bit adds.  So a
// complex128 gate runs faster as integer arithmetic where its amplitudes are comparable in size: those that a
// thread holds (one gate's pair or quadruple, or a register group's 16) share one exponent E, the largest of their components',
// and every component becomes a signed 64-bit integer
//     X = x * 2^(1081 - E)          (E: biased exponent; |X| < 2^59 on entry, 6 bits below the
//                                    last mantissa bit of the largest component)
// that stays in this form through all gates the thread applies.  A gate entry becomes
//     M = round(m * 2^61) = mh * 2^32 + ml,   X = h * 2^32 + l   (all four signed, l and ml balanced)
// and a product is three 32-bit multiply-adds into two 64-bit accumulators,
//     X M / 2^61 = 8 h mh + (h ml + l mh) / 2^29 + [l ml / 2^61],
// the bracket (at most 2 units, of either sign) dropped.
//
// Ranges, for gates unitary to 1e-9 (the host checks; other gates stay on FP64): a register group
// has 32 components, so its 2-norm, which gates keep, is below sqrt(32) 2^59 = 2^61.5 and so is
// every component ever formed; a row of a two-qubit gate has 8 real products with sum |h ml| <=
// sqrt(8) 2^29.5 2^31 = 2^62 and sum |l mh| <= 2^31 sqrt(8) 2^29 = 2^61.5: the middle accumulator
// stays below 2^63.
//
// Precision: a gate's output component is off by about a unit, 2^-59 of 2^E, where FP64 rounds four
// or eight times per gate, each time to 2^-53 of the partial sum; back in FP64 it is rounded once.
// So amplitudes near the largest gain, and those more than 2^6 below it, which FP64 would keep to 53 bits as
// long as no gate adds anything larger to them (a phase, a small angle, a product state), lose.  Callers
// therefore take this form only where the results draw on comparable amplitudes, and FP64 elsewhere: the
// per-gate sweeps decide group by group (k_gate.cu, apply_fx), sections chunk by chunk (block_fx.cuh,
// ChunkRange).  Zeros, ones and permutations stay exact.  Not for components that are not finite or for a
// largest one outside 2^-959 .. 2^1017 (fx::special).
#pragma once
#include <stdint.h>

namespace sv {
namespace fx {

constexpr int kOne = 1 << 29;  // mh of an entry of exactly 1 (ml = 0)

struct Real {  // one component: X = h * 2^32 + l
    int h, l;
};

struct Acc {
    long long hi = 0, mid = 1ll << 28;  // mid starts at the rounding half
};

__device__ __forceinline__ Real pack(long long v) {
    return Real{(int)(v >> 32) + (int)((unsigned)v >> 31), (int)v};
}

__device__ __forceinline__ long long value(const Real &x) {
    return (long long)((unsigned long long)(unsigned)x.h << 32) + x.l;
}

__device__ __forceinline__ void mac(Acc &a, const Real &x, int mh, int ml) {
    a.hi += (long long)x.h * mh;
    a.mid += (long long)x.h * ml;
    a.mid += (long long)x.l * mh;
}

__device__ __forceinline__ Real fin(const Acc &a) {
    return pack((long long)((unsigned long long)a.hi << 3) + (a.mid >> 29));
}

__device__ __forceinline__ Real negate(const Real &x) { return pack(-value(x)); }

// A double's own words, for gates that only exchange components and flip signs.
__device__ __forceinline__ Real from_bits(double x) { return Real{__double2hiint(x), __double2loint(x)}; }
__device__ __forceinline__ double to_bits(const Real &x) { return __hiloint2double(x.h, x.l); }
__device__ __forceinline__ Real flip_sign(const Real &x) { return Real{x.h ^ (int)0x80000000, x.l}; }

// |high word| and "any bit of the magnitude" of a component, for the exponent search.
__device__ __forceinline__ void scan(double x, int &top, int &any) {
    const int hi = __double2hiint(x) & 0x7FFFFFFF;
    top = max(top, hi);
    any |= hi | __double2loint(x);
}

// Whether components with largest high word `top` and bits `any` are outside the fixed-point range.
__device__ __forceinline__ bool special(int top, int any) {
    return (any != 0 && top < (64 << 20)) || top >= (2040 << 20);
}

// Shared exponent for `top` (an all-zero set gets one that maps every component to 0).
__device__ __forceinline__ int exponent(int top) { return max(top >> 20, 64); }

__device__ __forceinline__ Real from_double(double x, int E) {
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    const int d = min(E - ((hi >> 20) & 0x7FF), 63);  // a zero's distance is at least 64: shifted out
    const unsigned long long m = ((unsigned long long)(unsigned)((hi & 0xFFFFF) | 0x100000) << 32) | lo;
    unsigned long long v = (m << 6) >> d;
    const long long s = (long long)(hi >> 31);
    v = (v ^ (unsigned long long)s) - (unsigned long long)s;
    return pack((long long)v);
}

__device__ __forceinline__ double to_double(const Real &x, int E) {
    const unsigned long long v = (unsigned long long)value(x);
    const long long s = (long long)v >> 63;
    unsigned long long a = (v ^ (unsigned long long)s) - (unsigned long long)s;
    const int ah = (int)(a >> 32), al = (int)a;
    const int lz = ah ? __clz(ah) : 32 + __clz(al);
    a <<= lz & 63;
    // mantissa with its hidden bit added to exponent - 1; the rounding bit may carry into it
    unsigned long long b = (a >> 11) + ((a >> 10) & 1);
    b += (unsigned long long)(unsigned)(E + 4 - lz) << 52;
    b |= (unsigned long long)(s & (long long)0x8000000000000000ull);
    return __longlong_as_double((ah | al) ? (long long)b : 0);
}

}  // namespace fx
}  // namespace sv
