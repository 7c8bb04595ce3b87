// Sums of float64 products on the integer pipe (block fixed point).
//
// GB300 issues FP64 multiply-adds at 2 per clock and SM (0.63 T/s measured
// over the chip) and 32 x 32 + 64-bit integer multiply-adds (IMAD.WIDE) at 31
// (9.2 T/s).  A float64 factor becomes a signed 60-bit integer on the scale of
// the largest factor of its group, X = v 2^(1082 - e) truncated, e the largest
// biased exponent of the group (|X| < 2^60), split X = h 2^32 + l with both
// words signed.  A product then costs three IMAD.WIDE,
//   X Y = hX hY 2^64 + (hX lY + lX hY) 2^32 + lX lY,
// into two 64-bit accumulators; the last term, below 2^62, is dropped: it is
// 2^-58 of the largest product of the group, the truncation of the factors
// 2^-59.  A chain of FP64 multiply-adds rounds at 2^-53 of its running value in
// every step.  A group is the few values that a thread holds at a time: the values of a
// line of cell nodes, the rows of one sum.  Within it an error is bounded by the
// group's largest, so a group never spans results of their own.
//
// Values below 2^-959 (biased exponent under 64) lose bits and count as zero below
// 2^-1018, except in the cell pass, which scales such lines up; groups with an
// infinity or NaN, or whose products leave the float64 range, give NaN (the cell
// pass: what FP64 gives).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace afem {

struct Fx {
    int h, l;   // h 2^32 + l
};
// Two accumulators of a sum of products: hh counts 2^64, x counts 2^32.
struct FxAcc {
    long long hh, x;
};

constexpr unsigned kFxExpMask = 0x7FF00000u;
constexpr int kFxMinExp = 64;        // smallest group exponent
constexpr int kFxMaxSum = 3124;      // largest ex + ey whose scale is a normal number

// The biased exponent of v in bits 20..30 (sign and significand cleared).
__device__ __forceinline__ unsigned fx_expbits(double v) { return unsigned(__double2hiint(v)) & kFxExpMask; }

// v on the scale of the group exponent e >= kFxMinExp (and >= v's own).
__device__ __forceinline__ long long fx_int(double v, int e) {
    const unsigned hw = unsigned(__double2hiint(v)), lw = unsigned(__double2loint(v));
    const unsigned mh = (hw & 0xFFFFFu) | 0x100000u;
    int s = e - int((hw >> 20) & 0x7FFu);
    s = s < 63 ? s : 63;
    const unsigned long long m =
        ((static_cast<unsigned long long>(__funnelshift_l(lw, mh, 7)) << 32) | (lw << 7)) >> s;
    return int(hw) < 0 ? -static_cast<long long>(m) : static_cast<long long>(m);
}
__device__ __forceinline__ Fx fx_split(long long x) {
    Fx r;
    r.l = int(x);
    r.h = int(x >> 32) + int(unsigned(r.l) >> 31);
    return r;
}
__device__ __forceinline__ Fx fx_make(double v, int e) { return fx_split(fx_int(v, e)); }

// -a (l = -2^31 has no positive counterpart and borrows from h).
__device__ __forceinline__ Fx fx_neg(Fx a) {
    Fx r;
    r.l = int(0u - unsigned(a.l));
    r.h = (a.l == int(0x80000000u) ? 1 : 0) - a.h;
    return r;
}

__device__ __forceinline__ void fx_mad(FxAcc& a, Fx u, Fx v) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.hh) : "r"(u.h), "r"(v.h));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.x) : "r"(u.h), "r"(v.l));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.x) : "r"(u.l), "r"(v.h));
}
// The same with a factor u in constant memory, which the instruction takes as
// its operand (written as above it is moved to a register first: 17 % more
// instructions in the cell pass; the vector passes have 15 % fewer as above).
__device__ __forceinline__ void fx_mad_const(FxAcc& a, Fx u, Fx v) {
    a.hh += static_cast<long long>(u.h) * v.h;
    a.x += static_cast<long long>(u.h) * v.l;
    a.x += static_cast<long long>(u.l) * v.h;
}

// Moves the high word of x to hh.  A product adds less than 2^60 - 2^27 to x, so
// x holds 8 products from zero, or 7 and what a carry left (below 2^32).
__device__ __forceinline__ void fx_carry(FxAcc& a) {
    a.hh += a.x >> 32;
    a.x &= 0xFFFFFFFFll;
}

// The accumulated sum over 2^63, rounded to float64; the sum itself is this
// times fx_scale(ex + ey) with the group exponents of the factors (up to 32
// products between float64 sums: |hh| < 2^62).
__device__ __forceinline__ double fx_value(const FxAcc& a) { return __ll2double_rn((a.hh << 1) + (a.x >> 31)); }
// 2^(esum - 2101): subnormal, then zero, below the normal range (the sums it
// scales reach 2^62), NaN above it.
__device__ __forceinline__ double fx_scale_edge(int f) {
    return f > 0 ? __hiloint2double(0x7FF80000, 0) : f < -51 ? 0.0 : __longlong_as_double(1ll << (f + 51));
}
__device__ __forceinline__ double fx_scale(int esum) {
    const int f = esum - 1078;
    return unsigned(f - 1) < 2046u ? __hiloint2double(f << 20, 0) : fx_scale_edge(f);
}

// t 2^k rounded to binary32 (nearest, ties to even; results below the normal
// range become signed zeros, above it infinities, as narrow_f64).
__device__ __forceinline__ float fx_to_f32(long long t, int k) {
    const unsigned u = __float_as_uint(__ll2float_rn(t));   // exact exponent and rounding: t has no subnormals
    const int e = int((u >> 23) & 0xFFu), ef = e + k;
    const unsigned sign = u & 0x80000000u;
    if (e == 0 || ef <= 0) return __uint_as_float(sign);
    if (ef >= 255) return __uint_as_float(sign | 0x7F800000u);
    return __uint_as_float(u + (unsigned(k) << 23));
}
}  // namespace afem
