// 64-bit fixed-point arithmetic in place of binary64 instructions.  This GPU's
// FP64 unit runs at 1/64 of the FP32 rate (a warp instruction occupies it for 16
// cycles of the SM, 64 issue slots of a scheduler), so a handful of integer
// instructions per operation is several times faster, and a 64-bit integer
// scaled to a known bound carries more bits than a binary64 mantissa.
#pragma once

#include <cuda_runtime.h>

namespace pp {

typedef long long fx;               // value times a power of two that the code around it knows
typedef unsigned long long ufx;

// Exponent field (11 bits) of a binary64 value.
__device__ __forceinline__ int f64_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// The 53-bit mantissa of x, shifted left by 10 (bit 62 set); x's sign is not
// applied and zeros and subnormals are not told apart.
__device__ __forceinline__ ufx f64_mant(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    return (((ufx)((hi & 0xfffffu) | 0x100000u)) << 32 | lo) << 10;
}

// x times 2^(10 - s) / (one unit of its mantissa), rounded to nearest (ties
// away from zero); zeros and subnormals give 0.  1 <= s.
__device__ __forceinline__ fx f64_to_fx(double x, int s) {
    const int hi = __double2hiint(x);
    const ufx h = f64_mant(x) >> min(s - 1, 63);
    const fx v = (fx)((h + 1) >> 1);
    const fx r = hi < 0 ? -v : v;
    return (hi & 0x7ff00000) == 0 ? 0 : r;
}

// The nearest binary64 value of r 2^(be - 1086) (be: the biased exponent that
// |r| = 2^63 would get); |r| <= 2^63.  Results below the normal range become
// signed zero, above it infinite.
__device__ __forceinline__ double fx_to_f64(fx r, int be) {
    const ufx a = r < 0 ? 0ull - (ufx)r : (ufx)r;
    const int lz = __clzll((fx)a);
    const ufx m = a << (lz & 63);
    const int e = be - lz;
    const unsigned sign = (unsigned)((ufx)r >> 32) & 0x80000000u;
    ufx bits = ((ufx)(unsigned)(e - 1) << 52) + (m >> 11) + ((m >> 10) & 1u);
    if (e >= 0x7ff) bits = 0x7ffull << 52;
    if (a == 0 || e <= 0) bits = 0;
    return __longlong_as_double((fx)(bits | (ufx)sign << 32));
}

// A constant |c| <= 1 as two 31-bit limbs: c 2^61 = h 2^31 + l, 0 <= l < 2^31.
struct Limbs {
    int h, l;
};

// a c + b d with c, d in limbs; |a|, |b| < 2^61 and |c| + |d| <= 1.5 keep the
// sums inside 63 bits.  The value is cut below one unit after the sum of the
// two products' low parts.
__device__ __forceinline__ fx fx_mul2(fx a, Limbs c, fx b, Limbs d) {
    const int ah = (int)(a >> 31), al = (int)((unsigned)a & 0x7fffffffu);
    const int bh = (int)(b >> 31), bl = (int)((unsigned)b & 0x7fffffffu);
    const ufx low = (ufx)((fx)al * c.l) + (ufx)((fx)bl * d.l);   // below 2^63
    fx mid = (fx)(low >> 31) + (1ll << 29);                      // rounded at the cut by 30 bits
    mid += (fx)ah * c.l;
    mid += (fx)al * c.h;
    mid += (fx)bh * d.l;
    mid += (fx)bl * d.h;
    fx hi = (fx)ah * c.h;
    hi += (fx)bh * d.h;
    return 2 * hi + (mid >> 30);
}

}  // namespace pp
