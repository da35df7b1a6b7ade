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
// |r| = 2^63 would get); |r| <= 2^63.  `rare` (fx_rare of be, the same for a whole
// column): the result may lie outside the normal range, or be is FX_NAN or more, NaN.
constexpr int FX_NAN = 1 << 20;
static __device__ __noinline__ double fx_to_f64_rare(fx r, int be) {
    const ufx a = r < 0 ? 0ull - (ufx)r : (ufx)r;
    const int lz = __clzll((fx)a), e = be - lz;
    const ufx m = a << (lz & 63);
    ufx bits = ((ufx)(unsigned)(e - 1) << 52) + (m >> 11) + ((m >> 10) & 1u);
    if (e <= 0) bits = e < -52 ? 0 : ((m >> (11 - e)) + 1) >> 1;   // units of 2^-1074
    if (e >= 0x7ff) bits = 0x7ffull << 52;
    if (a == 0) bits = 0;
    if (be >= FX_NAN) bits = 0x7ff8ull << 48;
    return __longlong_as_double((fx)(bits | (ufx)((unsigned)((ufx)r >> 32) & 0x80000000u) << 32));
}
__device__ __forceinline__ bool fx_rare(int be) { return (unsigned)(be - 64) >= 0x7ffu - 65u; }   // be + 1 too
__device__ __forceinline__ double fx_to_f64(fx r, int be, bool rare) {
    const ufx a = r < 0 ? 0ull - (ufx)r : (ufx)r;
    const int lz = __clzll((fx)a);
    const ufx m = a << (lz & 63);
    const unsigned sign = (unsigned)((ufx)r >> 32) & 0x80000000u;
    ufx bits = ((ufx)(unsigned)(be - lz - 1) << 52) + (m >> 11) + ((m >> 10) & 1u);
    if (a == 0) bits = 0;
    double v = __longlong_as_double((fx)(bits | (ufx)sign << 32));
    if (rare && (a != 0 || be >= FX_NAN)) v = fx_to_f64_rare(r, be);
    return v;
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

// ---- one component of a stencil in fixed point, beside the other in binary64
// A binary64 multiply-add of a warp holds the SM's FP64 unit for 16 cycles; a
// kernel bound by it leaves three quarters of its issue slots empty.  The stencil
// kernels compute the real part with the FP64 unit and the imaginary part with
// integer instructions, which halves the unit's work.  Measured at
// 512 x 128 x 400: a half-sweep of the finest level 98.5 -> 72 us, the transfer
// kernels of a solve 2.65 -> 2.26 and 1.43 -> 1.02 ms, the solve 12.2 -> 9.5 ms.

// Coefficients: c = m 2^-e with m in [1/2, 1], m 2^61 in two limbs whose low word
// carries e in its lowest 7 bits (a binary64 mantissa leaves 8 empty).
// Every operand is aligned to the exponent of the largest *term*, so that the
// sum is cut some 2^-58 below it however far the operands lie apart -- binary64
// multiply-adds round 2^-53 below their partial sums.

// x aligned to the exponent field emax (bits 20..30 in place), `eb` its own
// field (less that of its coefficient), with GUARD empty bits below the sign:
// cut toward minus infinity; shifts beyond 63 give 0 or -1.
template <int GUARD> __device__ __forceinline__ fx fx_align(double x, int eb, int emax) {
    const unsigned s = (unsigned)(emax - eb + (GUARD << 20)) >> 20;
    ufx m;
    asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(f64_mant(x)), "r"(s));   // (amounts above 63 give 0)
    const fx sg = (fx)(__double2hiint(x) >> 31);
    return (fx)m ^ sg;
}
// Exponent field in place.
__device__ __forceinline__ int exp_bits(double x) { return __double2hiint(x) & 0x7ff00000; }
// The result where fixed point does not reach: NaN when an operand is above
// 2^977, infinite or NaN (squares of such values overflow: a solve with them
// ends as non-finite either way), 0 when all are below 2^-863 (their squares
// vanish; imaginary parts that are zero identically, those of modes 0 and N/2,
// among them).  `lo` and `hi`: the exponent field of the largest term, before
// and after a scale.
__device__ __forceinline__ double fx_ends(double r, int lo, int hi) {
    const bool z = lo < (160 << 20);
    return __hiloint2double(hi >= (2000 << 20) ? 0x7ff80000 : z ? 0 : __double2hiint(r), z ? 0 : __double2loint(r));
}
__device__ __forceinline__ double fx_ends(double r, int em) { return fx_ends(r, em, em); }
// The nearest binary64 value of r 2^(be - 1086), r in the normal range: one
// conversion by the FP64 unit (a little more than one of its slots; some 25
// integer instructions otherwise) and an exact change of the exponent.
__device__ __forceinline__ double fx_to_f64_normal(fx r, int be) {
    const double d = __ll2double_rn(r);
    return r ? __hiloint2double(__double2hiint(d) + ((be - 1086) << 20), __double2loint(d)) : 0.0;
}
// The same by integer instructions, ties to even: bit for bit the conversion's.
__device__ __forceinline__ double fx_to_f64_int(fx r, int be) {
    const ufx a = r < 0 ? 0ull - (ufx)r : (ufx)r;
    const int lz = __clzll((fx)a);
    const ufx m = a << (lz & 63);
    const ufx q = m + 0x3ffu + ((unsigned)(m >> 11) & 1u);         // (below 2^64: m < 2^64 - 2^10 for |r| < 2^63)
    const ufx bits = (q >> 11) + ((ufx)(unsigned)(be - lz - 1) << 52);
    const double d = __longlong_as_double((fx)(bits | (ufx)((unsigned)((ufx)r >> 32) & 0x80000000u) << 32));
    return r ? d : 0.0;
}
__device__ __forceinline__ int coef_exp(int2 c) { return (c.y & 127) << 20; }
__device__ __forceinline__ Limbs coef_limbs(int2 c) { return {c.x, c.y & ~127}; }

// b + hz (s + n) + hw w + he e (a Gauss-Seidel update).  All terms below 2^60.
// INT: the conversion by integer instructions -- where few warps are in flight, or
// the FP64 unit has more to do besides than the integer pipes (a half-sweep of many
// waves: 74 us with the unit, 79 without; a restriction 65 and 61; 48 x 16 x 20 in
// shared memory 282 and 270).
template <bool INT = false>
__device__ __forceinline__ double fx_update(double b, double s, double n, double w, double e, int2 hz, int2 hw, int2 he) {
    const int ez = coef_exp(hz), eb = exp_bits(b), es = exp_bits(s) - ez, en = exp_bits(n) - ez;
    const int ew = exp_bits(w) - coef_exp(hw), ee = exp_bits(e) - coef_exp(he);
    const int em = max(max(max(eb, es), max(en, ew)), ee);
    const fx x = fx_align<3>(s, es, em) + fx_align<3>(n, en, em);
    const fx y = fx_align<3>(w, ew, em), z = fx_align<3>(e, ee, em);
    const Limbs c = coef_limbs(hz), d = coef_limbs(hw), f = coef_limbs(he);
    const int xh = (int)(x >> 31), xl = (int)((unsigned)x & 0x7fffffffu), yh = (int)(y >> 31),
              yl = (int)((unsigned)y & 0x7fffffffu), zh = (int)(z >> 31), zl = (int)((unsigned)z & 0x7fffffffu);
    // (the products of the low limbs, below two units each, are left out)
    fx m1 = (fx)xh * c.l, m2 = (fx)xl * c.h, hi = (fx)xh * c.h;
    m1 += (fx)yh * d.l;
    m2 += (fx)yl * d.h;
    hi += (fx)yh * d.h;
    m1 += (fx)zh * f.l;
    m2 += (fx)zl * f.h;
    hi += (fx)zh * f.h;
    const fx r = 2 * hi + (m1 >> 30) + (m2 >> 30) + fx_align<3>(b, eb, em);
    return fx_ends(INT ? fx_to_f64_int(r, (em >> 20) + 4) : fx_to_f64_normal(r, (em >> 20) + 4), em);
}
template <bool INT = false>
__device__ __forceinline__ double fx_update(double b, double s, double n, double w, double e, int4 zw, int2 ev) {
    return fx_update<INT>(b, s, n, w, e, make_int2(zw.x, zw.y), make_int2(zw.z, zw.w), ev);
}
// b + cz (s + n) + cw w + ce e - d u, the coefficients given times 2^q (|q| < 60).
template <bool INT = false>
__device__ __forceinline__ double fx_residual(double b, double s, double n, double w, double e, double u, int2 cz, int2 cw,
                                              int2 ce, int2 cd, int q) {
    const int ez = coef_exp(cz), es = exp_bits(s) - ez, en = exp_bits(n) - ez, eb = exp_bits(b) + q * (1 << 20);
    const int ew = exp_bits(w) - coef_exp(cw), ee = exp_bits(e) - coef_exp(ce), eu = exp_bits(u) - coef_exp(cd);
    const int em = max(max(max(es, en), max(ew, ee)), max(eu, eb));
    const fx x = fx_align<3>(s, es, em) + fx_align<3>(n, en, em);
    const fx y = fx_align<3>(w, ew, em), z = fx_align<3>(e, ee, em);
    const fx v = fx_align<3>(u, eu, em);
    const Limbs c = coef_limbs(cz), d = coef_limbs(cw), f = coef_limbs(ce), g = coef_limbs(cd);
    const int xh = (int)(x >> 31), xl = (int)((unsigned)x & 0x7fffffffu), yh = (int)(y >> 31),
              yl = (int)((unsigned)y & 0x7fffffffu), zh = (int)(z >> 31), zl = (int)((unsigned)z & 0x7fffffffu),
              vh = (int)(v >> 31), vl = (int)((unsigned)v & 0x7fffffffu);
    fx m1 = (fx)xh * c.l, m2 = (fx)xl * c.h, hi = (fx)xh * c.h;
    m1 += (fx)yh * d.l;
    m2 += (fx)yl * d.h;
    hi += (fx)yh * d.h;
    m1 += (fx)zh * f.l;
    m2 += (fx)zl * f.h;
    hi += (fx)zh * f.h;
    m1 -= (fx)vh * g.l;
    m2 -= (fx)vl * g.h;
    hi -= (fx)vh * g.h;
    const fx r = 2 * hi + (m1 >> 30) + (m2 >> 30) + fx_align<3>(b, eb, em);
    const int emq = em - q * (1 << 20);
    const int be = (emq >> 20) + 4;
    return fx_ends(INT ? fx_to_f64_int(r, be) : fx_to_f64_normal(r, be), min(em, emq), max(em, emq));
}
// The same with four couplings of their own (per-row tables): b + hs s + hw w + he e + hn n.
struct FxCell {                  // sums of products of aligned operands with coefficients
    fx hi = 0, m1 = 0, m2 = 0;
    __device__ __forceinline__ void add(fx x, int2 c) {
        const Limbs l = coef_limbs(c);
        const int xh = (int)(x >> 31), xl = (int)((unsigned)x & 0x7fffffffu);
        hi += (fx)xh * l.h;
        m1 += (fx)xh * l.l;
        m2 += (fx)xl * l.h;
    }
    __device__ __forceinline__ void sub(fx x, int2 c) {
        const Limbs l = coef_limbs(c);
        const int xh = (int)(x >> 31), xl = (int)((unsigned)x & 0x7fffffffu);
        hi -= (fx)xh * l.h;
        m1 -= (fx)xh * l.l;
        m2 -= (fx)xl * l.h;
    }
    __device__ __forceinline__ fx total() const { return 2 * hi + (m1 >> 30) + (m2 >> 30); }
};
__device__ __forceinline__ double fx_update(double b, double s, double w, double e, double n, int4 sw, int4 en) {
    const int2 hs = make_int2(sw.x, sw.y), hw = make_int2(sw.z, sw.w), he = make_int2(en.x, en.y), hn = make_int2(en.z, en.w);
    const int eb = exp_bits(b), es = exp_bits(s) - coef_exp(hs), ew = exp_bits(w) - coef_exp(hw);
    const int ee = exp_bits(e) - coef_exp(he), et = exp_bits(n) - coef_exp(hn);
    const int em = max(max(max(es, et), max(ew, ee)), eb);
    FxCell t;
    t.add(fx_align<3>(s, es, em), hs);
    t.add(fx_align<3>(w, ew, em), hw);
    t.add(fx_align<3>(e, ee, em), he);
    t.add(fx_align<3>(n, et, em), hn);
    return fx_ends(fx_to_f64_normal(t.total() + fx_align<3>(b, eb, em), (em >> 20) + 4), em);
}
// b + cs s + cw w + ce e + cn n - d u, the coefficients given times 2^q.
__device__ __forceinline__ double fx_residual(double b, double s, double w, double e, double n, double u, int4 sw, int4 en,
                                              int2 d, int q) {
    const int2 cs = make_int2(sw.x, sw.y), cw = make_int2(sw.z, sw.w), ce = make_int2(en.x, en.y), cn = make_int2(en.z, en.w);
    const int eb = exp_bits(b) + q * (1 << 20), es = exp_bits(s) - coef_exp(cs), ew = exp_bits(w) - coef_exp(cw);
    const int ee = exp_bits(e) - coef_exp(ce), et = exp_bits(n) - coef_exp(cn), eu = exp_bits(u) - coef_exp(d);
    const int em = max(max(max(es, et), max(ew, ee)), max(eb, eu));
    FxCell t;
    t.add(fx_align<3>(s, es, em), cs);
    t.add(fx_align<3>(w, ew, em), cw);
    t.add(fx_align<3>(e, ee, em), ce);
    t.add(fx_align<3>(n, et, em), cn);
    t.sub(fx_align<3>(u, eu, em), d);
    const int emq = em - q * (1 << 20);
    return fx_ends(fx_to_f64_int(t.total() + fx_align<3>(b, eb, em), (emq >> 20) + 4), min(em, emq), max(em, emq));
}
// u + (9 c0 + 3 (+-c1) + 3 (+-c2) +- c3) / 16: bilinear interpolation, s1 s2 set for a minus.
__device__ __forceinline__ double fx_bilinear(double u, double c0, double c1, double c2, double c3, bool s1, bool s2) {
    const int em = max(max(max(exp_bits(u), exp_bits(c0)), max(exp_bits(c1), exp_bits(c2))), exp_bits(c3));
    const fx a = fx_align<4>(c0, exp_bits(c0), em);
    const fx m1 = s1 ? -1 : 0, m2 = s2 ? -1 : 0;   // (one's complement: a unit off)
    const fx t = (fx_align<4>(c1, exp_bits(c1), em) ^ m1) + (fx_align<4>(c2, exp_bits(c2), em) ^ m2);
    const fx r = 8 * a + a + 2 * t + t + (fx_align<4>(c3, exp_bits(c3), em) ^ m1 ^ m2);
    return fx_ends(fx_to_f64_normal((r >> 4) + fx_align<4>(u, exp_bits(u), em), (em >> 20) + 5), em);
}
// u + (3 c0 +- c1) / 4.
__device__ __forceinline__ double fx_linear(double u, double c0, double c1, bool s1) {
    const int em = max(max(exp_bits(u), exp_bits(c0)), exp_bits(c1));
    const fx a = fx_align<4>(c0, exp_bits(c0), em), m1 = s1 ? -1 : 0;
    const fx r = 2 * a + a + (fx_align<4>(c1, exp_bits(c1), em) ^ m1);
    return fx_ends(fx_to_f64_normal((r >> 2) + fx_align<4>(u, exp_bits(u), em), (em >> 20) + 5), em);
}


// Sums of products of a column's values, aligned to the column's largest exponent
// (fx_align<5>: below 2^58), with constants |c| <= 1 as c 2^61 = h 2^31 + l,
// |l| <= 2^30.  Up to 64 products with sum |c| <= 8: three multiply-adds of the
// integer pipe each in place of one that holds the FP64 unit for 16 cycles, and
// sums that do not depend on their order.
struct FxSum {
    fx hi = 0, m1 = 0, m2 = 0;
};
__device__ __forceinline__ int2 fx_split(fx x) {
    const int h = (int)((x + (1ll << 30)) >> 31);
    return make_int2(h, (int)(x - ((fx)h << 31)));
}
__device__ __forceinline__ int4 fx_split2(fx x, fx y) {
    const int2 a = fx_split(x), b = fx_split(y);
    return make_int4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void fx_mac(FxSum &s, int xh, int xl, int2 c) {
    s.hi += (fx)xh * c.x;
    s.m1 += (fx)xh * c.y;
    s.m2 += (fx)xl * c.x;
}
__device__ __forceinline__ fx fx_total(const FxSum &s) { return 2 * s.hi + (s.m1 >> 30) + (s.m2 >> 30); }
// A total as binary64, em the column's exponent field.
__device__ __forceinline__ double fx_column(fx r, int em) { return fx_ends(fx_to_f64_normal(r, (em >> 20) + 6), em); }

}  // namespace pp
