// Complex fixed-point arithmetic for the constant-matrix marches.
//
// On this part a warp's FP64 instruction occupies its SM sub-partition for 64 cycles (DFMA;
// 76 for DADD) and nothing overlaps it, while a 32 x 32 -> 64-bit integer multiply-add
// (mad.wide.s32) takes 2.1 cycles, a 64-bit add 2.3 and a shift 2.0 (measured with
// register-only loops at one, two and four warps per sub-partition).  A complex
// multiply-add is 256 cycles in FP64 and about 45 here.  A march has a bounded state and
// constant coefficients, so it can be held in 64-bit integers:
//   value        X = x 2^sc, |X| < 2^61, sc fixed per right-hand side at its start;
//   coefficient  C = c 2^61, |c| < 2, held as two signed 32-bit limbs C = Ch 2^32 + Cl.
// With X = Xh 2^32 + Xl, Xl signed as well, a product is
//   X C / 2^61 = 8 Xh Ch + (Xh Cl + Xl Ch) / 2^29 + Xl Cl / 2^61,
// the last term (at most two units) dropped: three multiply-adds per real product, summed in
// 64-bit accumulators and rounded to nearest once per sum.  The rounding error is an
// absolute one, about one unit of 2^-sc, where FP64 rounds each value to 53 bits.  Signed low
// limbs give the dropped term no mean: with an unsigned Xl it is a constant of up to one
// unit per coefficient, the same at every step, and 200 steps of the plain workload then
// ended 1.3e-13 off instead of 4e-14 in FP64.  Splitting at 32 bits costs one or two
// instructions (the low limb is the low register).  Where even two units show (coarse grids,
// S_0^2 ends: fx_full in swr_capi.cu) the last term is taken too (fx_mac_full).
//
// No accumulator wraps: over the (at most six) real products of one component, two of them
// with |X| < 2^61 and the others with |X| < 2^60,
//   |Xh Ch| <= 2^29 2^30 each, and
//   |Xh Cl + Xl Ch| summed <= (4 2^28 + 2 2^29) 2^31 + 2^31 2^29 sum|c| < 2^63
// for coefficients whose moduli sum to at most 2.6 (checked when they are converted).
#pragma once

#include <limits.h>
#include <stdint.h>
#include <string.h>

typedef long long fx_int;

struct FxC {             // complex value
    fx_int r, i;
};
struct FxS {             // its limbs
    int rh, rl, ih, il;
};
struct FxAcc {           // sums of products: high and middle parts of each component
    fx_int hr, mr, hi, mi;
};

__device__ __forceinline__ FxC fx_zero() { return FxC{0, 0}; }
__device__ __forceinline__ FxC fx_add(FxC a, FxC b) { return FxC{a.r + b.r, a.i + b.i}; }
// high limb rounded: the carry of the low word's top bit (two additions; a shift costs two)
__device__ __forceinline__ int fx_hi(fx_int x) {
    int h;
    asm("{\n\t.reg .u32 a, b;\n\tmov.b64 {a, b}, %1;\n\t"
        "add.cc.u32 a, a, 0x80000000;\n\taddc.u32 %0, b, 0;\n\t}"
        : "=r"(h)
        : "l"(x));
    return h;
}
__device__ __forceinline__ FxS fx_split(FxC x) {
    return FxS{fx_hi(x.r), (int)x.r, fx_hi(x.i), (int)x.i};
}
// 2 x - u by additions (a 64-bit shift costs two 2-cycle instructions, an addition 2.3)
__device__ __forceinline__ fx_int fx_twice_less(fx_int x, fx_int u) {
    fx_int d;
    asm("{\n\t.reg .s64 a;\n\tsub.s64 a, %1, %2;\n\tadd.s64 %0, a, %1;\n\t}" : "=l"(d) : "l"(x), "l"(u));
    return d;
}
__device__ __forceinline__ FxC fx_twice_less(FxC x, FxC u) {
    return FxC{fx_twice_less(x.r, u.r), fx_twice_less(x.i, u.i)};
}
// a = 0, with half a unit of the result (2^-29 of a middle unit) for rounding to nearest
__device__ __forceinline__ FxAcc fx_acc() {
    const fx_int half = (fx_int)1 << 28;
    return FxAcc{0, half, 0, half};
}
__device__ __forceinline__ fx_int fx_mw(int a, int b, fx_int c) {
    fx_int d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}
// a += x c  (c: the limbs (re high, re low, im high, im low)).  The coefficient's limbs take the
// minus sign: a low limb of x may be -2^31, whose negation wraps; fx_limbs makes no such one
__device__ __forceinline__ void fx_mac(FxAcc& a, FxS x, int4 c) {
    const int nz = -c.z, nw = -c.w;
    a.hr = fx_mw(x.ih, nz, fx_mw(x.rh, c.x, a.hr));
    a.mr = fx_mw(x.rl, c.x, fx_mw(x.rh, c.y, a.mr));
    a.mr = fx_mw(x.il, nz, fx_mw(x.ih, nw, a.mr));
    a.hi = fx_mw(x.ih, c.x, fx_mw(x.rh, c.z, a.hi));
    a.mi = fx_mw(x.rl, c.z, fx_mw(x.rh, c.w, a.mi));
    a.mi = fx_mw(x.il, c.x, fx_mw(x.ih, c.y, a.mi));
}
// the same with the products of the low limbs (their high words): an error of a few 2^-32
// units instead of about one, at half as much again; for the separators, whose values every
// node of their chunks sees
__device__ __forceinline__ void fx_mac_full(FxAcc& a, FxS x, int4 c) {
    fx_mac(a, x, c);
    a.mr += (fx_int)__mulhi(x.rl, c.y) - __mulhi(x.il, c.w);
    a.mi += (fx_int)__mulhi(x.rl, c.w) + __mulhi(x.il, c.y);
}
// fx_mac, or fx_mac_full where a march takes all its products whole (FULL, see swr_march_fx.cu)
template <bool FULL>
__device__ __forceinline__ void fx_mul(FxAcc& a, FxS x, int4 c) {
    if constexpr (FULL) fx_mac_full(a, x, c);
    else fx_mac(a, x, c);
}
__device__ __forceinline__ FxC fx_res(const FxAcc& a) {
    return FxC{8 * a.hr + (a.mr >> 29), 8 * a.hi + (a.mi >> 29)};
}
// the sum divided by 2^k (k < 0: times 2^-k), rounded once; the sum started from fx_acc_shr(k)
__device__ __forceinline__ FxAcc fx_acc_shr(int k) {
    const fx_int half = (fx_int)1 << (28 + min(k, 3));
    return FxAcc{0, half, 0, half};
}
// (k < 0: m gets its top bit set where the result would not stay below 2^top)
__device__ __forceinline__ FxC fx_res_shr(const FxAcc& a, int k, unsigned& m, int top = 58) {
    const int e = min(k, 3);
    if (k < 0) {
        const int b = top - 3 + k;
        const fx_int lim = (fx_int)1 << b;
        if ((unsigned long long)(a.hr + lim) >> (b + 1) || (unsigned long long)(a.hi + lim) >> (b + 1))
            m |= 0x80000000u;
    }
    FxC r = {(a.hr << (3 - e)) + (a.mr >> (29 + e)), (a.hi << (3 - e)) + (a.mi >> (29 + e))};
    if (k > 3) {
        const fx_int half = (fx_int)1 << (k - 4);
        r = FxC{(r.r + half) >> (k - 3), (r.i + half) >> (k - 3)};
    }
    return r;
}
// x / 2^k rounded to nearest (k >= 0), x 2^-k for k < 0
__device__ __forceinline__ fx_int fx_shr(fx_int x, int k) {
    if (k > 0) return (x + ((fx_int)1 << (k - 1))) >> k;
    return x << -k;
}
__device__ __forceinline__ FxC fx_shr(FxC x, int k) { return FxC{fx_shr(x.r, k), fx_shr(x.i, k)}; }
// the same with the rounding constant given (half = 2^(k-1), or 0 for k = 0)
__device__ __forceinline__ FxC fx_shr_c(FxC x, int k, fx_int half) {
    return FxC{(x.r + half) >> k, (x.i + half) >> k};
}
// c ? a : b without an indexed register array (see csel)
__device__ __forceinline__ FxC fx_sel(bool c, FxC a, FxC b) {
    FxC r;
    asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %4, 0;\n\t"
        "selp.b64 %0, %2, %5, q;\n\tselp.b64 %1, %3, %6, q;\n\t}"
        : "=l"(r.r), "=l"(r.i)
        : "l"(a.r), "l"(a.i), "r"((unsigned)c), "l"(b.r), "l"(b.i));
    return r;
}
__device__ __forceinline__ FxC fx_up(FxC v, int d) {
    return FxC{__shfl_up_sync(0xffffffffu, v.r, d), __shfl_up_sync(0xffffffffu, v.i, d)};
}
__device__ __forceinline__ FxC fx_down(FxC v, int d) {
    return FxC{__shfl_down_sync(0xffffffffu, v.r, d), __shfl_down_sync(0xffffffffu, v.i, d)};
}
__device__ __forceinline__ FxC fx_from(FxC v, int lane) {
    return FxC{__shfl_sync(0xffffffffu, v.r, lane), __shfl_sync(0xffffffffu, v.i, lane)};
}
// range check: OR of the high words offset by 2^k; bits from 2^(k+1) on are set if a component
// is outside [-2^(32+k), 2^(32+k))
template <int K>
__device__ __forceinline__ unsigned fx_range(unsigned m, FxC x) {
    return m | ((unsigned)(int)(x.r >> 32) + (1u << K)) | ((unsigned)(int)(x.i >> 32) + (1u << K));
}
// magnitude bits of the high words, OR-ed into m (sign folded)
__device__ __forceinline__ unsigned fx_mag(unsigned m, FxC x) {
    const int a = (int)(x.r >> 32), b = (int)(x.i >> 32);
    return m | (unsigned)(a ^ (a >> 31)) | (unsigned)(b ^ (b >> 31));
}
// a += x c for a real power of two c (high limb only)
__device__ __forceinline__ void fx_mac_pow2(FxAcc& a, FxS x, int ch) {
    a.hr = fx_mw(x.rh, ch, a.hr);
    a.mr = fx_mw(x.rl, ch, a.mr);
    a.hi = fx_mw(x.ih, ch, a.hi);
    a.mi = fx_mw(x.il, ch, a.mi);
}
// limbs of a coefficient
__host__ __device__ __forceinline__ int2 fx_limbs(double c) {
    // rint(c 2^61) from the bits of c (ties away from zero): a conversion instruction and the
    // scaling before it cost 64 cycles each
    fx_int b;
    memcpy(&b, &c, sizeof b);
    const int e = (int)((b >> 52) & 0x7ff) - 1023 + 61 - 52;      // c = m 2^(e - 61)
    const fx_int m = (b & 0xfffffffffffffLL) | (e > -1023 + 61 - 52 ? 0x10000000000000LL : 0);
    fx_int C = e >= 0 ? m << (e < 10 ? e : 10) : (e > -54 ? ((m >> (-e - 1)) + 1) >> 1 : 0);
    if (b < 0) C = -C;
    C += (int)C == INT_MIN;   // its low limb has a negative (see fx_mac)
    const int l = (int)C;
    return make_int2((int)((C - l) >> 32), l);
}
__host__ __device__ __forceinline__ int4 fx_coef(double re, double im) {
    const int2 a = fx_limbs(re), b = fx_limbs(im);
    return make_int4(a.x, a.y, b.x, b.y);
}
// 2^e as a double, -1022 <= e <= 1023
__device__ __forceinline__ double fx_pow2(int e) {
    return __longlong_as_double((long long)(e + 1023) << 52);
}
// smallest e with x <= 2^e (x > 0, finite)
__device__ __forceinline__ int fx_clog2(double x) {
    const int e = ilogb(x);
    return x > scalbn(1.0, e) ? e + 1 : e;
}
