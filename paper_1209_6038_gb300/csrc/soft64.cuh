// soft64.cuh -- IEEE double products on the integer pipes.
//
// An SM of this part issues one FP64 warp instruction every 19 cycles (a warp alone: one every 64, whatever
// its independent instructions), while the integer and FP32 pipes of its four schedulers stay nearly idle
// under the integrator: 76 issue slots pass per FP64 instruction and scheduler.  A correctly rounded double
// product takes about 30 integer instructions (four 32 x 32 -> 64 bit multiply-adds, one normalising shift,
// round to nearest even), 44 cycles of a scheduler with twelve resident warps, and runs beside the FP64 unit:
// equal numbers of these products and of hardware FMAs take 38 cycles per operation together, against 76 all
// in hardware (measured: 12 warps per SM, eight independent chains per thread).
//
// The results are those of __dmul_rn bit for bit wherever both factors and the product are normal numbers;
// callers see to that with s64_range and take the hardware operation elsewhere (zero, subnormal, infinite or
// NaN factors, extreme exponents).
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define S64_FN __host__ __device__ __forceinline__
#else
#define S64_FN inline
#endif

namespace ck {

// bits of a double, funnel shift, carry chains; the functions of this file compile for the host as well (the tests
// check them against exact arithmetic there)
S64_FN int s64_hi(double a) {
#ifdef __CUDA_ARCH__
    return __double2hiint(a);
#else
    long long b;
    memcpy(&b, &a, 8);
    return (int)(b >> 32);
#endif
}
S64_FN int s64_lo(double a) {
#ifdef __CUDA_ARCH__
    return __double2loint(a);
#else
    long long b;
    memcpy(&b, &a, 8);
    return (int)b;
#endif
}
S64_FN double s64_make(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t b = (uint64_t)hi << 32 | lo;
    double a;
    memcpy(&a, &b, 8);
    return a;
#endif
}
S64_FN int64_t s64_bits(double a) { return (int64_t)((uint64_t)(uint32_t)s64_hi(a) << 32 | (uint32_t)s64_lo(a)); }
S64_FN uint32_t s64_max(uint32_t a, uint32_t b) { return a > b ? a : b; }
S64_FN uint32_t s64_funnel(uint32_t lo, uint32_t hi, uint32_t sh) {  // high word of (hi : lo) << sh, 0 < sh < 32
#ifdef __CUDA_ARCH__
    return __funnelshift_l(lo, hi, sh);
#else
    return hi << sh | lo >> (32 - sh);
#endif
}
// (w3 : w2 : w1) = (hh : 0) + (cr : 0) + hi(p0)
S64_FN void s64_columns(uint64_t p0, uint64_t cr, uint64_t hh, uint32_t &w1, uint32_t &w2, uint32_t &w3) {
#ifdef __CUDA_ARCH__
    asm("add.cc.u32 %0, %3, %4;\n\taddc.cc.u32 %1, %5, %6;\n\taddc.u32 %2, %7, 0;"
        : "=r"(w1), "=r"(w2), "=r"(w3)
        : "r"((uint32_t)(p0 >> 32)), "r"((uint32_t)cr), "r"((uint32_t)(cr >> 32)), "r"((uint32_t)hh),
          "r"((uint32_t)(hh >> 32)));
#else
    const uint64_t a = (p0 >> 32) + (uint32_t)cr, b = (a >> 32) + (cr >> 32) + (uint32_t)hh;
    w1 = (uint32_t)a; w2 = (uint32_t)b; w3 = (uint32_t)((b >> 32) + (hh >> 32));
#endif
}
// round to nearest even: (rh : rl) = (mh + e : ml) + carry of (rest : low) + (half - 1 + last bit of ml)
S64_FN void s64_round(uint32_t low, uint32_t rest, uint32_t ml, uint32_t mh, uint32_t e, uint32_t &rl, uint32_t &rh) {
#ifdef __CUDA_ARCH__
    asm("{\n\t.reg .u32 t, k;\n\tand.b32 k, %4, 1;\n\tadd.cc.u32 t, k, 0xffffffff;\n\t"
        "addc.cc.u32 t, %2, 0xffffffff;\n\taddc.cc.u32 t, %3, 0x7fffffff;\n\taddc.cc.u32 %0, %4, 0;\n\t"
        "addc.u32 %1, %5, %6;\n\t}"
        : "=r"(rl), "=r"(rh)
        : "r"(low), "r"(rest), "r"(ml), "r"(mh), "r"(e));
#else
    const uint64_t half = (uint64_t)0x7fffffffu << 32 | 0xffffffffu, r = (uint64_t)rest << 32 | low;
    const uint64_t c = r + half + (ml & 1u) < r ? 1 : 0, t = (uint64_t)ml + c;
    rl = (uint32_t)t;
    rh = mh + e + (uint32_t)(t >> 32);
#endif
}

// Below S64_LIMIT iff 2^-127 <= |a| < 2^128 (the doubled high word drops the sign).  With every input of an
// expression in this range, products of up to seven of them stay normal.  Ranges are combined with max.
constexpr uint32_t S64_LIMIT = 0x1fe00000u;
S64_FN uint32_t s64_range(double a) { return (uint32_t)s64_hi(a) * 2u + 0x90000000u; }
S64_FN uint32_t s64_range(double a, double b) { return s64_max(s64_range(a), s64_range(b)); }
S64_FN bool s64_ok(uint32_t range) { return range < S64_LIMIT; }

// a * b rounded to nearest even; a, b and the product normal
S64_FN double s64_mul(double a, double b) {
    const uint32_t ah = (uint32_t)s64_hi(a), al = (uint32_t)s64_lo(a);
    const uint32_t bh = (uint32_t)s64_hi(b), bl = (uint32_t)s64_lo(b);
    const uint32_t am = (ah & 0xfffffu) | 0x100000u, bm = (bh & 0xfffffu) | 0x100000u;
    // the 106-bit product of the significands: w3 (10 bits) : w2 : w1 : low word of p0
    const uint64_t p0 = (uint64_t)al * bl;
    const uint64_t cr = (uint64_t)al * bm + (uint64_t)am * bl;
    const uint64_t hh = (uint64_t)am * bm;
    uint32_t w1, w2, w3;
    s64_columns(p0, cr, hh, w1, w2, w3);
    const uint32_t n = w3 >> 9;  // 1 when the product of the significands is 2 or more
    const uint32_t sh = 12u - n;
    const uint32_t mh = s64_funnel(w2, w3, sh), ml = s64_funnel(w1, w2, sh), rest = w1 << sh;
    // signs and exponents add modulo 2^32; the leading significand bit of mh adds one to the exponent
    const uint32_t e = n * 0x100000u + ((ah & 0xfff00000u) - 0x40000000u) + (bh & 0xfff00000u);
    uint32_t rl, rh;
    s64_round((uint32_t)p0, rest, ml, mh, e, rl, rh);
    return s64_make(rh, rl);
}

// true for +0 and -0
S64_FN bool s64_is_zero(double a) {
    return (((uint32_t)s64_hi(a) << 1) | (uint32_t)s64_lo(a)) == 0u;
}
// zero ? 0 : a, and a stand-in 1 for a factor that is exactly zero (its products are cleared afterwards)
S64_FN double s64_clear(bool zero, double a) { return zero ? 0.0 : a; }
S64_FN double s64_nonzero(bool zero, double a) { return zero ? 1.0 : a; }

// a / 2 for a in range
S64_FN double s64_half(double a) {
    return s64_make((uint32_t)s64_hi(a) - 0x100000u, (uint32_t)s64_lo(a));
}

// a <= b and a > b without the FP64 unit, for a, b >= 0 (not -0) or NaN of either sign: as the hardware's, false with
// a NaN (whose bits order above infinity, or below every number)
S64_FN bool s64_le_pos(double a, double b) {
    return s64_bits(a) <= s64_bits(b) && s64_bits(a) >= 0 && s64_bits(b) <= 0x7ff0000000000000ll;
}
S64_FN bool s64_gt_pos(double a, double b) {
    return s64_bits(a) > s64_bits(b) && s64_bits(b) >= 0 && s64_bits(a) <= 0x7ff0000000000000ll;
}
// a > 0 for any a (false for NaN)
S64_FN bool s64_positive(double a) {
    const int64_t b = s64_bits(a);
    return b > 0 && b <= 0x7ff0000000000000ll;
}
// a <= 0, a >= 0 for any a (false for NaN)
S64_FN bool s64_not_positive(double a) {
    const int64_t b = s64_bits(a);
    return b == 0 || (b < 0 && (uint64_t)b <= 0xfff0000000000000ull);
}
S64_FN bool s64_not_negative(double a) {
    const uint64_t b = (uint64_t)s64_bits(a);
    return b <= 0x7ff0000000000000ull || b == 0x8000000000000000ull;
}
S64_FN double s64_abs(double a) {
    return s64_make((uint32_t)s64_hi(a) & 0x7fffffffu, (uint32_t)s64_lo(a));
}
S64_FN bool s64_isnan(double a) {
    return (s64_bits(a) & 0x7fffffffffffffffll) > 0x7ff0000000000000ll;
}

// (float)a, rounded to nearest even, for a = +0 or 2^-125 <= a < 2^127; else ok is cleared
S64_FN float s64_to_float(double a, bool &ok) {
    const uint32_t h = (uint32_t)s64_hi(a), l = (uint32_t)s64_lo(a);
    const uint32_t u = s64_funnel(l, h, 3) - (896u << 23), rest = l << 3;
    const bool zero = (h | l) == 0u;
    if (!(zero || h - ((1023u - 125u) << 20) < (252u << 20))) ok = false;
    const uint32_t r = u + (rest > 0x80000000u - (u & 1u) ? 1u : 0u);  // the 29 bits dropped, to nearest even
#ifdef __CUDA_ARCH__
    return zero ? 0.f : __uint_as_float(r);
#else
    float f;
    memcpy(&f, &r, 4);
    return zero ? 0.f : f;
#endif
}
// a to single precision by truncation (relative error below 2^-23), of any sign, for 2^-125 <= |a| < 2^127; outside
// that the result is 0 or huge
S64_FN float s64_truncate(double a) {
    const uint32_t h = (uint32_t)s64_hi(a), m = h & 0x7fffffffu;
    uint32_t u = s64_funnel((uint32_t)s64_lo(a), m, 3) - (896u << 23);
    u = m < (898u << 20) ? 0u : m < (1150u << 20) ? u : 0x7f000000u;
    u |= h & 0x80000000u;
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float f;
    memcpy(&f, &u, 4);
    return f;
#endif
}
// (double)a for a positive normal float
S64_FN double s64_from_float(float a) {
#ifdef __CUDA_ARCH__
    const uint32_t u = __float_as_uint(a);
#else
    uint32_t u;
    memcpy(&u, &a, 4);
#endif
    return s64_make((u >> 3) + (896u << 20), u << 29);
}

}  // namespace ck
