// IEEE 754 binary64 arithmetic computed on the integer pipes.
//
// The FP64 pipe of sm_103a issues two thread instructions per cycle per SM
// (one warp instruction every 64 cycles per scheduler), while a scheduler
// issues one warp instruction every cycle to the integer and FP32 pipes.
// The flux kernels are bound by the FP64 pipe with the other pipes almost
// idle, so part of their arithmetic runs here instead.  The kernels call the
// reduced-range functions (*_mid, below): mul_mid and add_mid return the bits of
// the correctly rounded result that the DMUL / DADD instruction gives (IEEE
// 754-2008 Sect. 4.3.1, roundTiesToEven), so a product or sum may move between
// the pipes without changing one bit; recip_mid, harm_mid and sqrt_mid are
// within the bounds stated with them, a little above half a unit in the last
// place, and not correctly rounded.  mul_chk / add_chk and mul_rn / add_rn /
// sub_rn take every range; the tests' probe alone calls them.
//
// Method (the textbook integer formulation of binary floating point, e.g.
// J.-M. Muller et al., Handbook of Floating-Point Arithmetic, 2nd ed., 2018,
// Sects. 7.2-7.3, and D. Goldberg, "What every computer scientist should
// know about floating-point arithmetic", ACM Comput. Surv. 23 (1991), on
// guard digits and the sticky bit):
//   product: the 53 x 53-bit significand product is formed exactly in four
//     32 x 32 -> 64-bit integer multiply-adds; its top 53 bits are the
//     significand, the next bit is the guard bit and every lower bit is
//     OR-ed into a sticky bit; round up when guard and (sticky or the
//     significand's last bit).
//   sum: the operand of smaller magnitude is aligned to the larger in a
//     64-bit frame with 10 bits below the significand; bits shifted out are
//     OR-ed into the last bit of the frame, which makes the frame value odd
//     whenever the sum is inexact, so no rounding boundary (all of them
//     multiples of 2^8 in the frame) can lie between it and the exact sum;
//     then normalisation and the same rounding rule as the product.
// Carries of the rounding step propagate into the exponent field, which
// also gives the correct infinity on overflow.
//
// The integer path handles normal and zero operands whose exact result is
// normal or zero.  mul_chk / add_chk compute without a branch and clear a
// caller's flag for everything else (subnormal operands or results,
// infinities, NaNs, overflow before rounding); the *_mid functions clear it for
// operands that are neither zero nor of moderate exponent, and a kernel checks
// the flag once per evaluation and redoes that evaluation on the FP64 pipe.
// mul_rn / add_rn, single operations, take a slow path that is the hardware
// instruction itself.  Both redo paths sit in functions that are never
// inlined, so that no FP64 instruction stands on the fast path, not even
// predicated off (a predicated-off FP64 instruction still occupies the FP64
// pipe).
//
// The functions compile for the host as well (plain C++ on the same
// integer steps), where tests check them bit for bit against the host's
// IEEE arithmetic.
#pragma once
#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define EMU_HD __host__ __device__ __forceinline__
#else
#define EMU_HD inline
#endif

namespace jfnk {
namespace emu {

EMU_HD uint32_t hi_word(double x) {
#if defined(__CUDA_ARCH__)
    return (uint32_t)__double2hiint(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    return (uint32_t)(u >> 32);
#endif
}

EMU_HD uint32_t lo_word(double x) {
#if defined(__CUDA_ARCH__)
    return (uint32_t)__double2loint(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    return (uint32_t)u;
#endif
}

EMU_HD double from_words(uint32_t hi, uint32_t lo) {
#if defined(__CUDA_ARCH__)
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t u = ((uint64_t)hi << 32) | lo;
    double x;
    memcpy(&x, &u, 8);
    return x;
#endif
}

EMU_HD double from_bits(uint64_t u) { return from_words((uint32_t)(u >> 32), (uint32_t)u); }

// low 32 bits of (hi:lo) >> s, 0 <= s < 32
EMU_HD uint32_t shr_pair(uint32_t lo, uint32_t hi, uint32_t s) {
#if defined(__CUDA_ARCH__)
    return __funnelshift_r(lo, hi, s);
#else
    return (uint32_t)((((uint64_t)hi << 32) | lo) >> s);
#endif
}

// 1/f for f in (1, 2], within one unit in the last place (the MUFU pipe's
// approximation on the device)
EMU_HD uint32_t rcp_bits(uint32_t f) {
#if defined(__CUDA_ARCH__)
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(f)));
    return __float_as_uint(r);
#else
    float x, r;
    memcpy(&x, &f, 4);
    r = 1.0f / x;
    uint32_t u;
    memcpy(&u, &r, 4);
#if defined(EMU_RCP_ERROR)
    u += EMU_RCP_ERROR;          // tests: an approximation that is off by some units
#endif
    return u;
#endif
}

// 1/sqrt(f) for f in [1, 4), within a few units in the last place (MUFU)
EMU_HD uint32_t rsqrt_bits(uint32_t f) {
#if defined(__CUDA_ARCH__)
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(f)));
    return __float_as_uint(r);
#else
    float x, r;
    memcpy(&x, &f, 4);
    r = (float)(1.0 / __builtin_sqrt((double)x));
    uint32_t u;
    memcpy(&u, &r, 4);
#if defined(EMU_RCP_ERROR)
    u += 3 * EMU_RCP_ERROR;
#endif
    return u;
#endif
}

EMU_HD uint32_t mul_hi(uint32_t a, uint32_t b) {
#if defined(__CUDA_ARCH__)
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

// number of leading zero bits of a nonzero 64-bit value
EMU_HD int clz64(uint64_t x) {
#if defined(__CUDA_ARCH__)
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}

// a*b on the integer path, without a branch.  The return value is the
// correctly rounded product whenever a and b are normal or zero and the
// exact product is normal or zero; otherwise it is meaningless and ok is
// cleared (ok is never set, so a caller can check a whole sequence of
// operations once and redo it on the FP64 pipe where it failed).
EMU_HD double mul_chk(double a, double b, bool& ok) {
    const uint32_t ah = hi_word(a), al = lo_word(a), bh = hi_word(b), bl = lo_word(b);
    const uint32_t sign = (ah ^ bh) & 0x80000000u;
    // exponent fields in place (bits 20..30) and the product's before
    // normalisation; unsigned wrap-around rejects the out-of-range cases:
    // a and b normal, and the normalised exponent e0 (+1) within [1, 2046]
    const uint32_t ea = ah & 0x7ff00000u, eb = bh & 0x7ff00000u;
    const uint32_t e0 = ea + eb - 0x3ff00000u;
    const bool normal = (ea - 0x00100000u < 0x7fe00000u) & (eb - 0x00100000u < 0x7fe00000u) &
                        (e0 - 0x00100000u < 0x7fd00000u);
    // a zero times a finite number: a zero carrying the sign of the product
    const bool zero = ((((ah & 0x7fffffffu) | al) == 0u) | (((bh & 0x7fffffffu) | bl) == 0u)) &
                      (ea != 0x7ff00000u) & (eb != 0x7ff00000u);
    // significands with the hidden bit: (ma:al) and (mb:bl), 53 bits each
    const uint32_t ma = (ah & 0xfffffu) | 0x100000u, mb = (bh & 0xfffffu) | 0x100000u;
    // exact 106-bit product w3:w2:w1:w0 in four 32x32->64 multiply-adds
    const uint64_t t0 = (uint64_t)al * bl;
    const uint64_t t1 = (uint64_t)al * mb + (t0 >> 32);
    const uint64_t t2 = (uint64_t)ma * bl + (uint32_t)t1;
    const uint64_t t3 = (uint64_t)ma * mb + (t1 >> 32) + (t2 >> 32);
    const uint32_t w0 = (uint32_t)t0, w1 = (uint32_t)t2, w2 = (uint32_t)t3, w3 = (uint32_t)(t3 >> 32);
    // the product lies in [2^104, 2^106): s = 1 when bit 105 is set
    const uint32_t s = w3 >> 9;
    const uint32_t mlo = shr_pair(w1, w2, 20u + s);          // significand bits 0..31
    const uint32_t mhi = shr_pair(w2, w3, 20u + s);          // bits 32..52 (hidden bit at 20)
    // guard bit at the top of `rest`, the bits below it, w0 != 0 as bit 0;
    // round up (to nearest, ties to even) exactly when rest + 0x7fffffff +
    // the last significand bit carries out of 32 bits
    const uint32_t rest = (w1 << (12u - s)) | (uint32_t)(w0 != 0u);
    const uint32_t up = (uint32_t)(((uint64_t)rest + (0x7fffffffu + (mlo & 1u))) >> 32);
    // exponent field e0 + s: e0 + (s - 1) << 20 plus the hidden bit of mhi;
    // the rounding carry runs into the exponent (infinity on overflow)
    const uint32_t hi = sign + (e0 + (s << 20) - 0x00100000u) + mhi;
    const uint64_t bits = (((uint64_t)hi << 32) | mlo) + up;
    ok = ok & (normal | zero);
    return zero ? from_words(sign, 0u) : from_bits(bits);
}

// a+b on the integer path, without a branch; ok as for mul_chk (operands
// normal or zero, exact sum normal or zero).
EMU_HD double add_chk(double a, double b, bool& ok) {
    const uint32_t ah = hi_word(a), al = lo_word(a), bh = hi_word(b), bl = lo_word(b);
    const uint32_t am = ah & 0x7fffffffu, bm = bh & 0x7fffffffu;
    // x: the operand of larger magnitude (a on ties), y the other
    const bool swap = (bm > am) | ((bm == am) & (bl > al));
    const uint32_t xh = swap ? bh : ah, xl = swap ? bl : al;
    const uint32_t yh = swap ? ah : bh, yl = swap ? al : bl;
    const uint32_t ex = (xh >> 20) & 0x7ffu, ey = (yh >> 20) & 0x7ffu;
    const bool sub = ((ah ^ bh) & 0x80000000u) != 0u;
    // 64-bit frames: significand with hidden bit at bit 62, 10 bits below it
    const uint64_t X = ((uint64_t)((xh & 0xfffffu) | 0x100000u) << 42) | ((uint64_t)xl << 10);
    const uint64_t Y = ((uint64_t)((yh & 0xfffffu) | 0x100000u) << 42) | ((uint64_t)yl << 10);
    const uint32_t d = ex - ey < 63u ? ex - ey : 63u;          // Y >> 63 is 0: top bit at 62
    const uint64_t lost = Y & ((1ull << d) - 1ull);
    const uint64_t Ya = (Y >> d) | (uint64_t)(lost != 0ull);
    const uint64_t S0 = sub ? X - Ya : X + Ya;
    // normalise to bit 62: one place right after a carry (sticky kept),
    // left by the leading zeros after a cancellation
    const int lz = clz64(S0) - 1;                              // -1 .. 63 (63: S0 == 0)
    const uint64_t S = lz < 0 ? ((S0 >> 1) | (S0 & 1ull)) : (S0 << (uint32_t)(lz < 0 ? 0 : lz));
    const uint32_t e = ex - (uint32_t)lz;
    const uint32_t rem = (uint32_t)S & 0x3ffu;
    const uint64_t m = S >> 10;
    const uint64_t up = (uint64_t)((rem + (uint32_t)(m & 1ull)) > 0x200u);
    const uint64_t bits = ((((uint64_t)(xh & 0x80000000u)) << 32) | ((uint64_t)(e - 1u) << 52)) + m + up;
    // y == 0: the sum is x; two zeros of opposite signs give +0
    const bool yzero = ((yh & 0x7fffffffu) | yl) == 0u;
    const bool xzero = ((xh & 0x7fffffffu) | xl) == 0u;
    const bool normal = (ey != 0u) & (ex - 1u < 2046u);
    const bool exact0 = S0 == 0ull;                            // x - x: +0
    ok = ok & ((yzero & (ex != 0x7ffu)) | (normal & (exact0 | (e - 1u < 2046u))));
    const double viax = (sub & xzero) ? 0.0 : from_words(xh, xl);
    return yzero ? viax : (exact0 ? 0.0 : from_bits(bits));
}

// The range that the reduced checks below take: zero, or an exponent within
// 500 of one (a product of two such values, or a reciprocal, is normal, so one
// comparison per operand replaces the checks of the result).
EMU_HD bool mid_range(uint32_t hi_mag) { return hi_mag - 0x20b00000u < 0x3e800000u; }

// a*b as mul_chk for zero operands and operands of moderate exponent (ok is
// cleared for the others)
EMU_HD double mul_mid(double a, double b, bool& ok) {
    const uint32_t ah = hi_word(a), al = lo_word(a), bh = hi_word(b), bl = lo_word(b);
    const uint32_t am = ah & 0x7fffffffu, bm = bh & 0x7fffffffu;
    const uint32_t sign = (ah ^ bh) & 0x80000000u;
    const bool za = (am | al) == 0u, zb = (bm | bl) == 0u;
    ok = ok & (mid_range(am) | za) & (mid_range(bm) | zb);
    const uint32_t ma = (ah & 0xfffffu) | 0x100000u, mb = (bh & 0xfffffu) | 0x100000u;
    const uint64_t t0 = (uint64_t)al * bl;
    const uint64_t t1 = (uint64_t)al * mb + (t0 >> 32);
    const uint64_t t2 = (uint64_t)ma * bl + (uint32_t)t1;
    const uint64_t t3 = (uint64_t)ma * mb + (t1 >> 32) + (t2 >> 32);
    const uint32_t w0 = (uint32_t)t0, w1 = (uint32_t)t2, w2 = (uint32_t)t3, w3 = (uint32_t)(t3 >> 32);
    const uint32_t s = w3 >> 9;
    const uint32_t mlo = shr_pair(w1, w2, 20u + s), mhi = shr_pair(w2, w3, 20u + s);
    const uint32_t rest = (w1 << (12u - s)) | (uint32_t)(w0 != 0u);
    const uint32_t up = (uint32_t)(((uint64_t)rest + (0x7fffffffu + (mlo & 1u))) >> 32);
    const uint32_t e0 = (am & 0x7ff00000u) + (bm & 0x7ff00000u) - 0x40000000u;     // biased, less the hidden bit
    const uint32_t hi = sign + (e0 + (s << 20)) + mhi;
    const uint64_t bits = (((uint64_t)hi << 32) | mlo) + up;
    return (za | zb) ? from_words(sign, 0u) : from_bits(bits);
}

// 2^63 / s for s = S / 2^63 in [1, 2): R in (2^62, 2^63 (1 + 2^-58)], within 2^-58 of
// the quotient.  Newton's iteration r + r (1 - s r) in fixed point from a
// 24-bit approximation: 32 bits after the first step, all after the second
// (J.-M. Muller et al., Handbook of Floating-Point Arithmetic, 2nd ed., 2018,
// Sect. 4.7).
EMU_HD uint64_t recip_q63(uint64_t S) {
    const uint32_t sh = (uint32_t)(S >> 32), sl = (uint32_t)S;
    // f: the next float above sh / 2^31, so its reciprocal lies in [1/2, 1)
    // (held there against the approximation's error at 1/2) and its
    // significand with the hidden bit is the top of a 32-bit fraction
    const uint32_t rb = rcp_bits((sh >> 8) + 0x3f000001u);
    const uint32_t r0 = ((rb > 0x3f000000u ? rb : 0x3f000000u) << 8) | 0x80000000u;   // / 2^32
    // 31 bits: r1 / 2^31, from the error 2^31 - s r0 (|error| < 2^11)
    const int32_t e0 = (int32_t)(0x80000000u - mul_hi(sh, r0));
    const uint32_t r1 = (r0 >> 1) + (uint32_t)((int64_t)((int64_t)e0 * (int32_t)(r0 >> 1)) >> 31);
    // s r1 / 2^31 = 1 - e1 with |e1| < 2^-28: e1 in units of 2^-62
    const uint64_t lo = (uint64_t)sl * r1;
    const uint64_t mid = (uint64_t)sh * r1 + (lo >> 32);
    const int32_t e1 = (int32_t)((int64_t)(0x4000000000000000ull - mid) >> 4);   // 2^-58
    return ((uint64_t)r1 << 32) + (uint64_t)((int64_t)((int64_t)e1 * (int32_t)r1) >> 26);
}

// 1/d for d of moderate exponent (ok is cleared for others, zero included):
// within (1/2 + 2^-4) units in the last place of the exact reciprocal
EMU_HD double recip_mid(double d, bool& ok) {
    const uint32_t dh = hi_word(d), dl = lo_word(d);
    const uint32_t dm = dh & 0x7fffffffu;
    ok = ok & mid_range(dm);
    const uint32_t sh = shr_pair(dl, (dh & 0xfffffu) | 0x100000u, 21u), sl = dl << 11;
    const uint64_t R = recip_q63(((uint64_t)sh << 32) | sl);
    const uint64_t m = (R + 0x200ull) >> 10;                              // hidden bit at 52
    // biased exponent 2045 - that of d, less the hidden bit; sign of d
    const uint32_t hi = (dh & 0x80000000u) + (0x7fc00000u - (dm & 0x7ff00000u)) + (uint32_t)(m >> 32);
    return from_words(hi, (uint32_t)m);
}

// sqrt(x) for positive x of moderate exponent (ok is cleared for others, zero
// included): within (1/2 + 2^-3) units in the last place.  With x = s 4^k, s in
// [1, 4): a Newton step takes the 24-bit approximation of 1/sqrt(s) to 30 bits;
// g, s times that, is the root to 28 bits, and g + (s - g^2) / (2 g), with the
// remainder exact in 64 bits, leaves an error of 2^-56.
EMU_HD double sqrt_mid(double x, bool& ok) {
    const uint32_t xh = hi_word(x), xl = lo_word(x);
    ok = ok & mid_range(xh);                                             // false for negative x as well
    const uint32_t odd = (~xh >> 20) & 1u;                               // odd exponent: biased exponent even
    const uint32_t fb = shr_pair(xl, xh & 0xfffffu, 29u) + 0x3f800000u + (odd << 23);
    uint32_t rb = rsqrt_bits(fb);
    rb = rb > 0x3f000000u ? rb : 0x3f000000u;                            // [1/2, 1)
    rb = rb < 0x3f7fffffu ? rb : 0x3f7fffffu;
    const uint32_t r0 = (rb << 8) | 0x80000000u;                         // / 2^32
    const uint32_t sh0 = shr_pair(xl, (xh & 0xfffffu) | 0x100000u, 22u), sl0 = xl << 10;
    const uint64_t S = (((uint64_t)sh0 << 32) | sl0) << odd;             // s 2^62
    const uint32_t sh = (uint32_t)(S >> 32);
    // e = 1 - s r0^2 in units of 2^-30 (|e| < 2^11), r1 = r0 + r0 e / 2, / 2^31
    const int32_t e = (int32_t)(0x40000000u - mul_hi(sh, mul_hi(r0, r0)));
    const uint32_t h0 = r0 >> 1;
    const uint32_t r1 = h0 + (uint32_t)((int64_t)((int64_t)e * (int32_t)h0) >> 31);
    // g 2^31, a few units low so that it stays below 2 and the remainder is positive or small
    const uint32_t g = (uint32_t)(((uint64_t)sh * r1 - (4ull << 30)) >> 30);
    const int32_t d = (int32_t)((int64_t)(S - (uint64_t)g * g) >> 7);    // s - g^2 in units of 2^-55
    const uint64_t y = ((uint64_t)g << 31) + (uint64_t)((int64_t)((int64_t)d * (int32_t)(r1 >> 1)) >> 24);
    const uint64_t m = (y + 0x200ull) >> 10;                             // hidden bit at 52
    // biased exponent (e + 1023) / 2 rounded down, less the hidden bit
    const uint32_t hi = ((((xh >> 20) + 1023u) >> 1) << 20) - 0x00100000u + (uint32_t)(m >> 32);
    return from_words(hi, (uint32_t)m);
}

// x/2 for x of moderate exponent (ok is cleared for others, zero included)
EMU_HD double half_mid(double x, bool& ok) {
    const uint32_t xh = hi_word(x);
    ok = ok & mid_range(xh & 0x7fffffffu);
    return from_words(xh - 0x00100000u, lo_word(x));
}

// the larger of a non-negative number a and any b: the words of non-negative
// numbers are ordered as integers, and a negative b has a negative high word
EMU_HD double max_nonneg(double a, double b) {
    const uint32_t ah = hi_word(a), bh = hi_word(b), al = lo_word(a), bl = lo_word(b);
    const bool g = ((int32_t)ah > (int32_t)bh) | ((ah == bh) & (al > bl));
    return from_words(g ? ah : bh, g ? al : bl);
}

// a b / (a + b) for a, b of the same sign and moderate exponent, 0 where the
// signs differ or one is zero; within (1/2 + 2^-3) units in the last place.
// The limited slope of the flux kernels in one go: the sum is aligned but not
// rounded, and its reciprocal, the two products and one rounding follow in
// 64-bit fixed point, so the FP64 pipe keeps the differences a and b and the
// addition to the cell value.
EMU_HD double harm_mid(double a, double b, bool& ok) {
    const uint32_t ah = hi_word(a), al = lo_word(a), bh = hi_word(b), bl = lo_word(b);
    const uint32_t am = ah & 0x7fffffffu, bm = bh & 0x7fffffffu;
    const bool za = (am | al) == 0u, zb = (bm | bl) == 0u;
    ok = ok & (mid_range(am) | za) & (mid_range(bm) | zb);
    const bool off = ((ah ^ bh) >> 31) | za | zb;
    // x: the operand of larger exponent
    const bool swap = bm > am;
    const uint32_t xm = swap ? bm : am, xl = swap ? bl : al, ym = swap ? am : bm, yl = swap ? al : bl;
    const uint32_t xs = (xm & 0xfffffu) | 0x100000u, ys = (ym & 0xfffffu) | 0x100000u;
    const uint32_t dd = (xm >> 20) - (ym >> 20);
    const uint32_t d = dd < 63u ? dd : 63u;
    const uint64_t X = ((uint64_t)shr_pair(xl, xs, 22u) << 32) | (xl << 10);        // hidden bit at 62
    const uint64_t Y = ((uint64_t)shr_pair(yl, ys, 22u) << 32) | (yl << 10);
    const uint64_t S0 = X + (Y >> d);                                               // [2^62, 2^64)
    const uint32_t n = 1u - (uint32_t)(S0 >> 63);
    const uint64_t R = recip_q63(S0 << n);
    // w = X / S in (1/2, 1]: W / 2^63 = (X 2^n) R / 2^126, kept as W / 2
    const uint64_t Xn = X << n;
    const uint32_t xnh = (uint32_t)(Xn >> 32), xnl = (uint32_t)Xn, rh = (uint32_t)(R >> 32), rl = (uint32_t)R;
    const uint64_t W = (uint64_t)xnh * rh + mul_hi(xnh, rl) + mul_hi(xnl, rh);      // / 2^62, at most about 2^62
    const uint32_t wh = (uint32_t)(W >> 32), wl = (uint32_t)W;
    const uint32_t yh = (uint32_t)(Y >> 32), yw = (uint32_t)Y;
    // V = Y W / 2^64: y w 2^-2 of a significand with hidden bit at 62: [2^59, 2^61]
    const uint64_t V = (uint64_t)yh * wh + mul_hi(yh, wl) + mul_hi(yw, wh);
    const uint32_t s = (uint32_t)(V >> 60) != 0u;                                   // hidden bit at 60, else 59
    const uint64_t m = (V + (64ull << s)) >> (7u + s);                              // hidden bit at 52
    const uint32_t hi = (ah & 0x80000000u) + (ym & 0x7ff00000u) + (s << 20) - 0x00200000u + (uint32_t)(m >> 32);
    return off ? 0.0 : from_words(hi, (uint32_t)m);
}

// a + b for zero operands and operands of moderate exponent (ok is cleared for
// the others), correctly rounded; a zero result is positive.  As add_chk, but
// the result needs no range check: the bits of the smaller operand that fall
// below the 64-bit frame (ten bits under the larger one's last place) are folded
// into its lowest bit, and the sum is rounded to nearest, ties to even, after
// one normalising shift.
EMU_HD double add_mid(double a, double b, bool& ok) {
    const uint32_t ah = hi_word(a), al = lo_word(a), bh = hi_word(b), bl = lo_word(b);
    const uint32_t am = ah & 0x7fffffffu, bm = bh & 0x7fffffffu;
    const bool za = (am | al) == 0u, zb = (bm | bl) == 0u;
    ok = ok & (mid_range(am) | za) & (mid_range(bm) | zb);
    const bool swap = (((uint64_t)bm << 32) | bl) > (((uint64_t)am << 32) | al);
    const uint32_t xh = swap ? bh : ah, xl = swap ? bl : al, yh = swap ? ah : bh, yl = swap ? al : bl;
    const uint32_t xm = xh & 0x7fffffffu, ym = yh & 0x7fffffffu;
    const uint32_t dd = (xm >> 20) - (ym >> 20);
    const uint32_t d = dd < 62u ? dd : 62u;                          // far below, or a zero y: the lowest bit
    const uint64_t X = ((uint64_t)shr_pair(xl, (xm & 0xfffffu) | 0x100000u, 22u) << 32) | (xl << 10);
    const uint64_t Y = ((uint64_t)shr_pair(yl, (ym & 0xfffffu) | 0x100000u, 21u) << 32) | (yl << 11);   // twice y
    const uint64_t Yd = (Y >> (d + 1u)) | (uint64_t)((Y << (63u - d)) != 0ull);
    const uint64_t sub = (uint64_t)((ah ^ bh) >> 31);
    const uint64_t S = X + ((Yd ^ (0ull - sub)) + sub);
    const uint32_t lz = (uint32_t)clz64(S | 1ull);
    const uint64_t T = S << lz;                                      // top bit at 63
    const uint64_t m0 = T >> 11;                                     // hidden bit at 52
    const uint32_t rest = (uint32_t)T << 21;
    const uint32_t up = (uint32_t)(((uint64_t)rest + (0x7fffffffu + ((uint32_t)m0 & 1u))) >> 32);
    const uint64_t m = m0 + up;
    const uint32_t hi = (xh & 0x80000000u) + (xm & 0x7ff00000u) - (lz << 20) + (uint32_t)(m >> 32);
    return ((za & zb) | (S == 0ull)) ? 0.0 : from_words(hi, (uint32_t)m);
}

// single operations with the range check: true and r = a*b (a+b) on the
// integer path; false (r meaningless) outside its range
EMU_HD bool mul_fast(double a, double b, double& r) {
    bool ok = true;
    r = mul_chk(a, b, ok);
    return ok;
}

EMU_HD bool add_fast(double a, double b, double& r) {
    bool ok = true;
    r = add_chk(a, b, ok);
    return ok;
}

#if defined(__CUDA_ARCH__)
__device__ __noinline__ double mul_slow(double a, double b) { return __dmul_rn(a, b); }
__device__ __noinline__ double add_slow(double a, double b) { return __dadd_rn(a, b); }
#else
inline double mul_slow(double a, double b) { return a * b; }
inline double add_slow(double a, double b) { return a + b; }
#endif

// a*b and a+b, correctly rounded, on the integer pipes
EMU_HD double mul_rn(double a, double b) {
    double r;
    if (mul_fast(a, b, r)) return r;
    return mul_slow(a, b);
}

EMU_HD double add_rn(double a, double b) {
    double r;
    if (add_fast(a, b, r)) return r;
    return add_slow(a, b);
}

// -b: the sign bit flips on the integer pipe
EMU_HD double neg(double b) { return from_words(hi_word(b) ^ 0x80000000u, lo_word(b)); }

// a - b
EMU_HD double sub_rn(double a, double b) { return add_rn(a, neg(b)); }

}  // namespace emu
}  // namespace jfnk
