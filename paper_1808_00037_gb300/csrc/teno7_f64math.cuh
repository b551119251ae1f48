// teno7_f64math.cuh -- the parts of the FP64 path that need not run on the FP64
// pipe.
//
// GB300 issues one FP64 warp instruction per SM every 19 cycles (measured: add,
// multiply, FMA and compare alike, whatever the active lanes; 64 cycles from a
// single warp), while the FP32 and integer pipes take 2 to 4 per cycle.  So an
// FP64 instruction is worth some 40 integer or FP32 ones, and every decision
// that FP32 can take with a proven error bound is taken there, the FP64
// evaluation remaining for the windows the bound leaves open.  The decided
// bits are the FP64 evaluation's own.
//
// Host-compilable (T7_HD), so that the functions can be checked without a GPU.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define T7_HD __host__ __device__ __forceinline__
#else
#define T7_HD inline
#endif

namespace t7 {

T7_HD uint64_t f64_bits(double x) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    memcpy(&b, &x, 8);
    return b;
#endif
}
T7_HD double f64_of(uint64_t b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}
T7_HD float f32_of(uint32_t b) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float x;
    memcpy(&x, &b, 4);
    return x;
#endif
}
// Tests and maxima that would otherwise be FP64-pipe comparisons.
T7_HD bool f64_finite(double x) { return ((uint32_t)(f64_bits(x) >> 32) & 0x7fffffffu) < 0x7ff00000u; }
T7_HD bool f64_positive(double x) {  // x > 0 (false for NaN)
    const uint64_t b = f64_bits(x);
    return b - 1u < 0x7ff0000000000000ull;
}
// fmax of a non-negative x (not NaN) and a non-negative y or NaN
T7_HD double f64_max_pos(double x, double y) {
    const uint64_t bx = f64_bits(x), by = f64_bits(y);
    return f64_of(by > bx && by <= 0x7ff0000000000000ull ? by : bx);
}
T7_HD int f32_to_int(float x) {  // nearest integer, |x| < 2^31
#ifdef __CUDA_ARCH__
    return __float2int_rn(x);
#else
    return (int)lrintf(x);
#endif
}
// Approximate reciprocal, within 2 ulp; subnormal arguments and results (those of
// arguments above 2^126) count as zero.  (T7_HOST_ERR: a host check may scale the
// approximations by their error bound.)
#ifndef T7_HOST_ERR
#define T7_HOST_ERR
#endif
T7_HD float f32_flush(float x) { return fabsf(x) < 1.17549435e-38f ? copysignf(0.f, x) : x; }
T7_HD float f32_rcp(float x) {
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return f32_flush((1.0f / f32_flush(x)) T7_HOST_ERR);
#endif
}

T7_HD float f32_rsqrt(float x) {  // approximate 1/sqrt, within 2^-22
#ifdef __CUDA_ARCH__
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return (float)(1.0 / sqrt((double)f32_flush(x))) T7_HOST_ERR;
#endif
}

// --------------------------------------------------------------------------
// Correctly rounded FP64 quotient and square root without FP64 instructions
// (as FP64 code they take 140 to 165 cycles per warp and SM): a quotient of
// some 43 bits from FP32, its exact remainder modulo 2^64 from 32-bit integer
// products, one integer correction, and the remainder's comparison with half
// the divisor for the last bit.  No result lies on a rounding tie (a 54-bit
// quotient or root of 53-bit numbers never ends there).  Operands or results
// that are zero, subnormal, infinite or NaN go to the FP64 operation (zero
// numerators, common in resting gas, are answered at once).
//
// Quotient, with A, B the 53-bit mantissas and s = 1 if A < B, else 0: the FP32
// pair (qh, ql) approximates A/B within 2^-44, so Q0 = the integer nearest to it
// times 2^(52+s) is within 2^10 of A 2^(52+s) / B and the remainder
// A 2^(52+s) - Q0 B below 2^63; the FP32 correction then leaves a remainder of
// at most B (1/2 + 2^-10).
// --------------------------------------------------------------------------
T7_HD double div64(double a, double b) {
    const uint64_t xa = f64_bits(a), xb = f64_bits(b);
    const uint32_t ha = (uint32_t)(xa >> 32), hb = (uint32_t)(xb >> 32), la = (uint32_t)xa, lb = (uint32_t)xb;
    const int ea = (int)((ha >> 20) & 0x7ffu), eb = (int)((hb >> 20) & 0x7ffu);
    const uint32_t ma = (ha & 0xfffffu) | 0x100000u, mb = (hb & 0xfffffu) | 0x100000u;
    const uint32_t sign = (ha ^ hb) & 0x80000000u;
    const int s = (ma < mb || (ma == mb && la < lb)) ? 1 : 0;
    const int e = ea - eb + 1022 - s;  // exponent field of the result, less one
    if ((uint32_t)(ea - 1) >= 2046u || (uint32_t)(eb - 1) >= 2046u || (uint32_t)(e - 1) >= 2044u) {
        if (((ha << 1) | la) == 0u && (uint32_t)(eb - 1) < 2046u) return f64_of((uint64_t)sign << 32);
        return a / b;
    }
    // leading 24 bits in [1, 2) and the other 29
    const float ah = f32_of(0x3f800000u | ((ma << 3) & 0x7fffffu) | (la >> 29));
    const float bh = f32_of(0x3f800000u | ((mb << 3) & 0x7fffffu) | (lb >> 29));
    const float al = (float)(la & 0x1fffffffu) * 2.220446049250313e-16f;
    const float bl = (float)(lb & 0x1fffffffu) * 2.220446049250313e-16f;
    float r = f32_rcp(bh);
    r = fmaf(r, fmaf(-r, bl, fmaf(-r, bh, 1.f)), r);  // 1/B within 2^-23
    const float qh = ah * r;
    const float ql = fmaf(-qh, bl, fmaf(-qh, bh, ah) + al) * r;
    const int ih = (int)(qh * 16777216.f);                              // exact (qh > 1/2)
    const int il = f32_to_int(ql * (s ? 35184372088832.f : 17592186044416.f));  // ql 2^(44+s)
    const uint64_t Q0 = ((uint64_t)(uint32_t)ih << (28 + s)) + ((uint64_t)(int64_t)il << 8);
    const uint32_t q0 = (uint32_t)Q0, q1 = (uint32_t)(Q0 >> 32);
    const uint64_t A = (uint64_t)(la << (20 + s)) << 32;  // A 2^(52+s) mod 2^64
    const uint64_t R = A - ((uint64_t)q0 * lb + ((uint64_t)(q0 * mb + q1 * lb) << 32));
    const int c = f32_to_int((float)(int32_t)(R >> 32) * r * 9.5367431640625e-07f);  // R / B
    const uint64_t B = ((uint64_t)mb << 32) | lb;
    const int64_t R1 = (int64_t)(R - (uint64_t)(int64_t)c * B);
    const int64_t twice = R1 * 2;
    uint64_t Q = Q0 + (uint64_t)(int64_t)c;
    if (twice > (int64_t)B) Q++;
    if (twice < -(int64_t)B) Q--;
    return f64_of(((uint64_t)(sign | ((uint32_t)e << 20)) << 32) + Q);
}

// Square root of M 2^52, M = m 2^52 with m in [1, 4) and an even exponent: S0
// within 2^9 of it, the remainder M 2^52 - S0^2 modulo 2^64, one correction, and
// the last bit from M 2^52 <> (S +- 1/2)^2.
T7_HD double sqrt64(double x) {
    const uint64_t b = f64_bits(x);
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
    const int e = (int)(hi >> 20);  // sign included
    if ((uint32_t)(e - 1) >= 2046u) return sqrt(x);
    const int odd = (e & 1) ^ 1;  // the bias 1023 is odd
    const uint32_t m = (hi & 0xfffffu) | 0x100000u;
    const float scale = odd ? 2.f : 1.f;
    const float mh = f32_of(0x3f800000u | ((m << 3) & 0x7fffffu) | (lo >> 29)) * scale;
    const float ml = (float)(lo & 0x1fffffffu) * 2.220446049250313e-16f * scale;
    float y = f32_rsqrt(mh);
    float sh = mh * y;
    y = fmaf(0.5f * y, fmaf(-sh, y, 1.f), y);
    sh = mh * y;
    const float sl = (fmaf(-sh, sh, mh) + ml) * (0.5f * y);
    const int ih = (int)(sh * 16777216.f);                // exact (sh > 1/2)
    const int il = f32_to_int(sl * 4503599627370496.f);  // sl 2^52
    const uint64_t S0 = ((uint64_t)(uint32_t)ih << 28) + (uint64_t)(int64_t)il;
    const uint32_t s0 = (uint32_t)S0, s1 = (uint32_t)(S0 >> 32);
    const uint64_t M = (uint64_t)(lo << (20 + odd)) << 32;
    const uint64_t R = M - ((uint64_t)s0 * s0 + ((uint64_t)(2u * s0 * s1) << 32));
    const int c = f32_to_int((float)(int32_t)(R >> 32) * y * 4.76837158203125e-07f);  // R / (2 S)
    const uint64_t cc = (uint64_t)(int64_t)c;
    uint64_t S = S0 + cc;
    const int64_t R1 = (int64_t)(R - cc * (2u * S0 + cc));
    if (R1 > (int64_t)S) S++;
    else if (R1 <= -(int64_t)S) S--;
    return f64_of(((uint64_t)(uint32_t)(((e - 1023 - odd) >> 1) + 1022) << 52) + S);
}

// --------------------------------------------------------------------------
// Correctly rounded FP64 product on the integer pipe: four 32 x 32 -> 64-bit
// products of the mantissas, rounded to nearest even from the exact 117 bits.
// About 24 integer instructions (12 cycles per warp and SM, against 19 on the
// FP64 pipe, which meanwhile runs the sums).  One factor is prepared once
// (MulOp: mantissa left-justified in 64 bits, sign and exponent word less the
// bias); it may be zero.  The other, and a nonzero prepared one, must have a
// magnitude in [2^-400, 2^400): mul_ranged().
// --------------------------------------------------------------------------
struct MulOp {
    uint32_t xl, xh, e, mask;
};
// 0 when |x| is in [2^-400, 2^400), so that results of several values can be or-ed
T7_HD uint32_t mul_unranged(double x) {
    const uint32_t a = (uint32_t)(f64_bits(x) >> 32) & 0x7fffffffu;
    return a - ((1023u - 400u) << 20) >= (800u << 20) ? 1u : 0u;
}
T7_HD MulOp mul_op(double x) {
    const uint64_t b = f64_bits(x);
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
    MulOp o;
    o.mask = ((hi << 1) | lo) == 0u ? 0u : ~0u;
    o.xh = ((((hi & 0xfffffu) | 0x100000u) << 11) | (lo >> 21)) & o.mask;
    o.xl = lo << 11;
    o.e = (hi & 0xfff00000u) - 0x40000000u;
    return o;
}
T7_HD double mul64(const MulOp &x, double g) {
    const uint64_t b = f64_bits(g);
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b, gh = (hi & 0xfffffu) | 0x100000u;
    const uint64_t p0 = (uint64_t)x.xl * lo;
    const uint64_t p1 = (uint64_t)x.xh * lo + (p0 >> 32);
    const uint64_t p2 = (uint64_t)x.xl * gh + (uint32_t)p1;
    const uint64_t h = (uint64_t)x.xh * gh + (p1 >> 32) + (p2 >> 32);  // product >> 64: 53 or 52 bits
    const uint32_t hh = (uint32_t)(h >> 32), hl = (uint32_t)h, ll = (uint32_t)p0, lh = (uint32_t)p2;
    const int s = (hh & 0x100000u) ? 0 : 1;
    // 53-bit mantissa (mh, ml) and the 64 bits below it (rh, rl)
#ifdef __CUDA_ARCH__
    const uint32_t mh = __funnelshift_l(hl, hh, s), ml = __funnelshift_l(lh, hl, s), rh = __funnelshift_l(ll, lh, s);
#else
    const uint32_t mh = s ? (hh << 1) | (hl >> 31) : hh, ml = s ? (hl << 1) | (lh >> 31) : hl;
    const uint32_t rh = s ? (lh << 1) | (ll >> 31) : lh;
#endif
    const uint32_t up = ((ml & 1u) | (ll << s)) != 0u ? 0x80000000u : 0x7fffffffu;  // nearest, ties to even
    const uint64_t carry = ((uint64_t)rh + up) >> 32;
    const uint64_t m = (((uint64_t)mh << 32) | ml) + carry;
    const uint32_t rhi = (uint32_t)(m >> 32) + (x.e + (hi & 0xfff00000u) + (hh & 0x100000u));
    return f64_of(((uint64_t)(rhi & x.mask) << 32) | (uint32_t)m);
}

// --------------------------------------------------------------------------
// Shortcut of the cutoff test.  If tau < kt (beta_min + eps), every
// g_k = 1 + tau / (beta_k + eps) lies in [1, 1 + kt), so
// chi_k = g_k^6 / sum_j g_j^6 >= 1 / (3 (1 + kt)^6).  With
// 1 + kt = 0.9 (3 C_T)^(-1/6) that bound is C_T / 0.9^6 = 1.88 C_T: every
// stencil is kept, and the divisions and powers need not be evaluated.  The
// 10% margin in g (1.9x in chi) is far above the rounding of either
// precision, so the bits are exactly the ones the full evaluation gives.
// kt = 0 (the shortcut never applies) when C_T >= 1/3.  Host functions: the
// launchers evaluate kt once (in the kernels an FP64 pow per thread cost more
// than the whole scalar stage at 200 cells).
// --------------------------------------------------------------------------
inline double keep_all_factor(double CT) {
    return (CT > 0.0 && CT < 1.0 / 3.0) ? 0.9 * pow(3.0 * CT, -1.0 / 6.0) - 1.0 : 0.0;
}
inline float keep_all_factor(float CT) {
    return (CT > 0.f && CT < 1.f / 3.f) ? 0.9f * powf(3.f * CT, -1.f / 6.f) - 1.f : 0.f;
}

// Parameters of the FP64 cutoff test: epsilon, C_T and kt, and their FP32 forms
// (4 epsilon; C_T, or 0 where FP32 cannot hold it and only kept windows are
// decided there).
struct Cut64 {
    double eps, CT, kt;
    float e4, ktf, ctf;
};
T7_HD Cut64 cut64(double eps, double CT, double kt) {
    Cut64 K;
    K.eps = eps;
    K.CT = CT;
    K.kt = kt;
    K.e4 = (float)(4.0 * eps);
    K.ktf = (float)kt;
    K.ctf = CT > 1e-30 ? (float)CT : 0.f;
    return K;
}

// Five-point smoothness measure and cutoff bits (d0 | d1<<1 | d2<<2) of one
// window w0..w4 = f_{i-2} .. f_{i+2} in upwind order, in FP64 (Eqs.
// smooth_expl, tau5, TENO1 with C = 1 and q = 6, norm, seclect).
T7_HD unsigned cutoff_bits_f64(double w0, double w1, double w2, double w3, double w4, double eps, double CT,
                               double kt) {
    // Eq. smooth_expl
    double s0a = w0 - 4.0 * w1 + 3.0 * w2;
    double s0b = w0 - 2.0 * w1 + w2;
    double s2a = 3.0 * w2 - 4.0 * w3 + w4;
    double s2b = w2 - 2.0 * w3 + w4;
    double b0 = 0.25 * (s0a * s0a) + (13.0 / 12.0) * (s0b * s0b);
    double b2 = 0.25 * (s2a * s2a) + (13.0 / 12.0) * (s2b * s2b);
    // Eq. tau5, Eq. TENO1 with C = 1, q = 6 (squared, squared again, times square)
    double tau = fabs(b0 - b2);
    // every stencil kept (see keep_all_factor); beta_min >= 0, so tau < kt eps
    // already suffices and beta_1 is not needed
    if (tau < kt * eps) return 7u;
    double s1a = w1 - w3;
    double s1b = w1 - 2.0 * w2 + w3;
    double b1 = 0.25 * (s1a * s1a) + (13.0 / 12.0) * (s1b * s1b);
    if (tau < kt * (fmin(fmin(b0, b1), b2) + eps)) return 7u;
    double g0 = 1.0 + tau / (b0 + eps);
    double g1 = 1.0 + tau / (b1 + eps);
    double g2 = 1.0 + tau / (b2 + eps);
    double q0 = g0 * g0, q1 = g1 * g1, q2 = g2 * g2;
    double y0 = (q0 * q0) * q0, y1 = (q1 * q1) * q1, y2 = (q2 * q2) * q2;
    // Eqs. norm, seclect: delta = 0 iff chi < C_T
    double S = (y0 + y1) + y2;
    unsigned d0 = (y0 / S < CT) ? 0u : 1u;
    unsigned d1 = (y1 / S < CT) ? 0u : 1u;
    unsigned d2 = (y2 / S < CT) ? 0u : 1u;
    return d0 | (d1 << 1) | (d2 << 2);
}

// x = h + l + r with h the leading 24 bits of x (truncated), l the next 23 and
// |r| < 2^-46 |x|, by integer operations on x's bits and two FP32 operations.
// |x| < 2^-126 gives 0; a magnitude of 2^126 and more, infinities and NaN give
// an infinite h.
T7_HD void split_f32(double x, float &h, float &l) {
    const uint64_t b = f64_bits(x);
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
    const uint32_t a = hi & 0x7fffffffu, sign = hi & 0x80000000u;
    const uint32_t t = a - 0x38000000u;  // exponent rebiased
    uint32_t f = (t << 3) | (lo >> 29);
    if (t - 0x00100000u >= 0x0fc00000u) f = a < 0x38100000u ? 0u : 0x7f800000u;
    h = f32_of(f | sign);
    const float m = f32_of(0x4b000000u | ((lo >> 6) & 0x7fffffu)) - 8388608.f;  // bits 28..6 as an integer
    l = m * (f32_of((f & 0x7f800000u) | sign) * 1.4210854715202004e-14f);       // times 2^(e-46)
}

// The same bits as cutoff_bits_f64, decided in FP32 where its error bound
// allows it.  The window enters through its four first differences, each
// d_t = (h_{t+1} - h_t) + (l_{t+1} - l_t) within 2^-23 |d_t| + 2^-44 max|w|; the
// measures are linear in them, so each beta (times 4: s^2 + 13/3 r^2) is known
// within 2.2e-6 of itself plus A = 2^-60 max|w|^2 (1e-36 covers underflow).
//   kept     tau + 1e-5 (beta_0 + beta_2) + A < kt (0.9999 (beta_min + eps) - A)
//            implies tau < kt (beta_min + eps): all bits set (keep_all_factor).
//   decided  where tau > 0.003 (beta_0 + beta_2), A is below 1e-5 of the
//            smallest beta + eps, and the largest beta + eps below 2^125 (above
//            2^126 its reciprocal would vanish), g_k is known within 7.5e-4 and
//            chi_k / C_T within 2%: the FP32 comparison holds unless chi_k is
//            within 3% of C_T.
// Everything else, and what FP32 cannot hold, goes to the FP64 evaluation.
T7_HD unsigned cutoff_bits(double w0, double w1, double w2, double w3, double w4, const Cut64 &K) {
    float h0, h1, h2, h3, h4, l0, l1, l2, l3, l4;
    split_f32(w0, h0, l0);
    split_f32(w1, h1, l1);
    split_f32(w2, h2, l2);
    split_f32(w3, h3, l3);
    split_f32(w4, h4, l4);
    const float d1 = (h1 - h0) + (l1 - l0), d2 = (h2 - h1) + (l2 - l1);
    const float d3 = (h3 - h2) + (l3 - l2), d4 = (h4 - h3) + (l4 - l3);
    const float c = 13.f / 3.f;
    const float s0a = fmaf(3.f, d2, -d1), s0b = d2 - d1, s2a = fmaf(-3.f, d3, d4), s2b = d4 - d3;
    const float s1a = d2 + d3, s1b = d3 - d2;
    const float b0 = fmaf(c * s0b, s0b, s0a * s0a), b1 = fmaf(c * s1b, s1b, s1a * s1a);
    const float b2 = fmaf(c * s2b, s2b, s2a * s2a);
    const float W = fmaxf(fmaxf(fmaxf(fabsf(h0), fabsf(h1)), fmaxf(fabsf(h2), fabsf(h3))), fabsf(h4));
    const float A = fmaf(W * W, 8.673617379884035e-19f, 1e-36f);
    const float sum = b0 + b2, tau = fabsf(b0 - b2), bm = fminf(fminf(b0, b1), b2) + K.e4;
    if (fmaf(1e-5f, sum, tau) + A < K.ktf * fmaf(0.9999f, bm, -A)) return 7u;
    if (K.ctf > 0.f && tau > 0.003f * sum && A < 1e-5f * bm && fmaxf(fmaxf(b0, b1), b2) + K.e4 < 4e37f) {
        const float g0 = fmaf(tau, f32_rcp(b0 + K.e4), 1.f), g1 = fmaf(tau, f32_rcp(b1 + K.e4), 1.f);
        const float g2 = fmaf(tau, f32_rcp(b2 + K.e4), 1.f);
        const float gm = fmaxf(fmaxf(g0, g1), g2), rg = f32_rcp(gm);
        float x0 = g0 * rg, x1 = g1 * rg, x2 = g2 * rg;
        x0 *= x0;
        x1 *= x1;
        x2 *= x2;
        const float y0 = x0 * x0 * x0, y1 = x1 * x1 * x1, y2 = x2 * x2 * x2;
        const float thr = K.ctf * ((y0 + y1) + y2), band = 0.03f * thr;
        if (gm < 1e37f && fabsf(y0 - thr) > band && fabsf(y1 - thr) > band && fabsf(y2 - thr) > band)
            return (y0 < thr ? 0u : 1u) | ((y1 < thr ? 0u : 1u) << 1) | ((y2 < thr ? 0u : 1u) << 2);
    }
    return cutoff_bits_f64(w0, w1, w2, w3, w4, K.eps, K.CT, K.kt);
}

}  // namespace t7
