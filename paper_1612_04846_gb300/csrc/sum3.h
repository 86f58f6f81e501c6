// Sums of FP32 values with more than FP64's precision, on the FP32 pipe; for host and device code.
//
// GB300's FP64 pipe takes a warp instruction in 16 SM clocks, so FP64 additions that all warps of a kernel execute cost more
// than the FP32 products they add (a 1023^2, 8-system dot product: 4 us, and 3 us more for its 1216 x 8 block partials on one
// SM).  The FP32 products of a dot product are therefore added, eight at a time in FP32, into an unevaluated sum of three FP32
// values, with the error-free addition of Knuth (two_sum): s is the plain FP32 sum, c the FP32 sum of its rounding errors, e
// the sum of c's.  Only the additions to e round: after n additions the error is below n^3 2^-72 sum |x_i| (each of the n
// roundings is 2^-24 of an e of at most n^2 2^-48 sum |x_i|), against n 2^-53 sum |x_i| for n FP64 additions; n, the longest
// chain of additions from a product to the total, is at most a few hundred.  The same order of additions gives the same bits,
// and a.add(b) those of b.add(a).  Below the FP32 range's bottom (sums under 2^-96) words of the sum are FP32 denormals, as
// the FP32 products they come from are.
//
// Against pairs of FP32 values (48 bits, one renormalisation an addition), which this replaces, with the block partials half
// as large again and one barrier more in the one-launch solves: 1023^2, k = 7, 1870 -> 1886 us; sums over 511^2 plans 2630 ->
// 2699; variable 511^2 2437 -> 2463; sparse 63^3 3731 -> 3764; 63^2 48.0 -> 49.3; 383 x 255 335 -> 337; the results are the
// same bit for bit.  FP64 throughout: 1023^2 1958, sums 2958.
#pragma once
#include <math.h>
#include <string.h>

#ifndef BURA_HD
#ifdef __CUDACC__
#define BURA_HD __host__ __device__ __forceinline__
#else
#define BURA_HD inline
#endif
#endif

namespace bura {

// The FP32 operations, each rounded by itself (never contracted with the caller's).
BURA_HD float radd(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    return a + b;
#endif
}
BURA_HD float rmul(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}
BURA_HD float rfma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return fmaf(a, b, c);
#endif
}
BURA_HD float rdiv(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fdiv_rn(a, b);
#else
    return a / b;
#endif
}

// a + b = s + returned error, exactly
BURA_HD float two_sum_err(float a, float b, float& s) {
    const float t = radd(a, b), v = radd(t, -a);
    s = t;
    return radd(radd(a, -radd(t, -v)), radd(b, -v));
}

struct Sum3 {
    float s, c, e;
    BURA_HD void add(float x) {
        const float r = two_sum_err(s, x, s);
        e = radd(e, two_sum_err(c, r, c));
    }
    BURA_HD void add(const Sum3& o) {
        const float r = two_sum_err(s, o.s, s);
        const float q = two_sum_err(c, o.c, c);
        e = radd(radd(e, o.e), radd(q, two_sum_err(c, r, c)));
    }
    BURA_HD Sum3 negated() const { return {-s, -c, -e}; }
    // the same value with s its rounding to FP32, c that of the rest, e what is left
    BURA_HD Sum3 normal() const {
        Sum3 r;
        r.c = two_sum_err(s, c, r.s);
        r.e = two_sum_err(r.c, e, r.c);
        r.c = two_sum_err(r.s, r.c, r.s);
        r.e = two_sum_err(r.c, r.e, r.c);
        return r;
    }
    BURA_HD double value() const { return (double)s + ((double)c + (double)e); }
};

// x as such a sum, every bit of it within the FP32 range (rounded down at the range's bottom)
BURA_HD Sum3 sum3_of(double x) {
    Sum3 r{(float)x, 0.f, 0.f};
    double rest = x - (double)r.s;
    r.c = (float)rest;
    rest -= (double)r.c;
    r.e = (float)rest;
    if ((double)r.e > rest) r.e = nextafterf(r.e, -INFINITY);
    return r;
}

// a <= b, for b >= 0
BURA_HD bool sum3_le(const Sum3& a, const Sum3& b) {
    const float h = radd(a.s, -b.s);
    if (fabsf(h) > rmul(0x1p-8f, b.s)) return h < 0.f;  // (the other words are far below that)
    Sum3 d = a;
    d.add(b.negated());
    d = d.normal();
    return d.s <= 0.f;
}

// a / b rounded to FP32: long division in FP32, q0 + q1 + q2 with the remainders formed exactly (products split by a fused
// multiply-add), about 70 bits; then one rounding (q1 + q2 is first rounded to odd, so that the last addition rounds as if it
// had both).  Finite a, b != 0; their second words need not be below half a unit of the first.
BURA_HD float sum3_div(const Sum3& a, const Sum3& b) {
    const float q0 = rdiv(a.s, b.s), inv = rdiv(1.f, b.s);
    const float r0 = rfma(-q0, b.s, a.s);
    const float p = rmul(q0, b.c), pe = rfma(q0, b.c, -p);
    float v, t;
    const float w0 = two_sum_err(a.c, -p, t);
    float w = two_sum_err(r0, t, v);
    w = radd(radd(w, w0), radd(a.e, -rfma(q0, b.e, pe)));
    const float q1 = rmul(radd(v, w), inv);
    const float x = radd(rfma(-q1, b.s, v), rfma(-q1, b.c, w));
    const float q2 = rmul(x, inv);
    const float h = radd(q0, q1), m = radd(q1, -radd(h, -q0));  // (q1 is the smaller)
    float g;
    const float l = two_sum_err(m, q2, g);
    unsigned bits;
    memcpy(&bits, &g, sizeof bits);
    if (l != 0.f && (bits & 1u) == 0u) {
        bits += (l > 0.f) == (g > 0.f) ? 1u : ~0u;
        memcpy(&g, &bits, sizeof bits);
    }
    return radd(h, g);
}

// The sum of a warp's Sum3 by integer additions (one instruction for 32 lanes each, where a tree of shuffles takes five steps
// of 24): every lane's words become three limbs of 22 bits on the scale of the largest magnitude among the lanes (limb_top: its
// bits, the maximum over the lanes taken as an unsigned integer), whose sums over the lanes are exact.  Only the last limb
// rounds, at 2^-65 of the largest value.  (A 127^2 solve in one launch, 24 such sums: trees 113.0 us, limbs 113.2 with the
// words rebuilt by four additions, 2 us less with the carries in integers; 383 x 255: 403.9, 402.1, 2 us less.)
BURA_HD unsigned limb_top(const Sum3& v) {
    unsigned b[3], m = 0u;
    memcpy(b, &v, sizeof b);
    for (int i = 0; i < 3; ++i) {
        b[i] &= 0x7fffffffu;
        m = b[i] > m ? b[i] : m;
    }
    return m;
}
struct Limbs {
    unsigned top;  // exponent bits of the scale
    unsigned w[3];
};
BURA_HD float float_of(unsigned bits) {
    float f;
    memcpy(&f, &bits, sizeof f);
    return f;
}
// One lane's limbs; their sums over 32 lanes are modulo 2^32.
BURA_HD Limbs to_limbs(const Sum3& v, unsigned top) {
    const float magic = 12582912.f;  // 1.5 2^23: magic + x has the integer nearest to x in its low bits, |x| < 2^22
    const unsigned mbits = 0x4b400000u;
    Limbs l;
    l.top = top & 0x7f800000u;
    if (l.top < (30u << 23)) l.top = 30u << 23;
    const float scale = float_of(((127u + 127u + 21u) << 23) - l.top);  // the largest value: below 2^22
    const float x[3] = {rmul(v.s, scale), rmul(v.c, scale), rmul(v.e, scale)};
    float rest = 0.f;
    l.w[0] = l.w[1] = 0u;
    for (int i = 0; i < 3; ++i) {
        const float t0 = radd(x[i], magic);
        const float y = rmul(radd(x[i], -radd(t0, -magic)), 4194304.f);  // 2^22
        const float t1 = radd(y, magic);
        rest = radd(rest, radd(y, -radd(t1, -magic)));
        unsigned b;
        memcpy(&b, &t0, sizeof b);
        l.w[0] += b - mbits;
        memcpy(&b, &t1, sizeof b);
        l.w[1] += b - mbits;
    }
    const float t2 = rfma(rest, 2097152.f, magic);  // 2^21
    unsigned b;
    memcpy(&b, &t2, sizeof b);
    l.w[2] = b - mbits;
    return l;
}
// The value of limbs (a lane's, or their sums over 32 lanes), exactly: the carries go up, and the 71 bits become words of 23,
// 24 and 24 bits.
BURA_HD Sum3 from_limbs(const Limbs& l) {
    if (l.top == 0x7f800000u) return {float_of(0x7fffffffu), 0.f, 0.f};  // a value that is not finite
    const float u = float_of(l.top - (21u << 23));
    const int w2 = (int)l.w[2];
    const int w1 = (int)l.w[1] + (w2 >> 21);  // units of 2^-22, the rest below one of them
    const int w0 = (int)l.w[0] + (w1 >> 22);  // units
    const int r1 = w1 & 0x3fffff, r2 = w2 & 0x1fffff;
    return {rmul((float)(w0 & ~31), u), rmul((float)(((w0 & 31) << 19) | (r1 >> 3)) * 0x1p-19f, u),
            rmul((float)(((r1 & 7) << 21) | r2) * 0x1p-43f, u)};
}

}  // namespace bura
