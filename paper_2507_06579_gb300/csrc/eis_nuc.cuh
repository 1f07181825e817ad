// eis_nuc.cuh -- the ideal product of the giant steps: NUCOMP's partial
// reduction with nearest-integer Euclid runs in fp32 and everything else in
// 32 bits, for two reduced ideals of a discriminant d < 2^44.
//
// The forms (u, v, w) = (a, -b, (b^2 - d)/(4a)) of two reduced ideals have
// every coefficient below sqrt d < 2^22.  With F = gcd(u1, u2) = 1,
// beta u2 == 1 (mod u1), sigma = (v1 + v2)/2 and m = v2 - sigma, the product
// is the class of (u1 u2, ..), and NUCOMP (Shanks; Algorithm 2 of the paper)
// reaches a nearly reduced form of it from the remainders (p0, p1) of u1 by
// r = m beta mod u1 that bracket L = sqrt(sqrt d) and their cofactors
// (c0, c1), p0 c1 - p1 c0 = u1:
//   c(p, c) = (u2 p - m c)/u1,  d(p, c) = (sigma p - w2 c)/u1   (exact),
//   u3 = p0 c(p0,c0) - c0 d(p0,c0),  w3 = p1 c(p1,c1) - c1 d(p1,c1),
//   v3 = 2 c0 d(p1,c1) + sigma - 2 p0 c(p1,c1) - m.
// (The paper's listing divides by x and b_x for the second pair; both are the
// same linear map, because p0 c1 - p1 c0 = u1.)  The relation holds for any
// unimodular chain, so the Euclid runs take nearest-integer quotients:
//   * a quotient is one reciprocal, one FMA onto 1.5 2^23 and one subtraction,
//     with no correction: a quotient that is off by one, possible next to a
//     half-integer, still leaves a remainder below the divisor;
//   * every remainder and cofactor is an integer below 2^23 in magnitude
//     (|c_{i+1}| <= 2 u1 / |r_i|), so each FMA is exact;
//   * about 0.7 of the steps of the floor Euclid.
// The exact quotients by u1 are rounded from an fp32 estimate and corrected
// by the 32-bit remainder (the estimate is within a few units: every quotient
// is below 2^23 and each term carries a relative error of 2^-22).
// u3, v3 and the class's A, B, C are formed mod 2^32, which is enough: |u3|
// is below 2^26 (|p0| <= L, |c0| <= 2 u1/L, u2 <= u1), |v3| below 2^31, and the
// class needs the trailing zeros of C = 2 u3 alone.  A quotient of the last
// reduction that is off by one is another valid step: (P, Q) stays an ideal of
// the class, with the same rule for its generator.
//
// Measured against the textbook product: k_bsgs.cu (throughput) and k_query.cu
// (latency).
#pragma once

#include "eis_bsgs.cuh"

namespace eis {

// An ideal [a, (b + sqrt d)/2] with its class and w = (b^2 - d)/(4a).
struct NucIdeal {
    int32_t a, b, g, w;
};

EIS_HD float nuc_rcp(float x) {
#ifdef __CUDA_ARCH__
    return rcp_approx(x);
#else
    return 1.0f / x;
#endif
}

// x / y rounded to an integer (|x/y| < 2^22), y's reciprocal estimated: off
// by one at most next to half-integers.
EIS_HD float nuc_quot(float x, float y) {
#ifdef __CUDA_ARCH__
    return __fsub_rn(__fmaf_rn(x, rcp_approx(y), 12582912.0f), 12582912.0f);
#else
    return std::fma(x, 1.0f / y, 12582912.0f) - 12582912.0f;
#endif
}

EIS_HD float nuc_fma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return std::fma(a, b, c);
#endif
}

EIS_HD int32_t nuc_int(float v) {
#ifdef __CUDA_ARCH__
    return __float2int_rn(v);
#else
    return (int32_t)std::lrintf(v);
#endif
}

// gcd(u1, u2) (u1 >= u2 > 0) and beta with beta u2 == gcd (mod u1),
// |beta| < 2 u1.
EIS_HD float nuc_gcd(float u1, float u2, float &beta) {
    float r0 = u1, r1 = u2, t0 = 0.0f, t1 = 1.0f;
    for (;;) {
        float q = nuc_quot(r0, r1);
        r0 = nuc_fma(-q, r1, r0);
        t0 = nuc_fma(-q, t1, t0);
        if (r0 == 0.0f) {
            beta = r1 < 0.0f ? -t1 : t1;
            return fabsf(r1);
        }
        q = nuc_quot(r1, r0);
        r1 = nuc_fma(-q, r0, r1);
        t1 = nuc_fma(-q, t0, t1);
        if (r1 == 0.0f) {
            beta = r0 < 0.0f ? -t0 : t0;
            return fabsf(r0);
        }
    }
}

// x y - k m for the k nearest x y / m: the residue of x y mod m in
// (-1.2 m, 1.2 m), |x|, |y| < 2^23, 0 < m < 2^22, |x y / m| < 2^23.
EIS_HD int32_t nuc_mulmod(int32_t x, int32_t y, int32_t m, float rm) {
    const int32_t q = nuc_int((float)x * (float)y * rm);
    return (int32_t)((uint32_t)x * (uint32_t)y - (uint32_t)q * (uint32_t)m);
}

// (x p - y c) / m exactly (m divides it), the quotient below 2^24.
EIS_HD int32_t nuc_exact(int32_t x, int32_t p, int32_t y, int32_t c, int32_t m, float rm) {
    const int32_t q = nuc_int(nuc_fma((float)x, (float)p, -(float)y * (float)c) * rm);
    const int32_t r = (int32_t)((uint32_t)x * (uint32_t)p - (uint32_t)y * (uint32_t)c -
                                (uint32_t)q * (uint32_t)m);
    return q + nuc_int((float)r * rm);
}

// floor(x / y), |x|, |y| < 2^28, y != 0, |x / y| < 2^22, and x - q y.
EIS_HD int32_t nuc_floordiv(int32_t x, int32_t y, int32_t &rem) {
    int32_t q = nuc_int(floorf((float)x * nuc_rcp((float)y)));
    int32_t r = x - q * y;
    const int32_t ay = y < 0 ? -y : y;
    if ((y < 0 ? -r : r) < 0) {
        r += y;
        --q;
    } else if ((y < 0 ? -r : r) >= ay) {
        r -= y;
        ++q;
    }
    rem = r;
    return q;
}

enum { kNucOk = 0, kNucRetry = 1, kNucFail = 2 };

// reduce(X * Y).  kNucRetry: the norms have a common factor, or the
// remainders jump from above L to almost nothing (below 1 in 50): nothing is
// formed, and the caller steps X along its cycle or takes the general product.
// kNucFail: not expected.
EIS_HD int nuc_mul(const NucIdeal &X, const NucIdeal &Y, int32_t s, int32_t L, NucIdeal &out) {
    const bool sw = X.a < Y.a;
    const int32_t u1 = sw ? Y.a : X.a, u2 = sw ? X.a : Y.a;
    const int32_t v1 = -(sw ? Y.b : X.b), v2 = -(sw ? X.b : Y.b), w2 = sw ? X.w : Y.w;
    const int32_t sigma = (v1 + v2) / 2, m = v2 - sigma;
    float fb;
    const float F = nuc_gcd((float)u1, (float)u2, fb);
    if (F != 1.0f) return kNucRetry;
    const float r1 = nuc_rcp((float)u1);
    // remainders of u1 by r = m beta mod u1 down to L, with their cofactors
    float p0 = (float)u1, p1 = (float)nuc_mulmod(m, nuc_int(fb), u1, r1);
    float c0 = 0.0f, c1 = 1.0f;
    const float fL = (float)L;
    bool odd = false;
    for (;;) {
        if (!(fabsf(p0) > fL) || p1 == 0.0f) break;
        float q = nuc_quot(p0, p1);
        p0 = nuc_fma(-q, p1, p0);
        c0 = nuc_fma(-q, c1, c0);
        if (!(fabsf(p1) > fL) || p0 == 0.0f) {
            odd = true;
            break;
        }
        q = nuc_quot(p1, p0);
        p1 = nuc_fma(-q, p0, p1);
        c1 = nuc_fma(-q, c0, c1);
    }
    // p0 = the remainder at or below L, p1 the next; p0 c1 - p1 c0 = u1.  A
    // tiny p0 goes with a large c1 (|c1| <= 2 u1/|p0|), and |v3| < 4 L |c1| + 2^24
    // has to stay below 2^31.
    const int32_t by = nuc_int(odd ? -p1 : p0), bx = nuc_int(odd ? p0 : p1);
    const int32_t y = nuc_int(odd ? -c1 : c0), x = nuc_int(odd ? c0 : c1);
    if (fabsf(odd ? p1 : p0) > fL || fabsf(odd ? c0 : c1) * fL > 268435456.0f) return kNucRetry;
    const int32_t cx = nuc_exact(u2, bx, m, x, u1, r1), cy = nuc_exact(u2, by, m, y, u1, r1);
    const int32_t dx = nuc_exact(sigma, bx, w2, x, u1, r1), dy = nuc_exact(sigma, by, w2, y, u1, r1);
    const int32_t u3 = by * cy - y * dy;
    const int32_t v3 = (int32_t)(2u * ((uint32_t)y * (uint32_t)dx - (uint32_t)by * (uint32_t)cx)) + sigma - m;
    const uint32_t w3 = (uint32_t)bx * (uint32_t)cx - (uint32_t)x * (uint32_t)dx;
    // the class of gamma = (2 u3 x + v3 y + y sqrt d)/(2 u3)
    const uint32_t C2 = 2u * (uint32_t)u3;
    bool ok = u3 != 0;
    const int lg = gamma_class32(C2 * (uint32_t)x + (uint32_t)v3 * (uint32_t)y, (uint32_t)y, C2, ok);
    if (!ok) return kNucFail;
    // [|u3|, (-v3 + sqrt d)/2] with P moved into (s - Q, s], then rho steps
    int32_t Q = 2 * (u3 < 0 ? -u3 : u3);
    int32_t rem;
    const int32_t k = nuc_floordiv(s + v3, Q, rem);
    int32_t P = s - rem;
    int32_t Qm = (int32_t)((u3 > 0 ? 0u - 2u * w3 : 2u * w3) - (uint32_t)k * (uint32_t)(P - v3));
    int g = X.g + Y.g + 3 - lg;
    for (int it = 0; !(Q > 0 && P > 0 && P <= s && s - P < Q && Q <= s + P); ++it) {
        if (it >= 64) return kNucFail;
        // Q > 0: q = floor((P + s)/Q); Q < 0: floor((P + s + 1)/Q)
        const int32_t q = nuc_floordiv(P + s + (Q < 0), Q, rem);
        const int32_t Pn = q * Q - P;
        const int32_t Qn = Qm + q * (P - Pn);
        g += 1 + ((Pn >> 1) & 1);
        Qm = Q;
        P = Pn;
        Q = Qn;
    }
    out.a = Q >> 1;
    out.b = P;
    out.g = g % 3;
    out.w = -(Qm >> 1);
    return kNucOk;
}

// w = (b^2 - d)/(4a) of a reduced ideal, by exact division mod 2^32 (a is odd,
// |w| < 2^22): the inverse of a by Newton iteration.
EIS_HD int32_t nuc_w(int32_t a, int32_t b, int64_t d) {
    const uint32_t n = (uint32_t)(((int64_t)b * b - d) >> 2), ua = (uint32_t)a;
    uint32_t x = ua;  // a a == 1 (mod 8)
    for (int i = 0; i < 4; ++i) x *= 2u - ua * x;
    return (int32_t)(n * x);
}

// One baby step of a reduced ideal.
EIS_HD NucIdeal nuc_step(const NucIdeal &X, int32_t s) {
    const int32_t Q = 2 * X.a, P = X.b;
    int32_t rem;
    const int32_t q = nuc_floordiv(P + s, Q, rem);
    const int32_t Pn = q * Q - P;
    NucIdeal o;
    o.a = (-2 * X.w + q * (P - Pn)) >> 1;
    o.b = Pn;
    o.g = (X.g + 1 + ((Pn >> 1) & 1)) % 3;
    o.w = -X.a;
    return o;
}

// The first state from X on whose norm no prime up to 13 divides (at most `most`
// steps on, counted in `steps`): its products meet a common factor 1 time in 70,
// against 1 in 5.
EIS_HD NucIdeal nuc_coprime(NucIdeal X, int32_t s, int most, int &steps) {
    for (int i = 0; i < most; ++i) {
        const uint32_t a = (uint32_t)X.a;
        if (a % 3 && a % 5 && a % 7 && a % 11 && a % 13) break;
        X = nuc_step(X, s);
        ++steps;
    }
    return X;
}

// The lane search's wide stride: M = reduce(x J), x the first state from G on
// whose norm has no factor in common with J's (few d need more than two steps;
// one without the wide stride would take twice the giant steps), and Y the first
// from M on without small factors.  At most kStrideSteps steps in all (`steps`):
// they come out of the window's margin (eis_bsgs.cuh).  False: no product.
EIS_HD bool nuc_stride(const NucIdeal &G, const NucIdeal &J, int32_t s, int32_t L, NucIdeal &M,
                       NucIdeal &Y, int &steps) {
    NucIdeal x = G;
    int st = kNucRetry;
    for (steps = 0; steps < kStrideSteps; ++steps) {
        if (steps) x = nuc_step(x, s);
        st = nuc_mul(x, J, s, L, M);
        if (st != kNucRetry) break;
    }
    if (st != kNucOk) return false;
    Y = nuc_coprime(M, s, kStrideSteps - steps, steps);
    return true;
}

}  // namespace eis
