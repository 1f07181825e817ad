// eis_cubic.cuh -- cubic forms that decide most d of a range without their
// unit, shared by the kernel and the host model of the tests.
//
// Class field theory.  For d == 5 (mod 8) square-free, O = Z[sqrt d] has
// index 2 in O_K and #Cl(O) = 3 #Cl(O_K) iff d is in E, else they are equal
// (Lemma 1.1(iv)).  The index-3 subgroups of Cl(O) correspond to the cubic
// fields of discriminant d f^2 with f | 2 (Hasse; the dihedral extensions of
// ring class fields of conductor 1 and 2), those of Cl(O_K) to the fields of
// discriminant d.  Hence
//   a cubic field of discriminant 4d exists                 =>  d in E
//     (Cl(O) has more index-3 subgroups than Cl(O_K); Prop. 2.1);
//   none of discriminant 4d and none of discriminant d      =>  d not in E
//     (3 does not divide #Cl(O));
//   one of discriminant d, none of discriminant 4d          =>  undecided:
//     the walk or the search finds eps_d mod 2O_K as for any d.
//
// Forms.  Cubic rings up to isomorphism are the GL2(Z)-classes of integral
// binary cubic forms (a, b, c, e) = a x^3 + b x^2 y + c x y^2 + e y^3 with
// the same discriminant (Delone and Faddeev).  For square-free d == 5 (mod 8):
//   kind 1 (fields of discriminant d): a ring of discriminant d is maximal;
//     2 splits in it as a linear times a quadratic place, so the form is a
//     line times the irreducible quadratic mod 2:
//     (a, b, c, e) == (1,1,1,0), (0,1,1,1) or (1,0,0,1) mod 2.
//   kind 0 (fields of discriminant 4d): 2 is totally ramified, so the form
//     is the cube of a line mod 2 and does not vanish mod 4 on that line:
//     a odd, b and c even, e == 2 (mod 4);  a == 2 (mod 4), b and c even, e odd;
//     all odd, a + b + c + e == 2 (mod 4).  Conversely a form of discriminant
//     4d of this shape is maximal at 2 (and at every odd p, as p^2 does not
//     divide 4d), so it is a field: Q x K' would need disc K' = 4d, and
//     d == 1 (mod 4).
// A form of kind 1 may belong to Z x O_K; that class has one reduced form up
// to signs and translations, (0, 1, 1, (1-d)/4), so a reduced form with
// a >= 1 is a field.
//
// Reduction.  The Hessian (P, Q, R) = (b^2 - 3ac, bc - 9ae, c^2 - 3be) has
// 4PR - Q^2 = 3 disc; a form is reduced when |Q| <= P <= R.  Every class has a
// reduced form with a >= 0 and b >= 0 (signs of x and y).  With disc <= X:
// P <= sqrt X, a <= 2 X^(1/4) / sqrt 27, b < (2/sqrt 3) X^(1/4) (the maximum
// over a of 3a/2 + sqrt(sqrt X - 27 a^2/4)); Belabas, "A fast algorithm to
// compute cubic fields", 1997, has these bounds.
//
// Windows.  For given (a, b, c) and q = Q/P,
//   9a disc + 4c P^2 = P^2 h(q),   h(q) = 4b q - 3a q^2,   -1 <= q <= 1,
// so a window of discriminants is at most two bands of q, one on each side of
// the maximum q* = 2b/(3a) of h.  For given (a, b) the P that meet the window
// lie between the roots of P - kappa/P^2 = g, kappa = 27 a^2 disc / 4, at
// g = (b - 3a/2)^2 or 0 (the largest h) and g = (b + 3a/2)^2 (the least).
// Bands and roots are found in fp32 and widened past its error; each form
// found is then tested exactly, in integers.
#pragma once

#include <cmath>
#include <cstdint>

#include "eis_bsgs.cuh"

namespace eis {

constexpr int kCubicBlock = 8;  // values of b a unit of work holds (at most 16)

// One enumeration: the forms of kind `kind` whose d lies among the ncand
// candidates from d0 on.
struct CubicJob {
    uint64_t d0;      // first candidate
    uint64_t ncand;
    uint64_t bit0;    // its bit in the target bitmap
    uint32_t kind;    // 0: discriminant 4d, 1: discriminant d
    uint32_t amax;    // a = 1 .. amax
    uint32_t nblk;    // blocks of kCubicBlock b's: b < nblk * kCubicBlock
    uint32_t unit0;   // first unit of the job in the launch's numbering
    uint32_t slices;  // slices of a unit at a = 1
    uint32_t pad;
};

// Slices a unit (a; 8 b's) is cut into, of s1 at a = 1: the forms of a window
// thin out like 1/a^2, and a slice takes every S-th of 32 forms (but looks at
// every c, so that narrow windows have s1 = 1).
EIS_HD uint32_t cubic_slices(uint32_t a, uint32_t s1) { return a * a < s1 ? s1 / (a * a) : 1u; }

// Units of a's below `a` (per block of b's): sum of cubic_slices (s1 <= 64).
EIS_HD uint32_t cubic_slices_below(uint32_t a, uint32_t s1) {
    uint32_t n = a > 8 ? a - 8 : 0u;
    const uint32_t m = a < 8 ? a : 8u;
    for (uint32_t i = 1; i < m; ++i) n += cubic_slices(i, s1);
    return n;
}

EIS_HD float cubic_rcp(float x) {
#ifdef __CUDA_ARCH__
    return rcp_approx(x);
#else
    return 1.0f / x;
#endif
}

// sqrt to a relative error below 2^-21.
EIS_HD float cubic_sqrt(float x) {
#ifdef __CUDA_ARCH__
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return std::sqrt(x);
#endif
}

// 1.5 2^23 + x y rounded to an integer, |x y| < 2^22: its low bits are the
// integer's.
EIS_HD float cubic_rint(float x, float y) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(x, y, 12582912.0f);
#else
    return std::fma(x, y, 12582912.0f);
#endif
}

EIS_HD float cubic_fma(float x, float y, float z) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(x, y, z);
#else
    return std::fma(x, y, z);
#endif
}

EIS_HD int32_t cubic_ceil(float x) {
#ifdef __CUDA_ARCH__
    return __float2int_ru(x);
#else
    return (int32_t)std::ceil(x);
#endif
}

EIS_HD int32_t cubic_floor(float x) {
#ifdef __CUDA_ARCH__
    return __float2int_rd(x);
#else
    return (int32_t)std::floor(x);
#endif
}

// The root P > g of P - kappa/P^2 = g (g >= 0, kappa > 0) to a relative error
// below 4e-6: Newton on P^2 (P - g) - kappa from above (convex there, so
// every iterate stays above the root up to rounding).
EIS_HD float cubic_root(float g, float kappa) {
    float P = g + 1.01f * exp2f(log2f(kappa) * (1.0f / 3.0f));
    for (int i = 0; i < 7; ++i)
        P -= (P * P * (P - g) - kappa) * cubic_rcp(P * (3.0f * P - 2.0f * g));
    return P;
}

// floor(x / m) and the remainder for |x| < 2^24, 3 <= m < 2^15; rm = 1/m rounded.
// x is exact in fp32 and x rm errs by 2^-23 |x/m| < 1, so one correction each way.
EIS_HD int32_t cubic_floordiv(int32_t x, int32_t m, float rm, int32_t &rem) {
    int32_t q = (int32_t)floorf((float)x * rm);
    int32_t r = x - q * m;
    if (r < 0) {
        r += m;
        --q;
    }
    if (r >= m) {
        r -= m;
        ++q;
    }
    rem = r;
    return q;
}

// Constants of a job for one a.
struct CubicA {
    int32_t a, kind;
    float K0h, K0l;   // 9a disc at the window's least end, in two floats
    float dK;         // ... and what it grows by to the other, and by 10^-6 more: past the
                      // error of dK / P^2 (2^-22), whole candidates of a wide window
    float k0, k1;     // 27 a^2 disc / 4 there
    float pmax;       // sqrt of the largest discriminant, widened
    float r9a, r3a;   // 1/(9a), 1/(3a)
};

EIS_HD CubicA cubic_a(const CubicJob &j, int32_t a) {
    CubicA A;
    const int64_t m = j.kind ? 1 : 4;
    const int64_t D0 = m * (int64_t)j.d0, D1 = m * (int64_t)(j.d0 + 8 * (j.ncand - 1));
    A.a = a;
    A.kind = (int32_t)j.kind;
    const int64_t K0 = 9 * a * D0, K1 = 9 * a * D1;  // < 9 * 1115 * 2^46
    A.K0h = (float)K0;
    A.K0l = (float)(K0 - (int64_t)A.K0h);
    A.dK = (float)(K1 - K0) * 1.000001f;
    const float s = 0.75f * (float)a;
    A.k0 = s * A.K0h;
    A.k1 = s * (float)K1;
    A.pmax = cubic_sqrt((float)D1) * 1.000001f + 1.0f;
    A.r9a = 1.0f / (9.0f * (float)a);
    A.r3a = 1.0f / (3.0f * (float)a);
    return A;
}

// Whether (a, b) can start a form of the kind at all (parities).
EIS_HD bool cubic_pair_ok(int kind, int32_t a, int32_t b) {
    if (a & 1) return true;
    return kind ? (b & 1) != 0 : ((b & 1) == 0 && (a & 2) != 0);
}

// The end of the P range for (a, b): its least P (hi = 0) or largest (hi = 1),
// widened past the root's error.
EIS_HD float cubic_p_end(const CubicA &A, int32_t b, int hi) {
    const float fb = (float)b, fa = 1.5f * (float)A.a;
    float g;
    if (hi) {
        g = (fb + fa) * (fb + fa);
    } else {
        g = fb > fa ? (fb - fa) * (fb - fa) : 0.0f;
    }
    const float P = cubic_root(g, hi ? A.k1 : A.k0);
    if (hi) return fminf(P * 1.000006f + 1.0f, A.pmax);
    return P * 0.999994f - 1.0f;
}

// The c of (a, b): c = c_first + 2 i for 0 <= i < return value (c == b mod 2,
// P = b^2 - 3ac from plo to phi).
EIS_HD int32_t cubic_c_range(const CubicA &A, int32_t b, float plo, float phi, int32_t &c_first) {
    if (!(plo <= phi)) return 0;
    const int32_t lo = plo > 1.0f ? (int32_t)plo : 1, hi = (int32_t)phi;
    int32_t rem;
    int32_t c0 = cubic_floordiv(b * b - hi, 3 * A.a, A.r3a, rem);  // floor; one low at most
    c0 += (c0 ^ b) & 1;
    if (rem && ((c0 ^ b) & 1)) ++c0;
    const int32_t c1 = cubic_floordiv(b * b - lo, 3 * A.a, A.r3a, rem);
    c_first = c0;
    return c1 >= c0 ? (c1 - c0) / 2 + 1 : 0;
}

// The forms of one (a, b, c): Q = rho + 9a k.  Two bands of k,
// k = k[i] + (t << cubic_shift) for 0 <= t < n[i].
struct CubicBands {
    int32_t k[2], n[2];
};

// log2 of the step of k between forms of the kind: 1, or 2 where e is fixed
// mod 4.
EIS_HD int32_t cubic_shift(int kind, int32_t a) { return (!kind && (a & 1)) ? 2 : 1; }

// bc = 9a e0 + rho with rho small, e = e0 - k: rho, and the roundings that
// make up e0 = b cq + q2 (as cubic_rint's floats).
EIS_HD float cubic_rho(const CubicA &A, float fb, float fc, float &cq, float &q2) {
    const float m9a = 9.0f * (float)A.a;
    cq = cubic_rint(fc, A.r9a);
    const float bc0 = fb * cubic_fma(-m9a, cq - 12582912.0f, fc);  // exact, below 2^24
    q2 = cubic_rint(bc0, A.r9a);
    return cubic_fma(-m9a, q2 - 12582912.0f, bc0);
}

// Forms of a band qlo <= q <= qhi: its first k and their number.
EIS_HD void cubic_one_band(const CubicA &A, float qlo, float qhi, float P, float mlo, float mhi,
                           uint32_t kres, int32_t sh, int32_t &k0, int32_t &n) {
    const int32_t lo = cubic_ceil((fmaxf(qlo, -1.0f) * P - mlo) * A.r9a);
    const int32_t hi = cubic_floor((fminf(qhi, 1.0f) * P + mhi) * A.r9a);
    k0 = lo + (int32_t)((kres - (uint32_t)lo) & ((1u << sh) - 1u));
    n = hi >= k0 ? ((hi - k0) >> sh) + 1 : 0;
}

// Everything here is fp32: b, c and P are integers below 2^24, and
// n = 4c + 9a disc / P^2, which cancels, is formed from 9a disc and P^2 in two
// floats each, one step of Newton on the quotient.
EIS_HD CubicBands cubic_bands(const CubicA &A, int32_t b, int32_t c) {
    CubicBands B;
    B.n[0] = B.n[1] = B.k[0] = B.k[1] = 0;
    const int32_t a = A.a;
    const float fb1 = (float)b, fc = (float)c, fa = 3.0f * (float)a;
    const float P = cubic_fma(-fa, fc, fb1 * fb1);  // >= 1 (cubic_c_range)
    float cq, q2;
    const float rho = cubic_rho(A, fb1, fc, cq, q2);
    // e == er mod the step  <=>  k == e0 - er; only k's low bits count, so the bias
    // 0x4B400000 of the two roundings' bits may stay, and the product may wrap
    const int32_t sh = cubic_shift(A.kind, a);
    int32_t er;
    if (A.kind)
        er = (a & b & 1) ? 0 : 1;
    else
        er = !(a & 1) ? 1 : (b & 1) ? 2 - a - b - c : 2;
    const uint32_t kres = (uint32_t)b * float_bits(cq) + float_bits(q2) - (uint32_t)er;
    // h(q) between n0 and n1; u = sqrt(4b^2 - 3a n) at either end, on the side
    // that widens n / (2b + u)
    const float ph = P * P, pl = cubic_fma(P, P, -ph), rp = cubic_rcp(ph);
    const float z = A.K0h * rp;
    const float zc = (cubic_fma(-z, ph, A.K0h) + cubic_fma(-z, pl, A.K0l)) * rp;
    const float n0 = cubic_fma(4.0f, fc, z) + zc, n1 = cubic_fma(A.dK, rp, n0);
    const float fb = 2.0f * fb1, fb2 = fb * fb;
    const float t0 = cubic_fma(-fa, n0, fb2), t1 = cubic_fma(-fa, n1, fb2);
    // each end's own error: t is off by 2^-23 (4b^2 + |t|) at most.  (One error
    // for both, the larger, lost forms within 10^-6 of a wide window's least end:
    // where n < 0 the upper band takes the same roots, on the side that narrows
    // it by e / 2t, and its factors allow for that only while e <= 3e-6 t; n < 0
    // gives 4b^2 <= t.)
    const float e0 = 1e-6f * (2.0f * fb2 + fabsf(t0)), e1 = 1e-6f * (2.0f * fb2 + fabsf(t1));
    if (t0 + e0 < 0.0f) return B;  // the window lies above the largest h
    const float ua = cubic_sqrt(fmaxf(n0 >= 0.0f ? t0 + e0 : t0 - e0, 0.0f));
    const float ub = cubic_sqrt(fmaxf(n1 >= 0.0f ? t1 - e1 : t1 + e1, 0.0f));
    const float qs = fb * A.r3a;  // q*
    const float m = 1.0f + 2.5e-6f * P;
    // below q*: q = n / (2b + u)
    const float qa = n0 * cubic_rcp(fb + ua + 1e-30f);
    const float qb = t1 > e1 ? n1 * cubic_rcp(fb + ub) : qs;
    cubic_one_band(A, qa, qb, P, m + rho, m - rho, kres, sh, B.k[0], B.n[0]);
    // above q*: q = (2b + u) / (3a)
    if (qs <= 1.00001f)
        cubic_one_band(A, (fb + ub) * A.r3a * 0.999996f, (fb + ua) * A.r3a * 1.000004f, P, m + rho,
                       m - rho, kres, sh, B.k[1], B.n[1]);
    return B;
}

// The candidate (from the job's d0 on) that the form (a, b, c, e0 - k) of a
// band belongs to, or -1 when its discriminant is outside the window or the
// form is not reduced.  Exact: P, Q, R are below 2^31 for a form in or next to
// the window.
EIS_HD int64_t cubic_hit(const CubicA &A, int32_t b, int32_t c, int32_t k, uint64_t d0, uint64_t ncand) {
    const int kind = A.kind;
    const int32_t a = A.a;
    float cq, q2;
    const int32_t rho = (int32_t)cubic_rho(A, (float)b, (float)c, cq, q2);
    const int32_t e = b * ((int32_t)float_bits(cq) - 0x4B400000) + ((int32_t)float_bits(q2) - 0x4B400000) - k;
    const int32_t P = b * b - 3 * a * c, Q = rho + 9 * a * k;
    const int32_t R = (int32_t)((uint32_t)c * (uint32_t)c - 3u * (uint32_t)b * (uint32_t)e);
    if (Q > P || Q < -P || R < P) return -1;
    const int64_t D3 = 4 * (int64_t)P * R - (int64_t)Q * Q;  // 3 disc
    const int sh = kind ? 3 : 5;                             // 3 disc = 3d or 12d
    const int64_t V = D3 - (int64_t)(kind ? 3 * d0 : 12 * d0);  // 24 or 96 times the index
    if (V < 0 || (uint64_t)(V >> sh) >= 3 * ncand) return -1;
    return (int64_t)((uint32_t)(V >> sh) * 0xAAAAAAABu);     // exact division by 3
}

// Largest a and number of b blocks for discriminants up to X = D1.
inline void cubic_job_bounds(CubicJob &j) {
    const double X = (j.kind ? 1.0 : 4.0) * (double)(j.d0 + 8 * (j.ncand - 1));
    const double r = std::sqrt(std::sqrt(X));
    j.amax = (uint32_t)(2.0 * r / std::sqrt(27.0) * (1 + 1e-9)) + 1;
    const uint32_t bmax = (uint32_t)(2.0 * r / std::sqrt(3.0) * (1 + 1e-9)) + 1;
    j.nblk = bmax / kCubicBlock + 1;
    // about 0.41 (0.21) forms of kind 0 (1) a candidate, 0.6 of them at a = 1;
    // slices of at least 8192 forms
    const double forms = (j.kind ? 0.13 : 0.25) * (double)j.ncand / j.nblk;
    j.slices = (uint32_t)std::fmin(64.0, std::fmax(1.0, forms / 8192.0));
}

// Units of a job.
inline uint64_t cubic_units(const CubicJob &j) {
    return (uint64_t)j.nblk * cubic_slices_below(j.amax + 1, j.slices);
}

}  // namespace eis
