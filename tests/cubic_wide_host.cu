// cubic_wide_host.cu -- forms at one place of a (wide) job, enumerated here in
// double and 128-bit integers and then looked for among the values of b, c and
// k that the library's enumeration (eis_cubic.cuh) of the whole job visits.
// stdin: lines "d0 ncand kind i0 cnt" (the place: candidates i0 .. i0 + cnt - 1
// of the job); stdout: one line each of '0'/'1' per candidate (a form was found
// here and is visited there), the number of forms and of those not visited.
#include <cmath>
#include <cstdio>
#include <vector>

#include "eis_cubic.cuh"

using namespace eis;
typedef __int128 i128;

static bool visited(const CubicJob &j, int32_t a, int32_t b, int32_t c, int32_t e, int64_t index) {
    if (a > (int32_t)j.amax || b >= (int32_t)(j.nblk * kCubicBlock)) return false;
    if (!cubic_pair_ok((int)j.kind, a, b)) return false;
    const CubicA A = cubic_a(j, a);
    int32_t c0 = 0;
    const int32_t nc = cubic_c_range(A, b, cubic_p_end(A, b, 0), cubic_p_end(A, b, 1), c0);
    if (c < c0 || (c - c0) % 2 || (c - c0) / 2 >= nc) return false;
    const CubicBands B = cubic_bands(A, b, c);
    // Q = bc - 9ae = rho + 9a k
    float cq, q2;
    const int32_t rho = (int32_t)cubic_rho(A, (float)b, (float)c, cq, q2);
    const int64_t ak = (int64_t)b * c - 9 * (int64_t)a * e - rho;
    if (ak % (9 * a)) return false;
    const int64_t k = ak / (9 * a);
    const int sh = cubic_shift((int)j.kind, a);
    bool in = false;
    for (int w = 0; w < 2; ++w)
        if (B.n[w] > 0 && k >= B.k[w] && k <= (int64_t)B.k[w] + ((int64_t)(B.n[w] - 1) << sh) &&
            ((k - B.k[w]) & ((1 << sh) - 1)) == 0)
            in = true;
    return in && cubic_hit(A, b, c, (int32_t)k, j.d0, j.ncand) == index;
}

// The shapes of the two kinds (the head of eis_cubic.cuh).
static bool shape(int kind, int64_t a, int64_t b, int64_t c, int64_t e) {
    const int A = a & 1, B = b & 1, C = c & 1, F = e & 1;
    if (kind) return (A && B && C && !F) || (!A && B && C && F) || (A && !B && !C && F);
    if (A && !B && !C) return (e & 3) == 2;
    if ((a & 3) == 2 && !B && !C) return F;
    return A && B && C && F && ((a + b + c + e) & 3) == 2;
}

int main() {
    unsigned long long d0, ncand, i0, cnt;
    int kind;
    while (std::scanf("%llu %llu %d %llu %llu", &d0, &ncand, &kind, &i0, &cnt) == 5) {
        CubicJob j{};
        j.d0 = d0;
        j.ncand = ncand;
        j.kind = (uint32_t)kind;
        cubic_job_bounds(j);
        const int64_t m = kind ? 1 : 4;
        const int64_t Da = m * (int64_t)(d0 + 8 * i0), Db = m * (int64_t)(d0 + 8 * (i0 + cnt - 1));
        const double r = std::sqrt(std::sqrt((double)Db)), sq = std::sqrt((double)Db) + 1;
        const int amax = (int)(2 * r / std::sqrt(27.0)) + 1, bmax = (int)(2 * r / std::sqrt(3.0)) + 1;
        std::vector<char> bits(cnt + 1, '0');
        bits[cnt] = 0;
        unsigned long long forms = 0, lost = 0;
        for (int a = 1; a <= amax; ++a)
            for (int b = 0; b <= bmax; ++b) {
                if (a % 2 == 0 && (kind ? b % 2 == 0 : b % 2 == 1 || a % 4 == 0)) continue;
                const double kap = 27.0 * a * a / 4, top = (b + 1.5 * a) * (b + 1.5 * a);
                const double Pmin = std::cbrt(kap * Da) - 1;
                // c downwards: P = b^2 - 3ac upwards
                for (int64_t c = (int64_t)std::floor(((double)b * b - Pmin) / (3 * a)) + 1;; --c) {
                    const int64_t P = (int64_t)b * b - 3 * (int64_t)a * c;
                    if (P < 1) continue;
                    const double fP = (double)P;
                    if (fP > sq || fP - kap * Db / (fP * fP) > top + 1) break;
                    if ((b ^ c) & 1) continue;  // c == b (mod 2) in every shape
                    // (2b - 3aq)^2 between tb and ta
                    const double ta = 4 * (fP - kap * Da / (fP * fP)), tb = 4 * (fP - kap * Db / (fP * fP));
                    if (ta < -1e-6 * fP) continue;
                    const double ua = std::sqrt(std::fmax(ta, 0.0)), ub = std::sqrt(std::fmax(tb, 0.0));
                    for (int side = -1; side <= 1; side += 2) {
                        double q0 = (2 * b + side * ua) / (3 * a), q1 = (2 * b + side * ub) / (3 * a);
                        if (q0 > q1) std::swap(q0, q1);
                        q0 = std::fmax(q0, -1.0);
                        q1 = std::fmin(q1, 1.0);
                        if (q0 > q1 + 1e-6) continue;
                        // e = (bc - qP)/(9a)
                        const int64_t e0 = (int64_t)std::ceil(((double)b * c - q1 * fP) / (9 * a) - 0.01);
                        const int64_t e1 = (int64_t)std::floor(((double)b * c - q0 * fP) / (9 * a) + 0.01);
                        for (int64_t e = e0; e <= e1; ++e) {
                            if (!shape(kind, a, b, c, e)) continue;
                            const i128 D = (i128)b * b * c * c - 4 * (i128)a * c * c * c -
                                           4 * (i128)b * b * b * e - 27 * (i128)a * a * e * e +
                                           18 * (i128)a * b * c * e;
                            if (D < Da || D > Db) continue;
                            const int64_t Q = b * c - 9 * a * e, R = c * c - 3 * b * e;
                            if (Q > P || Q < -P || R < P) continue;
                            const int64_t index = (int64_t)((D - m * (int64_t)d0) / (8 * m));
                            ++forms;
                            if (visited(j, a, b, (int32_t)c, (int32_t)e, index))
                                bits[index - i0] = '1';
                            else
                                ++lost;
                        }
                    }
                }
            }
        std::printf("%s %llu %llu\n", bits.data(), forms, lost);
    }
    return 0;
}
