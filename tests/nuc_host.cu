// nuc_host.cu -- the giant steps' product (eis_nuc.cuh) on the host.  stdin:
// lines "d a1 b1 g1 a2 b2 g2"; stdout: status a b g w of reduce(X * Y), then
// the reference NUCOMP of eis_infra.cuh: ok a b g.
#include <cmath>
#include <cstdio>

#include "eis_nuc.cuh"

using namespace eis;

int main() {
    long long d, a1, b1, g1, a2, b2, g2;
    while (std::scanf("%lld %lld %lld %lld %lld %lld %lld", &d, &a1, &b1, &g1, &a2, &b2, &g2) == 7) {
        const int64_t s = (int64_t)isqrt44((uint64_t)d), L = (int64_t)isqrt44((uint64_t)s);
        const Ideal X{a1, b1, (int)g1}, Y{a2, b2, (int)g2};
        const NucIdeal nX{(int32_t)a1, (int32_t)b1, (int32_t)g1, (int32_t)lean_cG(X, d)};
        const NucIdeal nY{(int32_t)a2, (int32_t)b2, (int32_t)g2, (int32_t)lean_cG(Y, d)};
        NucIdeal o{0, 0, 0, 0};
        const int st = nuc_mul(nX, nY, (int32_t)s, (int32_t)L, o);
        Ideal r{0, 0, 0};
        const bool ok = ideal_mul_nucomp(X, Y, d, s, L, r);
        std::printf("%d %d %d %d %d %d %lld %lld %d\n", st, o.a, o.b, o.g, o.w, ok ? 1 : 0, (long long)r.a,
                    (long long)r.b, r.g);
    }
    return 0;
}
