// cubic_host.cu -- the cubic-form enumeration of eis_cubic.cuh on the host.
// stdin: lines "d0 ncand kind"; stdout: one line of '0'/'1' per candidate
// each, then the number of triples and of forms tested.
#include <cstdio>
#include <vector>

#include "eis_cubic.cuh"

using namespace eis;

int main() {
    unsigned long long d0, ncand;
    int kind;
    while (std::scanf("%llu %llu %d", &d0, &ncand, &kind) == 3) {
        CubicJob j{};
        j.d0 = d0;
        j.ncand = ncand;
        j.kind = (uint32_t)kind;
        cubic_job_bounds(j);
        std::vector<char> bits(ncand + 1, '0');
        bits[ncand] = 0;
        unsigned long long triples = 0, forms = 0, pairs = 0;
        for (int a = 1; a <= (int)j.amax; ++a) {
            const CubicA A = cubic_a(j, a);
            const int st = 1 << cubic_shift(kind, a);
            for (int b = 0; b < (int)j.nblk * kCubicBlock; ++b) {
                if (!cubic_pair_ok(kind, a, b)) continue;
                int32_t c0 = 0;
                const int32_t nc = cubic_c_range(A, b, cubic_p_end(A, b, 0), cubic_p_end(A, b, 1), c0);
                pairs += nc > 0;
                for (int32_t i = 0; i < nc; ++i) {
                    const int32_t c = c0 + 2 * i;
                    const CubicBands B = cubic_bands(A, b, c);
                    ++triples;
                    for (int w = 0; w < 2; ++w)
                        for (int32_t t = 0; t < B.n[w]; ++t) {
                            ++forms;
                            const int64_t h = cubic_hit(A, b, c, B.k[w] + st * t, d0, ncand);
                            if (h >= 0) bits[h] = '1';
                        }
                }
            }
        }
        std::printf("%s %llu %llu %llu\n", bits.data(), triples, forms, pairs);
    }
    return 0;
}
