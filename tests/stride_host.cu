// stride_host.cu -- host model of the lane search as its kernels run it
// (k_bsgs.cu): the table of marked states, nuc_stride, cycles of nuc_mul with
// steps where norms share a factor, the filter and the exact scan, look-ups of
// the first marked state of a cycle, composition from the state after it.
// stdin: lines "d N m verify"; stdout: status g cycles most_steps stride_steps
// filtered hit
//   status 0: centre in the baby walk, 1: found, 2: no search (too few marks),
//   3: a cycle past kCycleSteps; most_steps: the most steps before a product,
//   filtered: entries whose Q the filter does not hold; hit (verify): 1 when the
//   position found is l - j or l + j of the first period.
// Lines "d N m 2": stride only, from every table state as a_jl with every state
// as a_j': prints "4 pairs wide most_steps off" (off: strides with a wrong class
// or coefficient).
#include <cmath>
#include <cstdio>
#include <map>
#include <utility>
#include <vector>

#include "eis_nuc.cuh"

using namespace eis;

static int cls(int64_t P) { return 1 + (int)((P >> 1) & 1); }

struct St {
    int64_t P, Q, Qp;
};

static void step(St &w, int64_t s) {
    const int64_t q = (w.P + s) / w.Q, Pn = q * w.Q - w.P, Qn = w.Qp + q * (w.P - Pn);
    w.Qp = w.Q;
    w.Q = Qn;
    w.P = Pn;
}

struct Entry {
    int64_t Q, P;
    int S;
    int64_t j;
};

int main() {
    long long d_, N, m, verify;
    while (std::scanf("%lld %lld %lld %lld", &d_, &N, &m, &verify) == 4) {
        const int64_t d = d_;
        const int64_t s = (int64_t)isqrt44((uint64_t)d);
        const int32_t L = (int32_t)isqrt44((uint64_t)s);
        const double T = 1.39 / m * (double)s;
        const int64_t P1 = 2 * ((1 + s) / 2) - 1;
        St w{P1, (d - P1 * P1) / 2, 2};
        std::map<std::pair<int64_t, int64_t>, std::pair<int64_t, int>> pos;
        int64_t ell = 0;
        if (verify) {
            St v = w;
            int S = cls(v.P);
            for (ell = 1;; ++ell) {
                pos[{v.Q, v.P}] = {ell, S % 3};
                if (v.Q == 2) break;
                step(v, s);
                S += cls(v.P);
            }
        }
        std::vector<Entry> tab{{2, P1, 0, 0}};
        int S = cls(w.P) % 3, g = -1;
        for (int64_t j = 1; w.Q != 2; ++j) {
            if ((double)w.Q < T && (int)tab.size() < kBsgsKmax) tab.push_back({w.Q, w.P, S, j});
            if (j >= N || (int)tab.size() == kBsgsKmax) break;
            const St o = w;
            step(w, s);
            const int So = S;
            S = (S + cls(w.P)) % 3;
            if (w.Q == o.Q || w.P == o.P) {  // the centre
                g = (w.Q == o.Q ? 2 * So + cls(w.P) : 2 * So) % 3;
                break;
            }
        }
        if (w.Q == 2 && g < 0) g = S;
        if (g >= 0) {
            std::printf("0 %d 0 0 0 0 0\n", g);
            continue;
        }
        auto ideal = [&](const Entry &e) {
            return NucIdeal{(int32_t)(e.Q / 2), (int32_t)e.P, e.S, nuc_w((int32_t)(e.Q / 2), (int32_t)e.P, d)};
        };
        if (verify == 2) {
            long pairs = 0, wide = 0, most = 0, off = 0;
            for (size_t i = 1; i < tab.size(); ++i)
                for (size_t k = 1; k < i; ++k) {
                    NucIdeal M{1, 1, 0, 0}, Y{1, 1, 0, 0};
                    int steps = 0;
                    ++pairs;
                    if (!nuc_stride(ideal(tab[i]), ideal(tab[k]), (int32_t)s, L, M, Y, steps)) continue;
                    ++wide;
                    most = std::max(most, (long)steps);
                    for (const NucIdeal &x : {M, Y}) {
                        // (a class of position l is that of position 0: the first period's)
                        const auto it = pos.find({2 * (int64_t)x.a, x.b});
                        off += it == pos.end() || (int64_t)4 * x.a * x.w != (int64_t)x.b * x.b - d ||
                               (it->second.first > tab[i].j && it->second.second != x.g);
                    }
                }
            std::printf("4 %ld %ld %ld %ld\n", pairs, wide, most, off);
            continue;
        }
        const Entry ge = tab.back();
        if (ge.j < kBsgsMinJl) {
            std::printf("2 -1 0 0 0 0 0\n");
            continue;
        }
        uint32_t filter[kFilterWords] = {0};
        for (const Entry &e : tab) {
            uint32_t word, mask;
            bsgs_filter_bits(float_bits((float)e.Q), word, mask);
            filter[word] |= mask;
        }
        auto in_filter = [&](int64_t Q) {
            uint32_t word, mask;
            bsgs_filter_bits(float_bits((float)Q), word, mask);
            return (filter[word] & mask) == mask;
        };
        int filtered = 0;
        for (const Entry &e : tab) filtered += !in_filter(e.Q);
        size_t ej = tab.size() - 1;
        do --ej; while (ej > 0 && tab[ej].j + kBsgsWideGap > ge.j);
        const NucIdeal G = ideal(ge);
        NucIdeal mu = G, Y = G;
        int ssteps = 0;
        bool landed = ej > 0 && nuc_stride(G, ideal(tab[ej]), (int32_t)s, L, mu, Y, ssteps);
        if (!landed) mu = G;
        int status = -1, hit = 0, cycles = 0;
        uint32_t most = 0;
        int64_t abs_pos = ge.j, cur = ge.j;
        auto moved = [&]() {  // verify: the absolute position of mu
            const int64_t p = pos.at({2 * (int64_t)mu.a, mu.b}).first;
            abs_pos += ((p - cur) % ell + ell) % ell;
            cur = p;
        };
        if (landed && verify) moved();
        while (status < 0) {
            uint32_t steps = 0;
            while (!landed) {
                NucIdeal o{1, 1, 0, 0};
                const int st = nuc_mul(mu, Y, (int32_t)s, L, o);
                ++cycles;
                if (st == kNucOk) {
                    mu = o;
                    if (verify) moved();
                    landed = true;
                } else if (st == kNucFail || ++steps > kCycleSteps) {
                    status = st == kNucFail ? -2 : 3;
                    break;
                } else {
                    mu = nuc_step(mu, (int32_t)s);
                    if (verify) moved();
                }
            }
            if (status >= 0 || status == -2) break;
            landed = false;
            most = std::max(most, steps);
            for (;;) {  // to the first marked state
                mu = nuc_step(mu, (int32_t)s);
                if (verify) moved();
                if (2.0 * mu.a < T) break;
            }
            const NucIdeal x = mu;
            const int64_t at = abs_pos;
            mu = nuc_step(mu, (int32_t)s);
            if (verify) moved();
            if (in_filter(2 * (int64_t)x.a))
                for (const Entry &e : tab)
                    if (status < 0 && e.Q == 2 * (int64_t)x.a && (e.P == x.b || e.P == mu.b)) {
                        status = 1;
                        g = e.P == x.b ? (x.g - e.S + 3) % 3 : (x.g + e.S) % 3;
                        if (verify) hit = at == (e.P == x.b ? ell + e.j : ell - e.j) ? 1 : -1;
                    }
        }
        std::printf("%d %d %d %u %d %d %d\n", status, g, cycles, most, ssteps, filtered, hit);
    }
    return 0;
}
