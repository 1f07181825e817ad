// k_query.cu -- one membership query in one launch: the baby-step giant-step
// search of Algorithm 1 by one block, the square-free test by the others.
//
// A query is bound by the length of its serial chain, not by throughput, so
// the block shortens every part of it:
//  * the baby walk of N steps (warp 0; about 45 clocks a step, the chain
//    rcp -> quotient -> remainder -> Q') stores each state with one shared
//    store; the 8 warps insert the states afterwards, 2N / 256 rounds;
//  * 256 lanes of giant steps let N be a quarter of what 32 lanes want;
//  * thread t holds mu_t = S^(t+1), S = reduce(a_N a_{N/2}): once the first k
//    = 1, 2, 4, .. 128 are known, threads k .. 2k - 1 take mu_{t-k} S^k, and a
//    hit among them ends the search; after 256, rounds of mu_t S^256.
// All products are nuc_mul (eis_nuc.cuh) in one out-of-line copy (the kernel
// runs once, so its instructions come from L2).
//
// Coverage.  The table holds the window [R - delta_N, R + delta_N] whole
// (every state, and its mirror).  S is shorter than the window by
// delta_N - delta_{N/2}, at least N/4 pairs of steps of log 2 or more each;
// two neighbouring powers differ by S up to the offsets of the (at most 8)
// products they do not share, each below log 2 sqrt d, and their few steps to
// a norm without small factors.
//
// Measured, a call with its launch: 39 us against 161 us for d below 10^12, 58
// against 290 below 2^44 (one warp, table and giant steps alike); 75 and 102
// with the textbook product, whose 1100 serial instructions are 5 us; 43 and 60
// with two scans over the lanes (10 products deep) instead of the doubling (9,
// and 6 to 8 when a hit comes early).
#include "eis_common.cuh"
#include "eis_bsgs.cuh"
#include "eis_infra.cuh"
#include "eis_kernels.h"
#include "eis_nuc.cuh"

namespace eis {

namespace {

// Ideals as (a, b, class, w = (b^2 - d)/(4a)): reduce(X * Y), moved on to a
// norm without small factors; a = 0 when a factor has failed or a reduction
// runs away.  Where the norms share a factor X steps on and tries again, and
// after kQTries the textbook product takes the pair as it is.
constexpr int kQTries = 6;
__device__ __noinline__ int4 query_mul(int4 X, int4 Y, int64_t d, int32_t s, int32_t L) {
    if (!X.x || !Y.x) return make_int4(0, 0, 0, 0);
    NucIdeal x{X.x, X.y, X.z, X.w}, out{1, 1, 0, 0};
    const NucIdeal y{Y.x, Y.y, Y.z, Y.w};
    int st = kNucRetry;
    for (int t = 0; t < kQTries && st != kNucOk; ++t) {
        if (t) x = nuc_step(x, s);
        st = nuc_mul(x, y, s, L, out);
    }
    if (st != kNucOk) {
        Ideal o{1, 1, 0};
        int64_t Qm = 2;
        if (!lean_mul(Ideal{X.x, X.y, X.z}, Ideal{Y.x, Y.y, Y.z}, Y.w, d, s, o, Qm))
            return make_int4(0, 0, 0, 0);
        out = NucIdeal{(int32_t)o.a, (int32_t)o.b, o.g, (int32_t)(-Qm / 2)};
    }
    int steps = 0;
    out = nuc_coprime(out, s, 16, steps);
    return make_int4(out.a, out.b, out.g, out.w);
}

__device__ __forceinline__ int4 shfl4(int4 v, int src) {
    return make_int4(__shfl_sync(kFull, v.x, src), __shfl_sync(kFull, v.y, src),
                     __shfl_sync(kFull, v.z, src), __shfl_sync(kFull, v.w, src));
}

// Steps per centre test of the baby walk.
constexpr int kQGroup = 16;

// States 1 .. N+1 into st[] as (Q, num, S) (warp 0, every lane alike).
// Returns true with g = log eps_d when the centre comes within N steps.
template <bool kFast>
__device__ __forceinline__ bool query_walk(uint64_t d, int N, float4 *st, int lane, int &g, int &steps) {
    LeanState w;
    float C;
    steps = 0;
    if (lean_init<kFast>(d, w, C, g)) return true;
    if (lane == 0) {
        st[0] = make_float4(2.0f, 0.0f, 0.0f, 0.0f);
        st[1] = make_float4(w.Q, w.num, __int_as_float(w.acc), 0.0f);
    }
    for (int j = 1; j <= N; j += kQGroup) {
        const LeanState w0 = w;
        bool any = false;
#pragma unroll
        for (int i = 0; i < kQGroup; ++i) {
            any |= lean_step<kFast>(w, C);
            w.acc += w.x;
            // S_{j+1+i} = acc + steps (the 1 per step apart)
            if (lane == 0) st[j + 1 + i] = make_float4(w.Q, w.num, __int_as_float(w.acc + j + i), 0.0f);
        }
        if (any) {
            w = w0;
            for (int i = 0; i < kQGroup; ++i) {
                ++steps;
                const bool c = lean_step<kFast>(w, C);
                w.acc += w.x;
                if (c) break;
            }
            g = lean_finish(w, (uint32_t)steps);
            return true;
        }
        steps += kQGroup;
    }
    return false;
}

}  // namespace

// Block 0 searches; the others test d for square factors against the first
// nprimes primes of the table.  out is host memory mapped into the device,
// zeroed by the host before the launch.  N a multiple of 32; the table has
// 2^log2n >= 4N slots.
__global__ void __launch_bounds__(kQueryThreads) k_query(uint64_t d, const uint64_t *__restrict__ sqtab,
                                                         uint32_t nprimes, volatile QueryOut *out, int N,
                                                         int log2n, uint32_t max_rounds) {
    if (blockIdx.x > 0) {
        bool hit = false;
        for (uint32_t i = (blockIdx.x - 1) * blockDim.x + threadIdx.x; i < nprimes;
             i += (gridDim.x - 1) * blockDim.x)
            hit |= d * sqtab[2 * i] <= sqtab[2 * i + 1];
        if (hit) out->square = 1;
        return;
    }
    extern __shared__ uint64_t smem_q[];
    uint64_t *tab = smem_q;
    float4 *st = reinterpret_cast<float4 *>(smem_q + ((size_t)1 << log2n));  // N + 2 states
    __shared__ int sh_done, sh_g, sh_steps, sh_ok, sh_best[2];
    __shared__ int4 sh_mu[kQueryThreads];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool fast = d < kFastDLimit;
    if (warp == 0) {
        int g = 0, steps = 0;
        const bool done = fast ? query_walk<true>(d, N, st, lane, g, steps)
                               : query_walk<false>(d, N, st, lane, g, steps);
        if (lane == 0) {
            sh_done = done;
            sh_g = g;
            sh_steps = steps;
            sh_ok = 1;
            sh_best[0] = sh_best[1] = 0x7fffffff;
        }
    } else {
        for (uint32_t i = tid - 32; i < (1u << log2n); i += kQueryThreads - 32) tab[i] = 0;
    }
    __syncthreads();
    if (sh_done) {
        if (tid == 0) {
            out->baby = 1 + (uint32_t)sh_steps;
            out->result = 1 + sh_g;
        }
        return;
    }
    const int32_t s = (int32_t)isqrt44(d), L = (int32_t)isqrt44((uint64_t)s);
    // ---- the table: O_K again as (2, P_1), each state and its mirror
    bool ok = true;
    for (int j = 1 + tid; j <= N; j += kQueryThreads) {
        const float4 x = st[j];
        const int64_t Q = (int64_t)x.x, P = (int64_t)x.y - s;  // num = P + s (+ 1/2)
        const int64_t Pn = (int64_t)st[j + 1].y - s;
        const int S = (int)((uint32_t)__float_as_int(x.z) % 3u);
        if (j == 1) ok &= infra_insert_cas(tab, log2n, infra_key(2, P), 0, 0);
        ok &= infra_insert_cas(tab, log2n, infra_key(Q, P), 0, S);
        ok &= infra_insert_cas(tab, log2n, infra_key(Q, Pn), kMirror, S);
    }
    if (!ok) sh_ok = 0;
    __syncthreads();
    // ---- powers of S: mu_t of thread t, doubled level by level, each looked up
    // as it is made.  best: the first hit (-1: a product failed); two words in
    // turn, so that a level or round that goes on leaves its word as it was.
    auto state = [&](int j) {
        const float4 x = st[j];
        return make_int4((int)x.x / 2, (int)x.y - s, (int)((uint32_t)__float_as_int(x.z) % 3u),
                         -(int)st[j - 1].x / 2);
    };
    int4 mu = make_int4(0, 0, 0, 0);
    uint64_t e = 0;
    auto look = [&](int word) {
        e = mu.x ? infra_find(tab, log2n, infra_key(2 * (int64_t)mu.x, mu.y)) : 0;
        if (!mu.x)
            atomicMin(&sh_best[word], -1);
        else if (e)
            atomicMin(&sh_best[word], tid);
    };
    auto finish = [&](int best, uint32_t giants) {  // by every thread: best is decided
        if (tid == max(best, 0)) {
            const int Sj = (int)(e & 3);
            out->baby = 1 + (uint32_t)sh_steps;
            out->giant = giants;
            out->result = best < 0 ? -1 : 1 + ((e & 4) ? (mu.z + Sj) % 3 : (mu.z + 3 - Sj) % 3);
        }
    };
    if (warp == 0) {
        // the first 32 in one warp, by shuffles
        if (lane == 0) mu = query_mul(state(N), state(N / 2), (int64_t)d, s, L);
        __syncwarp();
#pragma unroll 1
        for (int k = 1; k < 32; k <<= 1) {
            const int4 o = shfl4(mu, lane & (k - 1)), P = shfl4(mu, k - 1);
            if (lane >= k && lane < 2 * k) mu = query_mul(o, P, (int64_t)d, s, L);
        }
        look(0);
        sh_mu[lane] = mu;
    }
    __syncthreads();
    if (sh_best[0] < kQueryThreads || !sh_ok) {
        finish(sh_ok ? sh_best[0] : -1, 6u + (uint32_t)tid);
        return;
    }
    int word = 1;
#pragma unroll 1
    for (int k = 32; k < kQueryThreads; k <<= 1) {
        if (tid >= k && tid < 2 * k) {
            mu = query_mul(sh_mu[tid - k], sh_mu[k - 1], (int64_t)d, s, L);
            look(word);
            sh_mu[tid] = mu;
        }
        __syncthreads();
        const int best = sh_best[word];
        if (best < kQueryThreads) {
            finish(best, 6u + (uint32_t)tid);
            return;
        }
        word ^= 1;
    }
    const int4 stride = sh_mu[kQueryThreads - 1];
    for (uint32_t r = 1; r < max_rounds; ++r) {
        mu = query_mul(mu, stride, (int64_t)d, s, L);
        look(word);
        __syncthreads();
        const int best = sh_best[word];
        if (best < kQueryThreads) {
            finish(best, 6u + kQueryThreads * r + (uint32_t)tid);
            return;
        }
        word ^= 1;
    }
    if (tid == 0) out->result = -1;  // no hit within max_rounds
}

}  // namespace eis
