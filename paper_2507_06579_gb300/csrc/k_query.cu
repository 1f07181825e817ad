// k_query.cu -- one membership query in one launch: the baby-step giant-step
// search of Algorithm 1 by one block, the square-free test by the others.
//
// A query is bound by the length of its serial chain, not by throughput, so
// the block shortens every part of it:
//  * the baby walk of N steps (warp 0; about 45 clocks a step, the chain
//    rcp -> quotient -> remainder -> Q') stores each state with one shared
//    store; the 8 warps insert the states afterwards, 2N / 256 rounds;
//  * 256 lanes of giant steps let N be a quarter of what 32 lanes want;
//  * lane t = 32 w + l holds mu = S^(t+1), S = reduce(a_N a_{N/2}): S^(l+1) by
//    a scan over the lanes (5 products deep), H = S^32, H^w by another (3),
//    and one product.  Later rounds multiply by H^8 = S^256.
// All products are nuc_mul (eis_nuc.cuh) in one out-of-line copy (the kernel
// runs once, so its instructions come from L2).
//
// Coverage.  The table holds the window [R - delta_N, R + delta_N] whole
// (every state, and its mirror).  S is shorter than the window by
// delta_N - delta_{N/2}, at least N/4 pairs of steps of log 2 or more each;
// two neighbouring powers differ by S up to the offsets of the (at most 9)
// products they do not share, each below log 2 sqrt d, and their few steps to
// a norm without small factors.
//
// Measured, a call with its launch: 43 us against 161 us for d below 10^12, 63
// against 290 below 2^44 (one warp, table and giant steps alike); 75 and 102
// with the textbook product, whose 1100 serial instructions are 5 us.
#include "eis_common.cuh"
#include "eis_bsgs.cuh"
#include "eis_infra.cuh"
#include "eis_kernels.h"
#include "eis_nuc.cuh"

namespace eis {

namespace {

constexpr int kQWarps = kQueryThreads / 32;

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
    out = nuc_coprime(out, s);
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
    // ---- S, then S^(l+1) on lane l (every warp alike)
    auto state = [&](int j) {
        const float4 x = st[j];
        return make_int4((int)x.x / 2, (int)x.y - s, (int)((uint32_t)__float_as_int(x.z) % 3u),
                         -(int)st[j - 1].x / 2);
    };
    int4 mu = query_mul(state(N), state(N / 2), (int64_t)d, s, L);
#pragma unroll 1
    for (int k = 1; k < 32; k <<= 1) {
        const int4 o = shfl4(mu, lane >= k ? lane - k : lane);
        if (lane >= k) mu = query_mul(mu, o, (int64_t)d, s, L);
    }
    auto found = [&](uint64_t e) {  // log eps_d from the table's entry at mu
        const int Sj = (int)(e & 3);
        return (e & 4) ? (mu.z + Sj) % 3 : (mu.z + 3 - Sj) % 3;
    };
    if (!__all_sync(kFull, mu.x != 0)) sh_ok = 0;
    uint64_t e = mu.x ? infra_find(tab, log2n, infra_key(2 * (int64_t)mu.x, mu.y)) : 0;
    const unsigned early = __ballot_sync(kFull, e != 0);  // the same in every warp
    __syncthreads();
    if (early || !sh_ok) {
        if (warp == 0 && lane == (early ? __ffs(early) - 1 : 0)) {
            out->baby = 1 + (uint32_t)sh_steps;
            out->giant = 6 + (uint32_t)lane;
            out->result = sh_ok ? 1 + found(e) : -1;
        }
        return;
    }
    // ---- H = S^32; lane i: H^(i+1); mu = S^(l+1) H^w, the stride H^8
    int4 h = shfl4(mu, 31);
#pragma unroll 1
    for (int k = 1; k < kQWarps; k <<= 1) {
        const int4 o = shfl4(h, lane >= k ? lane - k : lane);
        if (lane >= k && lane < kQWarps) h = query_mul(h, o, (int64_t)d, s, L);
    }
    const int4 stride = shfl4(h, kQWarps - 1);
    const int4 hw = shfl4(h, warp > 0 ? warp - 1 : 0);
    if (warp > 0) mu = query_mul(mu, hw, (int64_t)d, s, L);
    for (uint32_t r = 0; r < max_rounds; ++r) {
        // the first hit of the round; -1: a product failed.  (Two words in turn:
        // a round that goes on leaves its word as it was.)
        e = mu.x ? infra_find(tab, log2n, infra_key(2 * (int64_t)mu.x, mu.y)) : 0;
        if (!mu.x || !stride.x)
            atomicMin(&sh_best[r & 1], -1);
        else if (e)
            atomicMin(&sh_best[r & 1], tid);
        __syncthreads();
        const int best = sh_best[r & 1];
        if (best < kQueryThreads) {
            if (tid == max(best, 0)) {
                out->baby = 1 + (uint32_t)sh_steps;
                out->giant = 10 + kQueryThreads * r + (uint32_t)tid;
                out->result = best >= 0 ? 1 + found(e) : -1;
            }
            return;
        }
        mu = query_mul(mu, stride, (int64_t)d, s, L);
    }
    if (tid == 0) out->result = -1;  // no hit within max_rounds
}

}  // namespace eis
