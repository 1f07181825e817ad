// k_sieve.cu -- candidate sieve, survivor compaction and counting kernels.
//
// Candidates are d == 5 (mod 8) (Section 1: D = { d == 5 mod 8, square-free }).
// Such d are odd, so d is square-free iff no odd prime square p^2 divides it.
// For odd p, p^2 == 1 (mod 8), hence the candidates divisible by p^2 are
// exactly d = p^2 m with m == 5 (mod 8): consecutive hits are 8 p^2 apart in
// d, p^2 apart in candidate index.  Each CTA sieves one tile of 2^16
// candidates in shared memory (8 KB bitmap) and writes it to HBM once.
#include "eis_common.cuh"
#include "eis_kernels.h"

namespace eis {

namespace {

// Odd primes whose hits the whole CTA takes, one prime after another: p^2 < 4096
// (3 .. 61), p < 1024 with primes_only; larger ones are one thread's each.
constexpr uint32_t kCoopSquares = 17, kCoopPrimes = 171;

__device__ __forceinline__ void clear_bit(uint32_t *bits, uint32_t idx) {
    atomicAnd(&bits[idx >> 5], ~(1u << (idx & 31)));
}

}  // namespace

// K1: one CTA per tile.  sqfree bit k = [candidate k is square-free];
// tile_pop[t] = number of square-free candidates of tile t.
// primes_only: bit k = [candidate k is prime] instead (prime subsequence,
// Section 3.2).  For odd q (p^2, or p with primes_only) q m == 5 (mod 8) iff
// m == 5q (mod 8) (q^2 == 1 mod 8), so the multiples q m (for primes m >= 2)
// among the candidates are q apart in candidate index.
// Every thread finds the first multiple of its own primes, the one division a
// prime takes, before the CTA strides over the small ones' hits: with every
// thread dividing for every small prime the divisions were a chain of 17 (171 for
// primes).  [1e11 - 1e9, 1e11] 66 -> 22 us, 1.25e6 candidates 15.4 -> 6.4, primes
// of 2^28 integers 432 -> 147.
__global__ void __launch_bounds__(256) k_sieve(const Tile *__restrict__ tiles,
                                               const Seg *__restrict__ segs,
                                               const uint32_t *__restrict__ primes,
                                               uint32_t nprimes, uint32_t *__restrict__ sqfree,
                                               uint32_t *__restrict__ tile_pop, int primes_only) {
    __shared__ uint32_t bits[kTileWords];
    __shared__ uint32_t first[kCoopPrimes];
    __shared__ uint32_t red[32];
    const Tile t = tiles[blockIdx.x];
    const Seg s = segs[t.seg];
    const uint64_t dfirst = s.d0 + 8 * (t.cand0 - s.cand0);
    const uint64_t dlast = dfirst + 8 * (uint64_t)(t.ncand - 1);
    const uint32_t nw = (t.ncand + 31) >> 5;
    for (uint32_t w = threadIdx.x; w < nw; w += blockDim.x) {
        const uint32_t rem = t.ncand - w * 32;
        bits[w] = rem >= 32 ? kFull : ((1u << rem) - 1);
    }
    const uint32_t ncoop = min(nprimes, primes_only ? kCoopPrimes : kCoopSquares);
    if (threadIdx.x < ncoop) first[threadIdx.x] = kFull;
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < nprimes; j += blockDim.x) {
        const uint64_t p = primes[j], p2 = p * p;
        if (p2 > dlast) break;
        const uint64_t q = primes_only ? p : p2;
        uint64_t m = (dfirst + q - 1) / q;
        if (primes_only && m < 2) m = 2;
        m += (5 * q + 8 - m % 8) % 8;
        uint64_t k = (m * q - dfirst) >> 3;
        if (j < ncoop) {
            if (k < t.ncand) first[j] = (uint32_t)k;
        } else {
            for (; k < t.ncand; k += q) clear_bit(bits, (uint32_t)k);
        }
    }
    __syncthreads();
    for (uint32_t j = 0; j < ncoop; ++j) {
        const uint32_t k0 = first[j], p = primes[j], q = primes_only ? p : p * p;
        if (k0 == kFull) continue;
        for (uint32_t k = k0 + threadIdx.x * q; k < t.ncand; k += blockDim.x * q)
            clear_bit(bits, k);
    }
    __syncthreads();
    uint32_t pop = 0;
    const uint64_t wbase = t.cand0 >> 5;
    for (uint32_t w = threadIdx.x; w < nw; w += blockDim.x) {
        const uint32_t v = bits[w];
        sqfree[wbase + w] = v;
        pop += __popc(v);
    }
    pop = block_sum(pop, red);
    if (threadIdx.x == 0) tile_pop[blockIdx.x] = pop;
}

// The larger primes, one thread per prime and interval: primes[0 .. nprimes)
// with their squares' inverses (sqtab[2i + 1] = floor((2^64 - 1) / p^2)).  Their
// hits in an interval of n candidates are n / p^2, so that taking them tile by
// tile in k_sieve spent nearly all its divisions on primes without a hit in
// the tile, and a plan of a few tiles ran on as many SMs: 2.5e5 candidates
// below 2^44 (295,000 primes, 4 tiles) 883 -> 21 us with k_sieve, 1.2e6 near
// 10^11 86 -> 19.
// The quotient is one high product, off by at most one.
__global__ void __launch_bounds__(256) k_sieve_big(const Seg *__restrict__ segs, uint32_t nseg,
                                                   const uint32_t *__restrict__ primes,
                                                   const uint64_t *__restrict__ sqtab,
                                                   uint32_t nprimes, uint32_t *__restrict__ sqfree) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nprimes) return;
    const uint64_t p2 = (uint64_t)primes[i] * primes[i], lim = sqtab[2 * i + 1];
    for (uint32_t si = blockIdx.y; si < nseg; si += gridDim.y) {
        const Seg s = segs[si];
        if (s.ncand == 0) continue;
        const uint64_t dlast = s.d0 + 8 * (s.ncand - 1);
        if (p2 > dlast) continue;
        uint64_t m = __umul64hi(s.d0, lim);  // floor(d0 / p^2) or one less
        while (m * p2 < s.d0) ++m;
        m += (13 - m % 8) % 8;  // m == 5 (mod 8)
        for (uint64_t dh = m * p2; dh <= dlast; dh += 8 * p2) {
            const uint64_t bit = s.cand0 + ((dh - s.d0) >> 3);
            atomicAnd(&sqfree[bit >> 5], ~(1u << (bit & 31)));
        }
    }
}

// Exclusive scan of tile_pop into tile_off (single CTA) and the total.
__global__ void __launch_bounds__(1024) k_scan_tiles(const uint32_t *__restrict__ tile_pop,
                                                     uint32_t *__restrict__ tile_off,
                                                     uint32_t ntiles, uint32_t *__restrict__ total) {
    __shared__ uint32_t red[32];
    uint32_t carry = 0;
    for (uint32_t base = 0; base < ntiles; base += blockDim.x) {
        const uint32_t i = base + threadIdx.x;
        const uint32_t v = i < ntiles ? tile_pop[i] : 0;
        uint32_t tot;
        const uint32_t ex = block_excl_scan(v, red, &tot);
        if (i < ntiles) tile_off[i] = carry + ex;
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

// K1b: the square-free candidates of each tile, in increasing order, as
// a compact queue from tile_off[tile].  The tile is taken in chunks of 256
// bitmap words, one per thread and read coalesced.  A block scan of the
// words' popcounts places each word's survivors in a shared-memory stage,
// and the block copies the stage to the queue with consecutive threads
// writing consecutive entries, so the queue is written in whole lines.
// flags (or null): after k_select, only what the cubic forms left undecided.
__global__ void __launch_bounds__(256) k_compact(const Tile *__restrict__ tiles,
                                                 const uint32_t *__restrict__ sqfree,
                                                 const uint32_t *__restrict__ tile_off,
                                                 uint32_t *__restrict__ surv,
                                                 const uint32_t *__restrict__ flags,
                                                 const uint32_t *__restrict__ field,
                                                 const uint8_t *__restrict__ seg_field) {
    __shared__ uint32_t red[32];
    __shared__ uint32_t stage[256 * 32];  // one chunk: at most 8192 survivors
    const Tile t = tiles[blockIdx.x];
    const uint32_t nw = (t.ncand + 31) >> 5;
    const uint64_t wbase = t.cand0 >> 5;
    uint32_t out = tile_off[blockIdx.x];
    const bool use = field && seg_field[t.seg];
    for (uint32_t c0 = 0; c0 < nw; c0 += 256) {
        const uint32_t w = c0 + threadIdx.x;
        uint32_t x = (w < nw) ? sqfree[wbase + w] : 0u;
        if (flags && x) x = left_word(x, flags[wbase + w], use ? field[wbase + w] : kFull);
        uint32_t tot;
        uint32_t o = block_excl_scan((uint32_t)__popc(x), red, &tot);
        const uint32_t cbase = (uint32_t)(t.cand0 + 32u * w);
        while (x) {
            stage[o++] = cbase + (uint32_t)(__ffs(x) - 1);
            x &= x - 1;
        }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < tot; i += 256) surv[out + i] = stage[i];
        out += tot;
        __syncthreads();
    }
}

// K4: per-interval counts.  counts[2*seg] += #E, counts[2*seg+1] += #D over
// the tile's words (ballot/popcount data already packed in the bitmaps).
// With glog, cls[3*seg + g] += #{d : log eps_d = g} for g = 0, 1, 2 (the
// class of eps_d in F_4* = {1, omega, omega^2}).
__global__ void __launch_bounds__(256) k_count(const Tile *__restrict__ tiles,
                                               const uint32_t *__restrict__ flags,
                                               const uint32_t *__restrict__ sqfree,
                                               unsigned long long *__restrict__ counts,
                                               const uint8_t *__restrict__ glog,
                                               unsigned long long *__restrict__ cls) {
    __shared__ uint32_t red[32];
    const Tile t = tiles[blockIdx.x];
    const uint32_t nw = (t.ncand + 31) >> 5;
    const uint64_t wbase = t.cand0 >> 5;
    uint32_t e = 0, dd = 0;
    for (uint32_t w = threadIdx.x; w < nw; w += blockDim.x) {
        e += __popc(flags[wbase + w]);
        dd += __popc(sqfree[wbase + w]);
    }
    e = block_sum(e, red);
    __syncthreads();
    dd = block_sum(dd, red);
    if (threadIdx.x == 0) {
        atomicAdd(&counts[2 * t.seg], (unsigned long long)e);
        atomicAdd(&counts[2 * t.seg + 1], (unsigned long long)dd);
    }
    if (glog && cls) {
        // sixteen bytes a load (a tile begins at a multiple of 32); byte by byte
        // a tile took 120 us, now 20 (6 in the short tiles of a small plan)
        uint32_t c[3] = {0, 0, 0};
        const uint32_t n16 = t.ncand / 16;
        const uint4 *g16 = reinterpret_cast<const uint4 *>(glog + t.cand0);
        for (uint32_t k = threadIdx.x; k < n16; k += blockDim.x) {
            const uint4 v = g16[k];
            for (int g = 0; g < 3; ++g) {
                const uint32_t want = 0x01010101u * (g + 1);
                c[g] += (__popc(__vcmpeq4(v.x, want)) + __popc(__vcmpeq4(v.y, want)) +
                         __popc(__vcmpeq4(v.z, want)) + __popc(__vcmpeq4(v.w, want))) >> 3;
            }
        }
        for (uint32_t k = n16 * 16 + threadIdx.x; k < t.ncand; k += blockDim.x) {
            const uint32_t v = glog[t.cand0 + k];
            c[0] += (v == 1);
            c[1] += (v == 2);
            c[2] += (v == 3);
        }
        for (int g = 0; g < 3; ++g) {
            __syncthreads();
            const uint32_t sum = block_sum(c[g], red);
            if (threadIdx.x == 0) atomicAdd(&cls[3 * t.seg + g], (unsigned long long)sum);
        }
    }
}

// Byte codes per candidate: 0 = not in D, 1 = in D \ E, 2 = in E.
__global__ void __launch_bounds__(256) k_expand_codes(const uint32_t *__restrict__ flags,
                                                      const uint32_t *__restrict__ sqfree,
                                                      uint64_t ncand, uint8_t *__restrict__ codes) {
    for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < ncand;
         k += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t b = 1u << (k & 31);
        const uint32_t sq = sqfree[k >> 5] & b, fl = flags[k >> 5] & b;
        codes[k] = fl ? 2 : (sq ? 1 : 0);
    }
}

// L2 flush helper for benchmarks: overwrite a buffer larger than L2.
__global__ void k_fill(uint32_t *__restrict__ buf, uint64_t nwords, uint32_t v) {
    for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < nwords;
         k += (uint64_t)gridDim.x * blockDim.x)
        buf[k] = v;
}

// Up to 4096 the tile's own pass over the primes is short.
int launch_sieve(uint32_t ntiles, cudaStream_t st, const Tile *tiles, const Seg *segs, uint32_t nseg,
                 const uint32_t *primes, const uint64_t *sqtab, uint32_t nprimes, uint32_t nsmall,
                 uint32_t np, uint32_t *sqfree, uint32_t *tile_pop, int primes_only) {
    const bool big = !primes_only && np > nsmall + 512;
    k_sieve<<<ntiles, 256, 0, st>>>(tiles, segs, primes, big ? nsmall : nprimes, sqfree, tile_pop,
                                    primes_only);
    if (!big) return 1;
    const uint32_t n = np - nsmall;
    // a thread takes several intervals with its prime when there are many
    const uint32_t gx = (n + 255) / 256, gy = 2432 / gx + 1;
    k_sieve_big<<<dim3(gx, nseg < gy ? nseg : gy), 256, 0, st>>>(
        segs, nseg, primes + nsmall, sqtab + 2 * nsmall, n, sqfree);
    return 2;
}

}  // namespace eis
