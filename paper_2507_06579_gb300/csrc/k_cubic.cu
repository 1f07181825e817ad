// k_cubic.cu -- the cubic-form enumeration over a plan's intervals
// (eis_cubic.cuh) and what it leaves to the walk and the search.
//
//  k_cubic   marks the d of every reduced form in the jobs' windows: kind 0
//            (discriminant 4d) in the flag bitmap, kind 1 (discriminant d) in
//            a second bitmap.
//  k_select  flags &= square-free; counts what is left per tile.
#include "eis_common.cuh"
#include "eis_cubic.cuh"
#include "eis_kernels.h"

namespace eis {

namespace {

__device__ __forceinline__ int32_t warp_incl_scan(int32_t v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// Least lane whose inclusive prefix exceeds t (the owner of item t).
__device__ __forceinline__ int scan_owner(int32_t incl, int32_t t) {
    int lo = 0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1)
        if (__shfl_sync(kFull, incl, lo + s - 1) <= t) lo += s;
    return lo;
}

}  // namespace

// One warp per unit (a; 8 consecutive b; a slice of the forms), units taken
// from a global counter, large b first (a unit has about 8 b / 3 values of c,
// so that the last units are the short ones).  The warp finds the 8 ranges of
// c and takes each 32 c at a time, one per lane; the lanes' bands of forms are
// laid out flat and tested 32 at a time, so that lanes stay busy whether a
// window holds thousands of forms per (b, c) or none.
// Bound by instruction issue (150 warp instructions for 32 (b, c), 82% of the
// issue slots busy); the bitmaps stay in L2.  Measured: 0.3 ms for windows up
// to 10^7 wide near 10^11, 1.1 ms near 10^12, and 0.8 ms for the 10^9 window
// below 10^11, whose pass went from 827 to 45 ms (walk) and from 425 to 38 ms
// (lane search) when the forms came in: 1.2e7 of its 1.0e8 d are left, with a
// third of the period.
__global__ void __launch_bounds__(256) k_cubic(const CubicJob *__restrict__ jobs, uint32_t njobs,
                                               uint32_t nunits, uint32_t *__restrict__ next_ptr,
                                               uint32_t *__restrict__ bits0,
                                               uint32_t *__restrict__ bits1) {
    const int lane = threadIdx.x & 31;
    for (;;) {
        uint32_t u = 0;
        if (lane == 0) u = atomicAdd(next_ptr, 1u);
        u = __shfl_sync(kFull, u, 0);
        if (u >= nunits) break;
        uint32_t jl = 0, jh = njobs;  // the last job with unit0 <= u
        while (jh - jl > 1) {
            const uint32_t mid = (jl + jh) >> 1;
            if (jobs[mid].unit0 <= u) jl = mid; else jh = mid;
        }
        const CubicJob job = jobs[jl];
        const uint32_t s1 = job.slices, v = u - job.unit0;
        const uint32_t nsl = s1 == 1 ? job.amax : cubic_slices_below(job.amax + 1, s1);
        const uint32_t blk = job.nblk - 1 - v / nsl;
        uint32_t slice = v % nsl, a = s1 == 1 ? 8 : 1, nslices = 1;
        while (a < 8 && slice >= (nslices = cubic_slices(a, s1))) slice -= cubic_slices(a++, s1);
        if (a == 8) {
            a = (s1 == 1 ? 1 : 8) + slice;
            slice = 0;
            nslices = 1;
        }
        const int kind = (int)job.kind;
        const CubicA A = cubic_a(job, (int32_t)a);
        const int32_t sh = cubic_shift(kind, A.a);
        uint32_t *__restrict__ bits = kind ? bits1 : bits0;
        const int32_t b0 = (int32_t)(blk * kCubicBlock);
        // lanes 2i and 2i + 1 find the two ends of pair i's range of P
        const float pend = cubic_p_end(A, b0 + (lane >> 1), lane & 1);
        const int32_t bm = b0 + (lane & 15);
        const float plo = __shfl_sync(kFull, pend, 2 * (lane & 15));
        const float phi = __shfl_sync(kFull, pend, 2 * (lane & 15) + 1);
        int32_t c_first = 0, nc = 0;
        if (lane < kCubicBlock && cubic_pair_ok(kind, A.a, bm)) nc = cubic_c_range(A, bm, plo, phi, c_first);
        for (uint32_t pairs = __ballot_sync(kFull, nc > 0); pairs; pairs &= pairs - 1) {
            const int pair = __ffs(pairs) - 1;
            const int32_t b = b0 + pair, items = __shfl_sync(kFull, nc, pair);
            const int32_t cf = __shfl_sync(kFull, c_first, pair) + 2 * lane;
            for (int32_t base = 0; base < items; base += 32) {
                const int32_t c = cf + 2 * base;
                CubicBands B = cubic_bands(A, b, c);
                if (base + lane >= items) B.n[0] = B.n[1] = 0;
                const int32_t len = B.n[0] + B.n[1];
                if (!__any_sync(kFull, len > 0)) continue;
                const int32_t lin = warp_incl_scan(len, lane);
                const int32_t total = __shfl_sync(kFull, lin, 31);
                for (int32_t t0 = 32 * (int32_t)slice; t0 < total; t0 += 32 * (int32_t)nslices) {
                    const int32_t t = t0 + lane;
                    const int own = scan_owner(lin, min(t, total - 1));
                    const int32_t i = t - __shfl_sync(kFull, lin - len, own);
                    const int32_t n0 = __shfl_sync(kFull, B.n[0], own);
                    const int32_t ka = __shfl_sync(kFull, B.k[0], own);
                    const int32_t kb = __shfl_sync(kFull, B.k[1], own);
                    const int32_t k = i < n0 ? ka + (i << sh) : kb + ((i - n0) << sh);
                    if (t < total) {
                        const int64_t h = cubic_hit(A, b, c + 2 * (own - lane), k, job.d0, job.ncand);
                        if (h >= 0) {
                            const uint64_t bit = job.bit0 + (uint64_t)h;
                            atomicOr(&bits[bit >> 5], 1u << (bit & 31));
                        }
                    }
                }
            }
        }
    }
}

// After the sieve and k_cubic: flags &= square-free, and per tile the number
// of candidates left to the walk (`left_word`).  flags null: only the count.
// glog (or null): 1 where the flag is set.
__global__ void __launch_bounds__(256) k_select(const Tile *__restrict__ tiles,
                                                const uint32_t *__restrict__ sqfree,
                                                uint32_t *__restrict__ flags,
                                                const uint32_t *__restrict__ field,
                                                const uint8_t *__restrict__ seg_field,
                                                uint8_t *__restrict__ glog,
                                                uint32_t *__restrict__ tile_pop) {
    __shared__ uint32_t red[32];
    const Tile t = tiles[blockIdx.x];
    const uint32_t nw = (t.ncand + 31) >> 5;
    const uint64_t wbase = t.cand0 >> 5;
    const bool use = field && seg_field[t.seg];
    uint32_t pop = 0;
    for (uint32_t w = threadIdx.x; w < nw; w += blockDim.x) {
        const uint32_t sq = sqfree[wbase + w], f = flags ? flags[wbase + w] & sq : 0u;
        if (flags) flags[wbase + w] = f;
        pop += __popc(left_word(sq, f, use ? field[wbase + w] : kFull));
        if (glog)
            for (uint32_t x = f; x; x &= x - 1) glog[32 * (wbase + w) + (__ffs(x) - 1)] = 1;
    }
    pop = block_sum(pop, red);
    if (threadIdx.x == 0) tile_pop[blockIdx.x] = pop;
}

}  // namespace eis
