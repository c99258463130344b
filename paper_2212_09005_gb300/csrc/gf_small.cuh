// Small batches in one CTA. A call of a few thousand keys spends its time in
// launches (a GQF sort: 16 of them, a TCF insert: 18), not in work, so such a
// batch is sorted in the shared memory of one CTA by a single kernel.
#pragma once

#include <stdint.h>

namespace gf {

static constexpr int SM_T = 1024;       // threads of the CTA
static constexpr uint32_t SM_HOT = 48;  // keys of one bucket above which the comparison ranks give way

// exclusive scan of one value per thread over the CTA; *total: their sum
__device__ __forceinline__ uint32_t small_scan(uint32_t v, uint32_t *s_warp, uint32_t *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    __syncthreads();  // s_warp may still be read from the last call
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t w = s_warp[lane], wi = w;  // SM_T / 32 == 32 warps
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
        if (lane >= o) wi += y;
    }
    *total = __shfl_sync(0xffffffffu, wi, 31);
    return incl - v + __shfl_sync(0xffffffffu, wi - w, warp);
}

// Sorts a[0 .. n) ascending (n <= CAP, distinct values; b: CAP words, cnt: CAP
// + 1 words of scratch). bucket(v) < CAP does not decrease with v and spreads
// the values evenly (they start with hash bits), so that a bucket holds about
// one: each value takes its place in its bucket by an atomic, then ranks
// itself among its bucket's few. A hot bucket (equal keys: SM_HOT of them or
// more) sends the batch to a bitonic sort instead, whose time does not depend
// on the values. Six barriers against the 78 stages of the bitonic sort.
template <int CAP, class Bucket>
__device__ __forceinline__ void small_sort(uint64_t *a, uint64_t *b, uint32_t *cnt, uint32_t *s_warp, uint32_t n,
                                           Bucket bucket)
{
    constexpr int PER = CAP / SM_T;
    static_assert(CAP % SM_T == 0 && (CAP & (CAP - 1)) == 0, "whole values per thread, a power of two for the stages");
    for (uint32_t k = threadIdx.x; k <= CAP; k += SM_T) cnt[k] = 0;
    __syncthreads();
    uint64_t v[PER];
    uint32_t bk[PER], at[PER];
    bool hot = false;
#pragma unroll
    for (int u = 0; u < PER; u++) {
        const uint32_t i = threadIdx.x + u * SM_T;
        if (i < n) {
            v[u] = a[i];
            bk[u] = bucket(v[u]);
            at[u] = atomicAdd(&cnt[bk[u]], 1u);
            hot |= at[u] >= SM_HOT;
        }
    }
    if (__syncthreads_or(hot)) {
        uint32_t m = 1;
        while (m < n) m <<= 1;
        for (uint32_t i = n + threadIdx.x; i < m; i += SM_T) a[i] = ~0ull;
        for (uint32_t k = 2; k <= m; k <<= 1)
            for (uint32_t j = k >> 1; j > 0; j >>= 1) {
                __syncthreads();
                for (uint32_t t = threadIdx.x; t < m / 2; t += SM_T) {
                    const uint32_t lo = ((t & ~(j - 1)) << 1) | (t & (j - 1)), hi = lo | j;
                    const uint64_t x = a[lo], y = a[hi];
                    if ((x > y) == ((lo & k) == 0)) {
                        a[lo] = y;
                        a[hi] = x;
                    }
                }
            }
        __syncthreads();
        return;
    }
    {
        uint32_t c[PER], sum = 0, total;
#pragma unroll
        for (int u = 0; u < PER; u++) {
            c[u] = cnt[threadIdx.x * PER + u];
            sum += c[u];
        }
        uint32_t run = small_scan(sum, s_warp, &total);
#pragma unroll
        for (int u = 0; u < PER; u++) {
            cnt[threadIdx.x * PER + u] = run;
            run += c[u];
        }
        if (threadIdx.x == 0) cnt[CAP] = n;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; u++)
        if (threadIdx.x + u * SM_T < n) b[cnt[bk[u]] + at[u]] = v[u];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; u++) {
        if (threadIdx.x + u * SM_T < n) {
            const uint32_t s = cnt[bk[u]], e = cnt[bk[u] + 1];
            uint32_t r = s;
            for (uint32_t j = s; j < e; j++) r += b[j] < v[u];
            a[r] = v[u];  // a is read no more: every value is in v and in b
        }
    }
    __syncthreads();
}

}  // namespace gf
