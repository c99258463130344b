// Two-choice filter (TCF), paper Sec. 4, for sm_103a.
//
// Table: nb blocks of 32 bytes (one DRAM sector), B = 256 / f tags each, plus a
// backing table of nbk buckets of 8 uint64 entries (Sec. 4.1, "Backing table").
//
// Query (Sec. 4): probe both candidate blocks with one 32-byte load each and a
// SIMD compare (__vcmpeq2 / __vcmpeq4), then the backing bucket (L2-resident)
// if the tag was in neither block.
//
// Bulk insert, deterministic mode (Sec. 4.1 shortcut + Sec. 4 two choices +
// Sec. 4.1 backing table + Sec. 4.2 sorted blocks). Each block phase groups
// its candidates by block (by units of blocks in shared memory, by a counting
// sort over all blocks, or by one over the blocks that are touched, whichever
// suits the table and the batch), then one thread per block takes the k
// smallest (tag, batch index) candidates that fit, merges them into its sorted
// block, and emits the rest to the next phase:
//   A shortcut into b1 while fill + j < 3B/4, B the less-full block under the
//   post-A fills, C the other block, D the backing bucket.
// Blocks keep a fill byte array beside them so that the two-choice decision
// reads 1 byte from L2 instead of a 32-byte sector from HBM.
//
// Point mode (Alg. 1): one thread per key; the tag goes into the first EMPTY
// or TOMBSTONE slot by an atomic compare-and-swap, retried a bounded number of
// times; deletes swap the tag for TOMBSTONE.
//
// Values (Sec. 1 and Sec. 4: small values stored with the items): with v
// value bits a slot holds the (f - v)-bit tag above the value. The phases
// carry whole slots; g and the bucket use the tag alone; matching masks the
// value bits; a value query answers the smallest value stored with the key's
// fingerprint in its blocks and backing bucket.
#include <type_traits>
#include <vector>

#include "gf_coop.h"
#include "gf_internal.cuh"
#include "gf_packed.cuh"
#include "gf_small.cuh"

namespace gf {

static constexpr int TPB = 256;
static constexpr uint32_t BK_W = 8;  // backing bucket entries
static constexpr int MAXSEL = 32;    // largest B

// ---------------------------------------------------------------------------
// 32-byte block in registers
// ---------------------------------------------------------------------------
template <int F>
struct Blk {
    static constexpr int B = 256 / F;
    uint32_t w[8];

    __device__ __forceinline__ void load(const uint8_t *blocks, uint64_t b)
    {
        const uint4 *p = reinterpret_cast<const uint4 *>(blocks + b * 32);
        const uint4 lo = p[0], hi = p[1];
        w[0] = lo.x; w[1] = lo.y; w[2] = lo.z; w[3] = lo.w;
        w[4] = hi.x; w[5] = hi.y; w[6] = hi.z; w[7] = hi.w;
    }
    // Queries and point updates take a block as one 256-bit access: a warp's
    // random blocks cost one pass of the L1's tags instead of two (2^23 queries
    // on 2^24 slots: 138 us before, 117 now).
    __device__ __forceinline__ void load_ro(const uint8_t *blocks, uint64_t b)
    {
        asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
            : "l"(blocks + b * 32));
    }
    __device__ __forceinline__ void load_l2(const uint8_t *blocks, uint64_t b)
    {
        asm volatile("ld.global.cg.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                     : "l"(blocks + b * 32)
                     : "memory");
    }
    __device__ __forceinline__ void store(uint8_t *blocks, uint64_t b) const
    {
        uint4 *p = reinterpret_cast<uint4 *>(blocks + b * 32);
        p[0] = make_uint4(w[0], w[1], w[2], w[3]);
        p[1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
    __device__ __forceinline__ uint32_t tag(int s) const
    {
        if (F == 16) return (w[s >> 1] >> ((s & 1) * 16)) & 0xffffu;
        return (w[s >> 2] >> ((s & 3) * 8)) & 0xffu;
    }
    // the tag part of every lane of a word (all ones without values)
    static __device__ __forceinline__ uint32_t lane_mask(uint32_t vmask)
    {
        return F == 16 ? (0xffffu & ~vmask) * 0x00010001u : (0xffu & ~vmask) * 0x01010101u;
    }
    // some slot holds tag t (t: the slot with value 0; lm from lane_mask)
    __device__ __forceinline__ bool has(uint32_t t, uint32_t lm) const
    {
        uint32_t m = 0;
        if (F == 16) {
            uint32_t tt = t | (t << 16);
#pragma unroll
            for (int k = 0; k < 8; k++) m |= __vcmpeq2(w[k] & lm, tt);
        } else {
            uint32_t tt = t * 0x01010101u;
#pragma unroll
            for (int k = 0; k < 8; k++) m |= __vcmpeq4(w[k] & lm, tt);
        }
        return m != 0;
    }
    // smallest value stored with tag t, or the lane maximum when none is
    __device__ __forceinline__ uint32_t min_value(uint32_t t, uint32_t lm) const
    {
        uint32_t b = 0xffffffffu;
        if (F == 16) {
            const uint32_t tt = t | (t << 16);
#pragma unroll
            for (int k = 0; k < 8; k++) b = __vminu2(b, (w[k] & ~lm) | ~__vcmpeq2(w[k] & lm, tt));
            return min(b & 0xffffu, b >> 16);
        } else {
            const uint32_t tt = t * 0x01010101u;
#pragma unroll
            for (int k = 0; k < 8; k++) b = __vminu4(b, (w[k] & ~lm) | ~__vcmpeq4(w[k] & lm, tt));
            b = __vminu4(b, b >> 16);
            return min(b & 0xffu, (b >> 8) & 0xffu);
        }
    }
    // tags >= 2 (neither EMPTY nor TOMBSTONE)
    __device__ __forceinline__ int live() const
    {
        int c = 0;
        if (F == 16) {
#pragma unroll
            for (int k = 0; k < 8; k++) c += __popc(__vcmpgeu2(w[k], 0x00020002u));
            return c >> 4;
        } else {
#pragma unroll
            for (int k = 0; k < 8; k++) c += __popc(__vcmpgeu4(w[k], 0x02020202u));
            return c >> 3;
        }
    }
    __device__ __forceinline__ int nonzero() const
    {
        int c = 0;
        if (F == 16) {
#pragma unroll
            for (int k = 0; k < 8; k++) c += __popc(__vcmpne2(w[k], 0u));
            return c >> 4;
        } else {
#pragma unroll
            for (int k = 0; k < 8; k++) c += __popc(__vcmpne4(w[k], 0u));
            return c >> 3;
        }
    }
    // bit s set where slot s holds tag t
    __device__ __forceinline__ uint32_t eq_slots(uint32_t t, uint32_t lm) const
    {
        uint32_t sm = 0;
        if (F == 16) {
            const uint32_t tt = t | (t << 16);
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const uint32_t m = __vcmpeq2(w[k] & lm, tt);
                sm |= ((m & 1u) | ((m >> 15) & 2u)) << (2 * k);
            }
        } else {
            const uint32_t tt = t * 0x01010101u;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const uint32_t m = __vcmpeq4(w[k] & lm, tt);
                sm |= ((m & 1u) | ((m >> 7) & 2u) | ((m >> 14) & 4u) | ((m >> 21) & 8u)) << (4 * k);
            }
        }
        return sm;
    }
    // bits of word k below bit position bp of the 256-bit block
    static __device__ __forceinline__ uint32_t low_bits(int k, int bp)
    {
        const int lo = bp - 32 * k;
        return lo >= 32 ? 0xffffffffu : (lo <= 0 ? 0u : ((1u << lo) - 1u));
    }
    // slot pos is removed: slots above it move down by one, the last becomes EMPTY
    __device__ __forceinline__ void delete_at(int pos)
    {
        const int bp = pos * F;
        uint32_t nw[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const uint32_t sh = k < 7 ? __funnelshift_r(w[k], w[k + 1], F) : (w[7] >> F);
            const uint32_t lo = low_bits(k, bp);
            nw[k] = (w[k] & lo) | (sh & ~lo);
        }
#pragma unroll
        for (int k = 0; k < 8; k++) w[k] = nw[k];
    }
    // Merge k new tags (the high words of r[0 .. k), ascending) into the f0
    // sorted tags of the block (f0 + k <= B, k <= 8) with a bitonic merge on
    // packed lanes: empty lanes become the largest tag value, the new tags go
    // descending into the top lanes, and log2(B) half-cleaner stages of SIMD
    // min / max sort the lanes ascending; lanes from f0 + k on are cleared.
    // Equal tags are indistinguishable, so the result equals the stable merge.
    __device__ __forceinline__ void merge_new(uint32_t f0, uint32_t k, const uint64_t (&r)[8])
    {
#pragma unroll
        for (int q = 0; q < 8; q++) w[q] |= ~low_bits(q, (int)(f0 * F));
#pragma unroll
        for (int m = 0; m < 8; m++) {
            if (m < (int)k) {
                constexpr int LPW = 32 / F;  // lanes per word
                const int L = B - 1 - m;
                const int sh = (L % LPW) * F;
                const uint32_t lane_mask = (F == 16 ? 0xffffu : 0xffu) << sh;
                w[L / LPW] = (w[L / LPW] & ~lane_mask) | ((uint32_t)(r[m] >> 32) << sh);
            }
        }
        // word-level half-cleaners: distances of 4, 2 and 1 words
#pragma unroll
        for (int dw = 4; dw >= 1; dw >>= 1) {
#pragma unroll
            for (int q = 0; q < 8; q++) {
                if ((q & dw) == 0) {
                    const uint32_t a = w[q], c = w[q + dw];
                    w[q] = F == 16 ? __vminu2(a, c) : __vminu4(a, c);
                    w[q + dw] = F == 16 ? __vmaxu2(a, c) : __vmaxu4(a, c);
                }
            }
        }
        // lane-level half-cleaners inside each word
#pragma unroll
        for (int q = 0; q < 8; q++) {
            uint32_t x = w[q];
            if (F == 8) {  // lanes two apart: swap the 16-bit halves
                const uint32_t y = __byte_perm(x, 0u, 0x1032u);
                x = __byte_perm(__vminu4(x, y), __vmaxu4(x, y), 0x7610u);
            }
            if (F == 16) {  // lanes one apart: the two halves
                const uint32_t y = __byte_perm(x, 0u, 0x1032u);
                x = __byte_perm(__vminu2(x, y), __vmaxu2(x, y), 0x7610u);
            } else {        // lanes one apart: bytes 0/1 and 2/3
                const uint32_t y = __byte_perm(x, 0u, 0x2301u);
                x = __byte_perm(__vminu4(x, y), __vmaxu4(x, y), 0x7250u);
            }
            w[q] = x;
        }
#pragma unroll
        for (int q = 0; q < 8; q++) w[q] &= low_bits(q, (int)((f0 + k) * F));
    }
    // pack B tags (ascending, zero padded) from an array
    __device__ __forceinline__ void pack(const uint32_t *t)
    {
#pragma unroll
        for (int k = 0; k < 8; k++) {
            if (F == 16) w[k] = (t[2 * k] & 0xffffu) | (t[2 * k + 1] << 16);
            else w[k] = (t[4 * k] & 0xffu) | ((t[4 * k + 1] & 0xffu) << 8) | ((t[4 * k + 2] & 0xffu) << 16) |
                        (t[4 * k + 3] << 24);
        }
    }
};

// sort up to 8 records held in registers (absent ones are ~0 and sort last):
// a 19-comparator network of depth 6, or 5 comparators for the first 4
// when no lane of the warp has more; callers index the array only in
// unrolled loops, which keeps it in registers
__device__ __forceinline__ void cswap(uint64_t &a, uint64_t &b)
{
    const uint64_t lo = a < b ? a : b, hi = a < b ? b : a;
    a = lo;
    b = hi;
}
__device__ __forceinline__ void sort4(uint64_t (&r)[8])
{
    cswap(r[0], r[1]); cswap(r[2], r[3]);
    cswap(r[0], r[2]); cswap(r[1], r[3]);
    cswap(r[1], r[2]);
}
__device__ __forceinline__ void sort8(uint64_t (&r)[8])
{
    cswap(r[0], r[2]); cswap(r[1], r[3]); cswap(r[4], r[6]); cswap(r[5], r[7]);
    cswap(r[0], r[4]); cswap(r[1], r[5]); cswap(r[2], r[6]); cswap(r[3], r[7]);
    cswap(r[0], r[1]); cswap(r[2], r[3]); cswap(r[4], r[5]); cswap(r[6], r[7]);
    cswap(r[2], r[4]); cswap(r[3], r[5]);
    cswap(r[1], r[4]); cswap(r[3], r[6]);
    cswap(r[1], r[2]); cswap(r[3], r[4]); cswap(r[5], r[6]);
}
__device__ __forceinline__ void sort_small(uint64_t (&r)[8], uint32_t cnt)
{
    const uint32_t wmax = __reduce_max_sync(__activemask(), cnt);
    if (wmax > 4) sort8(r);
    else if (wmax > 1) sort4(r);
}

// keep the `have` smallest values seen so far in a[0..have), ascending, at most k
__device__ __forceinline__ int topk_push(uint64_t *a, int have, int k, uint64_t v)
{
    if (have == k) {
        if (k == 0 || v >= a[k - 1]) return have;
        have--;
    }
    int j = have;
    while (j > 0 && a[j - 1] > v) {
        a[j] = a[j - 1];
        j--;
    }
    a[j] = v;
    return have + 1;
}

// ---------------------------------------------------------------------------
// Query (both modes)
// ---------------------------------------------------------------------------
// VAL: answer the smallest value stored with the key's fingerprint in its two
// blocks and its backing bucket, 0xFF when there is none; else 1 / 0.
template <int F, bool VAL>
__global__ void __launch_bounds__(TPB) tcf_query_kernel(const uint64_t *__restrict__ keys, uint64_t n,
                                                        TcfGeom G, const uint8_t *__restrict__ blocks,
                                                        const uint64_t *__restrict__ bk,
                                                        const DevCounters *ctr,
                                                        uint8_t *__restrict__ out)
{
    const bool backing = ctr->backing != 0;
    const uint32_t lm = Blk<F>::lane_mask(G.vmask);
    const uint64_t em = ~(uint64_t)G.vmask;
    for (uint64_t i = blockIdx.x * (uint64_t)TPB + threadIdx.x; i < n; i += (uint64_t)gridDim.x * TPB) {
        KeyInfo k = tcf_keyinfo(__ldcs(keys + i), G);  // keys and answers stream past the L2
        Blk<F> x, y;
        x.load_ro(blocks, k.b1);
        y.load_ro(blocks, k.b2);
        if (VAL) {
            uint32_t best = min(x.min_value(k.t, lm), y.min_value(k.t, lm));
            if (backing) {
                const uint64_t e = tcf_entry(k, G.f);
                const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(bk + tcf_bucket_of(e, G) * BK_W);
#pragma unroll
                for (int s = 0; s < 4; s++) {
                    const ulonglong2 v = __ldg(p + s);
                    if ((v.x & em) == e) best = min(best, (uint32_t)v.x & G.vmask);
                    if ((v.y & em) == e) best = min(best, (uint32_t)v.y & G.vmask);
                }
            }
            __stcs(out + i, (uint8_t)(best <= G.vmask ? best : 0xffu));
            continue;
        }
        bool hit = x.has(k.t, lm) || y.has(k.t, lm);
        if (!hit && backing) {
            uint64_t e = tcf_entry(k, G.f);
            const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(bk + tcf_bucket_of(e, G) * BK_W);
#pragma unroll
            for (int s = 0; s < 4; s++) {
                ulonglong2 v = __ldg(p + s);
                hit |= ((v.x & em) == e) | ((v.y & em) == e);
            }
        }
        __stcs(out + i, (uint8_t)(hit ? 1 : 0));
    }
}

// ---------------------------------------------------------------------------
// Counting-sort grouping kernels
// ---------------------------------------------------------------------------
// source of a phase's candidate list
enum Src : int { SRC_KEYS = 0, SRC_PEND_U32 = 1, SRC_PEND_U64 = 2 };
// how a candidate picks its destination
enum Dst : int { DST_B1 = 0, DST_TARGET = 1, DST_ALT = 2, DST_B2 = 3, DST_BUCKET = 4 };

// Key i of the call: hashed here, or (group calls) read from the prepared
// keys, whose block indices already address the group's concatenated arrays;
// b2 is read only by the destinations that need it.
template <int DST>
__device__ __forceinline__ KeyInfo key_at(const uint64_t *keys, const TcfPrep &P, uint64_t i, const TcfGeom &G)
{
    if (P.bt) {
        const uint64_t v = P.bt[i];
        KeyInfo k;
        k.b1 = v >> 32;
        k.t = (uint32_t)v;
        k.b2 = (DST == DST_TARGET || DST == DST_B2) ? P.b2[i] : 0;
        return k;
    }
    KeyInfo k = tcf_keyinfo(keys[i], G);
    if (P.vals) k.t |= P.vals[i] & G.vmask;
    return k;
}

__device__ __forceinline__ uint64_t dest_of(int dst, const KeyInfo &k, uint64_t pend_word, const TcfGeom &G,
                                            const uint8_t *fill, const TcfPrep &P, uint64_t i)
{
    switch (dst) {
    case DST_B1: return k.b1;
    case DST_B2: return k.b2;
    case DST_TARGET: return fill[k.b1] <= fill[k.b2] ? k.b1 : k.b2;
    case DST_ALT: return pend_word >> 32;
    default: return P.bt ? (uint64_t)P.bucket[i] : tcf_bucket_of(tcf_entry(k, G.f), G);
    }
}

// Traced launches whose work is only known on the device record it here
// (units is null when tracing is off)
__device__ __forceinline__ void note_units(unsigned long long *units, uint64_t v)
{
    if (units && blockIdx.x == 0 && threadIdx.x == 0) *units = v;
}

// A CTA's share of a sparse phase's candidates: one contiguous, warp-aligned
// chunk (the touched destinations it finds are listed from the chunk's start)
__device__ __forceinline__ void cta_chunk(uint64_t n, uint64_t &c0, uint64_t &c1)
{
    const uint64_t per = (((n + gridDim.x - 1) / gridDim.x) + 31) & ~31ull;
    c0 = per * blockIdx.x;
    if (c0 > n) c0 = n;
    c1 = c0 + per < n ? c0 + per : n;
}

// Dense phases count every candidate per destination; sparse phases (few
// candidates, as in the later phases) also list each destination the first
// time it is hit, per CTA chunk, in tlist[c0 ..] with the count in tcount.
template <int SRC, int DST, bool SPARSE>
__device__ __forceinline__ void tcf_group_hist_body(const uint64_t *__restrict__ keys, const TcfPrep prep,
                                                    uint64_t n_keys, const void *pend, const unsigned *npend,
                                                    TcfGeom G, const uint8_t *fill, uint32_t *cnt, uint32_t *tlist,
                                                    uint32_t *tcount, unsigned long long *units)
{
    const uint64_t n = (SRC == SRC_KEYS) ? n_keys : (uint64_t)*npend;
    note_units(units, n);
    __shared__ unsigned s_n;
    uint64_t c0 = 0, c1 = n, step = (uint64_t)gridDim.x * TPB, j = blockIdx.x * (uint64_t)TPB + threadIdx.x;
    if (SPARSE) {
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        cta_chunk(n, c0, c1);
        step = TPB;
        j = c0 + threadIdx.x;
    }
    for (; j < c1; j += step) {
        uint64_t pw = 0, i = j;
        if (SRC == SRC_PEND_U32) i = static_cast<const uint32_t *>(pend)[j];
        if (SRC == SRC_PEND_U64) {
            pw = static_cast<const uint64_t *>(pend)[j];
            i = pw & 0xffffffffu;
        }
        KeyInfo k = key_at<DST>(keys, prep, i, G);
        const uint64_t d = dest_of(DST, k, pw, G, fill, prep, i);
        if (SPARSE) {
            if (atomicAdd(&cnt[d], 1u) == 0u) tlist[c0 + atomicAdd(&s_n, 1u)] = (uint32_t)d;
        } else {
            atomicAdd(&cnt[d], 1u);  // no result used: a reduction the L2 applies without a reply
        }
    }
    if (SPARSE) {
        __syncthreads();
        if (threadIdx.x == 0) tcount[blockIdx.x] = s_n;
    }
}

template <int SRC, int DST, bool SPARSE>
__global__ void __launch_bounds__(TPB) tcf_group_hist(const uint64_t *__restrict__ keys, const TcfPrep prep,
                                                      uint64_t n_keys, const void *pend, const unsigned *npend,
                                                      TcfGeom G, const uint8_t *fill, uint32_t *cnt,
                                                      uint32_t *tlist, uint32_t *tcount, const unsigned *gate,
                                                      unsigned long long *units)
{
    if (gate && !*gate) return;
    tcf_group_hist_body<SRC, DST, SPARSE>(keys, prep, n_keys, pend, npend, G, fill, cnt, tlist, tcount, units);
}

// Sparse phases: every touched destination gets a contiguous segment of the
// record array (CTA-wide scan of the counts, one atomic per 256 destinations)
// and an entry in the dense touched list. Same grid as the histogram.
__device__ __forceinline__ void tcf_alloc_body(const unsigned *npend, uint64_t n_keys,
                                               const uint32_t *__restrict__ tlist,
                                               const uint32_t *__restrict__ tcount, const uint32_t *cnt,
                                               uint32_t *off, uint32_t *dlist, uint64_t *seg, unsigned *cursor,
                                               unsigned *nlist, unsigned long long *units)
{
    __shared__ uint32_t s_w[TPB / 32];
    __shared__ uint32_t s_base, s_lbase;
    const uint64_t n = npend ? (uint64_t)*npend : n_keys;
    uint64_t c0, c1;
    cta_chunk(n, c0, c1);
    const uint32_t m = tcount[blockIdx.x];
    if (units && threadIdx.x == 0 && m) atomicAdd(units, (unsigned long long)m);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint32_t j0 = 0; j0 < m; j0 += TPB) {
        const uint32_t j = j0 + threadIdx.x;
        const uint32_t d = j < m ? tlist[c0 + j] : 0u;
        const uint32_t c = j < m ? cnt[d] : 0u;
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_w[warp] = incl;
        __syncthreads();
        uint32_t pre = 0, tot = 0;
#pragma unroll
        for (int w = 0; w < TPB / 32; w++) {
            if (w < warp) pre += s_w[w];
            tot += s_w[w];
        }
        if (threadIdx.x == 0) {
            s_base = atomicAdd(cursor, tot);
            s_lbase = atomicAdd(nlist, m - j0 < (uint32_t)TPB ? m - j0 : (uint32_t)TPB);
        }
        __syncthreads();
        if (j < m) {
            const uint32_t start = s_base + pre + incl - c;
            off[d] = start;
            dlist[s_lbase + threadIdx.x] = d;
            seg[s_lbase + threadIdx.x] = ((uint64_t)start << 32) | c;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(TPB) tcf_alloc(const unsigned *npend, uint64_t n_keys,
                                                 const uint32_t *__restrict__ tlist,
                                                 const uint32_t *__restrict__ tcount, const uint32_t *cnt,
                                                 uint32_t *off, uint32_t *dlist, uint64_t *seg, unsigned *cursor,
                                                 unsigned *nlist, unsigned long long *units)
{
    tcf_alloc_body(npend, n_keys, tlist, tcount, cnt, off, dlist, seg, cursor, nlist, units);
}

// rec = (tag << 32) | batch index, or the backing entry with the index in recI
template <int SRC, int DST>
__device__ __forceinline__ void tcf_group_scatter_body(const uint64_t *__restrict__ keys, const TcfPrep prep,
                                                       uint64_t n_keys, const void *pend, const unsigned *npend,
                                                       TcfGeom G, const uint8_t *fill, uint32_t *cnt,
                                                       const uint32_t *__restrict__ off, uint64_t *rec,
                                                       uint32_t *recI, unsigned long long *units)
{
    const uint64_t n = (SRC == SRC_KEYS) ? n_keys : (uint64_t)*npend;
    note_units(units, n);
    for (uint64_t j = blockIdx.x * (uint64_t)TPB + threadIdx.x; j < n; j += (uint64_t)gridDim.x * TPB) {
        uint64_t pw = 0, i = j;
        if (SRC == SRC_PEND_U32) i = static_cast<const uint32_t *>(pend)[j];
        if (SRC == SRC_PEND_U64) {
            pw = static_cast<const uint64_t *>(pend)[j];
            i = pw & 0xffffffffu;
        }
        KeyInfo k = key_at<DST>(keys, prep, i, G);
        uint64_t d = dest_of(DST, k, pw, G, fill, prep, i);
        uint32_t pos = off[d] + atomicSub(&cnt[d], 1u) - 1u;
        if (DST == DST_BUCKET) {
            rec[pos] = prep.bt ? prep.e[i] : tcf_entry(k, G.f);
            recI[pos] = (uint32_t)i;
        } else {
            rec[pos] = ((uint64_t)k.t << 32) | i;
        }
    }
}

template <int SRC, int DST>
__global__ void __launch_bounds__(TPB) tcf_group_scatter(const uint64_t *__restrict__ keys, const TcfPrep prep,
                                                         uint64_t n_keys, const void *pend, const unsigned *npend,
                                                         TcfGeom G,
                                                         const uint8_t *fill, uint32_t *cnt,
                                                         const uint32_t *__restrict__ off, uint64_t *rec,
                                                         uint32_t *recI, const unsigned *gate,
                                                         unsigned long long *units)
{
    if (gate && !*gate) return;
    tcf_group_scatter_body<SRC, DST>(keys, prep, n_keys, pend, npend, G, fill, cnt, off, rec, recI, units);
}

// ---------------------------------------------------------------------------
// Bulk insert: per-block acceptance
// ---------------------------------------------------------------------------
// phase 0 (A): cap = 3B/4, rejects -> pend_u32; phase 1 (B): cap = B, rejects
// -> pend_u64 (alt block << 32 | index); phase 2 (C): cap = B, rejects -> pend_u32
// The blocks of a phase: every block with the scanned offsets (dense phases),
// or only the touched ones with their segments (sparse phases, dlist set).
struct PhaseDst {
    const uint32_t *off;     // dense: nb + 1 scanned offsets
    const uint32_t *dlist;   // sparse: touched destinations
    const uint64_t *seg;     // sparse: start << 32 | count
    const unsigned *nlist;   // sparse: number of touched destinations
    uint64_t nrec = 0;       // sparse: number of candidates (0: not told)
};

__device__ __forceinline__ uint64_t phase_count(const PhaseDst &P, uint64_t dense_n)
{
    return P.dlist ? (uint64_t)*P.nlist : dense_n;
}

// destination j of the phase with its record range [s, e)
__device__ __forceinline__ uint64_t phase_dst(const PhaseDst &P, uint64_t j, uint32_t &s, uint32_t &e)
{
    if (P.dlist) {
        const uint64_t sg = P.seg[j];
        s = (uint32_t)(sg >> 32);
        e = s + (uint32_t)sg;
        return P.dlist[j];
    }
    s = P.off[j];
    e = P.off[j + 1];
    return j;
}

// Touched destinations of many candidates each (copies of a key) take long, and
// lanes of a warp wait for one another: such a phase's destinations go round the
// warps first, then to their lanes. 2^18 keys, a hundred copies of each, on 2^20
// blocks, an insert and a remove: 1.32 and 3.55 ms with a warp's lanes side by
// side, 0.51 and 0.58 so.
__device__ __forceinline__ bool phase_spread(const PhaseDst &P, uint64_t nd) { return P.nrec >= 8 * nd && P.nrec; }

// what this thread takes in the round from t0 on
__device__ __forceinline__ uint64_t phase_pos(bool spread, uint64_t t0)
{
    const uint64_t warps = (uint64_t)gridDim.x * (TPB / 32);
    const uint64_t w = blockIdx.x * (uint64_t)(TPB / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    return t0 + (spread ? lane * warps + w : w * 32 + lane);
}

// f(record) for each of [s, e), four loads in flight (one by one, each load's
// latency counts: 32768 copies of one key, a remove 236 ms, 131 so)
template <bool MANY, class Fn>
__device__ __forceinline__ void each_record(const uint64_t *__restrict__ rec, uint32_t s, uint32_t e, Fn f)
{
    if constexpr (MANY) {
        for (uint32_t q = s; q < e; q += 4) {
            uint64_t r[4];
#pragma unroll
            for (uint32_t u = 0; u < 4; u++) r[u] = q + u < e ? rec[q + u] : 0ull;
#pragma unroll
            for (uint32_t u = 0; u < 4; u++)
                if (q + u < e) f(r[u]);
        }
    } else {
        for (uint32_t q = s; q < e; q++) f(rec[q]);
    }
}

// the same for a bucket's candidates: f(entry, index). MANY: one at a time where
// they are in shared memory, and few.
template <bool MANY, class Entry, class Index, class Fn>
__device__ __forceinline__ void each_candidate(uint32_t cnt, Entry entry, Index index, Fn f)
{
    constexpr uint32_t U = MANY ? 4 : 1;
    for (uint32_t q = 0; q < cnt; q += U) {
        uint64_t ee[U];
        uint32_t ii[U];
#pragma unroll
        for (uint32_t u = 0; u < U; u++) {
            ee[u] = q + u < cnt ? entry(q + u) : 0ull;
            ii[u] = q + u < cnt ? index(q + u) : 0u;
        }
#pragma unroll
        for (uint32_t u = 0; u < U; u++)
            if (q + u < cnt) f(ee[u], ii[u]);
    }
}

// A warp reserves room for all its lanes' entries of a pending list with one
// atomic; lane l's entries start at the returned position. Every lane of the
// warp must call it.
__device__ __forceinline__ uint32_t warp_reserve(unsigned *counter, uint32_t mine)
{
    const int lane = threadIdx.x & 31;
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    uint32_t base = 0;
    if (lane == 31 && total) base = atomicAdd(counter, total);
    base = __shfl_sync(0xffffffffu, base, 31);
    return base + incl - mine;
}

// Candidates that a per-block step passes on, collected per warp in shared
// memory and written out with one reservation on the list's counter per
// full buffer, instead of one returning atomic per warp and iteration. The
// order of a pending list is free: every later phase orders its candidates
// by (tag, batch index) itself. Exactly one of o32 / o64 is set; `n` is the
// same in every lane, and every lane of the warp calls reserve and flush.
static constexpr uint32_t SINK_CAP = 256;  // entries per warp

struct RejSink {
    uint64_t *buf;
    uint32_t n;
    uint32_t *o32;
    uint64_t *o64;
    unsigned *ctr;

    __device__ __forceinline__ void flush()
    {
        const int lane = threadIdx.x & 31;
        __syncwarp();
        uint32_t base = 0;
        if (lane == 0 && n) base = atomicAdd(ctr, n);
        base = __shfl_sync(0xffffffffu, base, 0);
        for (uint32_t q = lane; q < n; q += 32) {
            if (o64) o64[base + q] = buf[q];
            else o32[base + q] = (uint32_t)buf[q];
        }
        __syncwarp();
        n = 0;
    }
    // this lane's first position for `mine` entries; `direct` when the warp's
    // entries exceed a buffer and go straight to the list
    __device__ __forceinline__ uint32_t reserve(uint32_t mine, bool &direct)
    {
        const int lane = threadIdx.x & 31;
        uint32_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        if (n + total > SINK_CAP) flush();
        if (total > SINK_CAP) {
            uint32_t base = 0;
            if (lane == 31) base = atomicAdd(ctr, total);
            base = __shfl_sync(0xffffffffu, base, 31);
            direct = true;
            return base + incl - mine;
        }
        direct = false;
        const uint32_t pos = n + incl - mine;
        n += total;
        return pos;
    }
    __device__ __forceinline__ void put(bool direct, uint32_t &slot, uint64_t v)
    {
        if (!direct) buf[slot] = v;
        else if (o64) o64[slot] = v;
        else o32[slot] = (uint32_t)v;
        slot++;
    }
};

// Candidates of one block or bucket above which a warp takes an insert's step
// (copies of one key): 32768 of them in a batch of 2^18 took one thread 36 ms, a
// warp 3.7.
static constexpr uint32_t DST_HOT = 512;

// the smallest (v, i) over the warp
__device__ __forceinline__ void warp_min_pair(uint64_t &v, uint32_t &i)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t y = __shfl_xor_sync(0xffffffffu, v, o);
        const uint32_t k = __shfl_xor_sync(0xffffffffu, i, o);
        if (y < v || (y == v && k < i)) {
            v = y;
            i = k;
        }
    }
}

// the insert step of block b with records [s, e) (the whole warp calls it): the
// next smallest record once per free slot, then the rest into the pending list
template <int F>
__device__ __noinline__ void hot_block_insert(uint8_t *blocks, uint8_t *fill, uint64_t b, uint32_t f0, uint32_t cap,
                                              const uint64_t *rec, uint32_t s, uint32_t e, int phase, uint32_t *pend32,
                                              uint64_t *pend64, unsigned *npend, uint64_t nb, uint32_t vbits,
                                              const TcfPrep prep)
{
    const uint32_t lane = threadIdx.x & 31, k = cap > f0 ? min(e - s, cap - f0) : 0u;
    uint64_t thr = 0;
    if (k) {
        Blk<F> blk;
        blk.load(blocks, b);
        for (uint32_t j = 0; j < k; j++) {
            uint64_t m = ~0ull;
            uint32_t none = 0;
#pragma unroll 4
            for (uint32_t q = s + lane; q < e; q += 32) {
                const uint64_t r = rec[q];
                if ((j == 0 || r > thr) && r < m) m = r;
            }
            warp_min_pair(m, none);
            thr = m;
            uint64_t r8[8] = {thr, 0, 0, 0, 0, 0, 0, 0};
            blk.merge_new(f0 + j, 1, r8);
        }
        if (lane == 0) {
            blk.store(blocks, b);
            fill[b] = (uint8_t)(f0 + k);
        }
    }
    for (uint32_t q0 = s; q0 < e; q0 += 32) {
        const uint64_t r = q0 + lane < e ? rec[q0 + lane] : 0ull;
        const bool left = q0 + lane < e && !(k > 0 && r <= thr);
        const unsigned lefts = __ballot_sync(0xffffffffu, left);
        uint32_t base = 0;
        if (lane == 0 && lefts) base = atomicAdd(npend, __popc(lefts));
        base = __shfl_sync(0xffffffffu, base, 0) + __popc(lefts & ((1u << lane) - 1u));
        if (!left) continue;
        const uint32_t i = (uint32_t)r;
        if (phase == 1) {  // the other block of the pair
            const uint64_t alt = prep.bt ? (prep.bt[i] >> 32) + prep.b2[i] - b : b ^ tcf_g((uint32_t)(r >> 32) >> vbits, nb);
            pend64[base] = (alt << 32) | i;
        } else {
            pend32[base] = i;
        }
    }
    __syncwarp();
}

// The grid-stride loops of the per-block kernels step whole warps, so that
// every lane reaches the sink's reserve in every iteration and its flush
// after the last one.
// COOP: as the cooperative launch takes them, hot blocks by a warp and a phase's
// destinations spread (the kernel over every block keeps its 48 registers without).
template <int F, bool COOP>
__device__ __forceinline__ void tcf_block_insert_body(TcfGeom G, uint8_t *blocks, uint8_t *fill, PhaseDst P,
                                                      const uint64_t *__restrict__ rec, int phase, uint32_t cap,
                                                      uint32_t *pend32, uint64_t *pend64, unsigned *npend,
                                                      const TcfPrep prep, unsigned long long *units)
{
    constexpr int B = Blk<F>::B;
    __shared__ uint64_t s_sink[TPB / 32][SINK_CAP];
    RejSink sink{s_sink[threadIdx.x >> 5], 0u, phase == 1 ? nullptr : pend32, phase == 1 ? pend64 : nullptr, npend};
    const uint64_t nd = phase_count(P, G.nb);
    if (P.dlist) note_units(units, nd);  // units: blocks with candidates
    const uint64_t stride = (uint64_t)gridDim.x * TPB;
    const bool spread = COOP && phase_spread(P, nd);
    for (uint64_t t0 = COOP ? 0 : blockIdx.x * (uint64_t)TPB + (threadIdx.x & ~31u); t0 < nd; t0 += stride) {
        const uint64_t j = COOP ? phase_pos(spread, t0) : t0 + (threadIdx.x & 31);
        uint32_t s = 0, e = 0, k = 0, f0 = 0;
        uint64_t b = 0, thr = 0;  // records <= thr are accepted
        if (j < nd) {
            b = phase_dst(P, j, s, e);
            f0 = fill[b];  // dense phases: b = j, so this load goes out with the offsets'
        }
        if (units && !P.dlist) {
            const unsigned t = __ballot_sync(0xffffffffu, s != e);
            if ((threadIdx.x & 31) == 0 && t) atomicAdd(units, (unsigned long long)__popc(t));
        }
        for (unsigned hot = COOP ? __ballot_sync(0xffffffffu, e - s > DST_HOT) : 0u; hot; hot &= hot - 1) {
            const int src = __ffs(hot) - 1;
            hot_block_insert<F>(blocks, fill, __shfl_sync(0xffffffffu, b, src), __shfl_sync(0xffffffffu, f0, src), cap, rec,
                                __shfl_sync(0xffffffffu, s, src), __shfl_sync(0xffffffffu, e, src), phase, pend32, pend64,
                                npend, G.nb, G.vbits, prep);
            if ((int)(threadIdx.x & 31) == src) s = e;
        }
        if (j < nd) {
            if (s != e) {
                const uint32_t cnt = e - s;
                k = cap > f0 ? min(cnt, cap - f0) : 0u;
                if (k > 0 && cnt <= 8) {
                    // few candidates: all loads in flight at once, a sorting
                    // network in registers, a bitonic merge into the block
                    Blk<F> blk;
                    blk.load(blocks, b);
                    uint64_t r8[8];
#pragma unroll
                    for (int q = 0; q < 8; q++) r8[q] = q < (int)cnt ? rec[s + q] : ~0ull;
                    sort_small(r8, cnt);
#pragma unroll
                    for (int q = 0; q < 8; q++)
                        if (q == (int)k - 1) thr = r8[q];
                    blk.merge_new(f0, k, r8);
                    blk.store(blocks, b);
                    fill[b] = (uint8_t)(f0 + k);
                } else if (k > 0) {
                    Blk<F> blk;
                    blk.load(blocks, b);
                    uint64_t a[MAXSEL];
                    int have = 0;
                    each_record<COOP>(rec, s, e, [&](uint64_t r) { have = topk_push(a, have, (int)k, r); });
                    thr = a[k - 1];
                    uint32_t t_out[B];
                    int ia = 0, ib = 0;
#pragma unroll
                    for (int p = 0; p < B; p++) {
                        uint32_t ta = (ia < (int)f0) ? blk.tag(ia) : 0xffffffffu;
                        uint32_t tb = (ib < (int)k) ? (uint32_t)(a[ib] >> 32) : 0xffffffffu;
                        if (ta == 0xffffffffu && tb == 0xffffffffu) {
                            t_out[p] = 0;
                        } else if (ta <= tb) {
                            t_out[p] = ta;
                            ia++;
                        } else {
                            t_out[p] = tb;
                            ib++;
                        }
                    }
                    blk.pack(t_out);
                    blk.store(blocks, b);
                    fill[b] = (uint8_t)(f0 + k);
                }
            }
        }
        const uint32_t nrej = (e - s) - k;
        bool direct;
        uint32_t slot = sink.reserve(nrej, direct);
        if (nrej == 0) continue;
        auto pass_on = [&](uint64_t r) {
            if (k > 0 && r <= thr) return;
            const uint32_t i = (uint32_t)r;
            if (phase == 1) {
                // the other block of the pair: b1 + b2 - b
                uint64_t alt = prep.bt ? (prep.bt[i] >> 32) + prep.b2[i] - b
                                       : b ^ tcf_g((uint32_t)(r >> 32) >> G.vbits, G.nb);
                sink.put(direct, slot, (alt << 32) | i);
            } else {
                sink.put(direct, slot, i);
            }
        };
        if (COOP && e - s > 8) each_record<COOP>(rec, s, e, pass_on);
        else each_record<false>(rec, s, e, pass_on);
    }
    sink.flush();
}

template <int F>
__global__ void __launch_bounds__(TPB) tcf_block_insert(TcfGeom G, uint8_t *blocks, uint8_t *fill, PhaseDst P,
                                                        const uint64_t *__restrict__ rec, int phase,
                                                        uint32_t cap, uint32_t *pend32, uint64_t *pend64,
                                                        unsigned *npend, const TcfPrep prep, const unsigned *gate,
                                                        unsigned long long *units)
{
    if (gate && !*gate) return;
    tcf_block_insert_body<F, false>(G, blocks, fill, P, rec, phase, cap, pend32, pend64, npend, prep, units);
}

// One backing bucket q: cnt candidates (entry(j), index(j)) taken in (entry,
// index) order while there is room; the rest are FULL
template <bool MANY, class Entry, class Index>
__device__ __forceinline__ void bucket_insert_step(uint64_t *bk, uint64_t q, uint32_t cnt, Entry entry, Index index,
                                                   uint8_t *status, DevCounters *ctr)
{
    uint64_t cur[BK_W];
    int used = 0;
    for (int j = 0; j < (int)BK_W; j++) {
        cur[j] = bk[q * BK_W + j];
        used += cur[j] != 0;
    }
    const uint32_t k = min(cnt, BK_W - (uint32_t)used);
    // select the k smallest (entry, index) pairs by repeated minimum
    uint64_t pe = 0;
    uint32_t pi = 0;
    bool have_prev = false;
    uint64_t acc_e[BK_W];
    for (uint32_t m = 0; m < k; m++) {
        uint64_t be = ~0ull;
        uint32_t bi = 0xffffffffu;
        each_candidate<MANY>(cnt, entry, index, [&](uint64_t ee, uint32_t ii) {
            bool after = !have_prev || ee > pe || (ee == pe && ii > pi);
            bool better = ee < be || (ee == be && ii < bi);
            if (after && better) {
                be = ee;
                bi = ii;
            }
        });
        acc_e[m] = be;
        pe = be;
        pi = bi;
        have_prev = true;
    }
    // merge accepted (ascending) into the bucket's sorted entries
    uint64_t outv[BK_W];
    int ia = 0, ib = 0;
    for (int p = 0; p < (int)BK_W; p++) {
        uint64_t va = ia < used ? cur[ia] : ~0ull;
        uint64_t vb = ib < (int)k ? acc_e[ib] : ~0ull;
        if (va == ~0ull && vb == ~0ull) outv[p] = 0;
        else if (va <= vb) { outv[p] = va; ia++; }
        else { outv[p] = vb; ib++; }
    }
    for (int j = 0; j < (int)BK_W; j++) bk[q * BK_W + j] = outv[j];
    if (k > 0) atomicAdd(&ctr->backing, (unsigned long long)k);
    if (k < cnt) {
        // rejected: every pair after the k-th accepted one
        each_candidate<MANY>(cnt, entry, index, [&](uint64_t ee, uint32_t ii) {
            bool acc = k > 0 && (ee < pe || (ee == pe && ii <= pi));
            if (!acc) {
                if (status) status[ii] = FILTER_KEY_FULL;
                atomicAdd(&ctr->failed, 1ull);
            }
        });
        atomicOr(&ctr->status, ST_FULL);
    }
}

// One backing bucket q: per stored entry, the smallest batch indices among
// the cnt candidates with that entry remove one copy each
template <bool MANY, class Entry, class Index>
__device__ __forceinline__ void bucket_remove_step(const TcfGeom &G, uint64_t *bk, uint64_t q, uint32_t cnt, Entry entry,
                                                   Index index, uint8_t *status, DevCounters *ctr)
{
    // distinct stored entries without their values (the bucket is sorted,
    // so copies are adjacent) with their first position and copy counts
    uint64_t cur[BK_W], dv[BK_W];
    uint32_t dp[BK_W], dc[BK_W], used[BK_W], thr[BK_W];
    int nd = 0;
    for (int j = 0; j < (int)BK_W; j++) {
        const uint64_t v = bk[q * BK_W + j];
        cur[j] = v;
        if (!v) continue;
        const uint64_t mv = v & ~(uint64_t)G.vmask;
        if (nd > 0 && dv[nd - 1] == mv) {
            dc[nd - 1]++;
        } else {
            dv[nd] = mv;
            dp[nd] = (uint32_t)j;
            dc[nd] = 1;
            nd++;
        }
    }
    // for each stored entry, the dc smallest candidate indices with that entry match
    for (int d = 0; d < nd; d++) {
        uint64_t a[BK_W];
        int have = 0;
        each_candidate<MANY>(cnt, entry, index, [&](uint64_t v, uint32_t ii) {
            if (v == dv[d]) have = topk_push(a, have, (int)dc[d], (uint64_t)ii);
        });
        used[d] = (uint32_t)have;
        thr[d] = have ? (uint32_t)a[have - 1] : 0u;
    }
    int removed = 0;
    uint64_t outv[BK_W];
    int o = 0;
    for (int d = 0; d < nd; d++) {
        removed += (int)used[d];
        for (uint32_t c = used[d]; c < dc[d]; c++) outv[o++] = cur[dp[d] + c];
    }
    for (int j = o; j < (int)BK_W; j++) outv[j] = 0;
    if (removed) {
        for (int j = 0; j < (int)BK_W; j++) bk[q * BK_W + j] = outv[j];
        atomicAdd(&ctr->backing, (unsigned long long)(-(long long)removed));
    }
    if (!status) return;
    each_candidate<MANY>(cnt, entry, index, [&](uint64_t v, uint32_t ii) {
        bool matched = false;
        for (int d = 0; d < nd; d++)
            if (dv[d] == v && used[d] > 0 && ii <= thr[d]) matched = true;
        if (!matched) status[ii] = FILTER_KEY_NOT_FOUND;
    });
}

// the insert step of bucket q with cnt candidates, by the whole warp
__device__ __noinline__ void hot_bucket_insert(uint64_t *bk, uint64_t q, uint32_t cnt, const uint64_t *rec,
                                               const uint32_t *recI, uint8_t *status, DevCounters *ctr)
{
    const uint32_t lane = threadIdx.x & 31;
    uint64_t cur[BK_W], pe = 0;
    uint32_t used = 0, pi = 0;
#pragma unroll
    for (int j = 0; j < (int)BK_W; j++) {
        cur[j] = bk[q * BK_W + j];
        used += cur[j] != 0;
    }
    __syncwarp();
    const uint32_t k = BK_W - used;  // (fewer than the candidates)
    for (uint32_t m = 0; m < k; m++) {
        uint64_t be = ~0ull;
        uint32_t bi = 0xffffffffu;
#pragma unroll 4
        for (uint32_t j = lane; j < cnt; j += 32) {
            const uint64_t ee = rec[j];
            const uint32_t ii = recI[j];
            if ((m == 0 || ee > pe || (ee == pe && ii > pi)) && (ee < be || (ee == be && ii < bi))) {
                be = ee;
                bi = ii;
            }
        }
        warp_min_pair(be, bi);
        pe = be;
        pi = bi;
        // into the sorted entries, free ones (0) last
        uint64_t v = be;
#pragma unroll
        for (int j = 0; j < (int)BK_W; j++) {
            const uint64_t x = cur[j];
            if (v && (x == 0 || v < x)) {
                cur[j] = v;
                v = x;
            }
        }
    }
    if (lane == 0 && k) {
#pragma unroll
        for (int j = 0; j < (int)BK_W; j++) bk[q * BK_W + j] = cur[j];
        atomicAdd(&ctr->backing, (unsigned long long)k);
    }
    for (uint32_t j = lane; j < cnt; j += 32) {
        const uint64_t ee = rec[j];
        const uint32_t ii = recI[j];
        if (!(k > 0 && (ee < pe || (ee == pe && ii <= pi))) && status) status[ii] = FILTER_KEY_FULL;
    }
    if (lane == 0) {
        atomicAdd(&ctr->failed, (unsigned long long)(cnt - k));
        atomicOr(&ctr->status, ST_FULL);
    }
    __syncwarp();
}

// backing buckets of a phase: candidates (entry in rec, index in recI)
template <bool HOT>
__device__ __forceinline__ void tcf_bucket_insert_body(TcfGeom G, uint64_t *bk, PhaseDst P,
                                                       const uint64_t *__restrict__ rec,
                                                       const uint32_t *__restrict__ recI, uint8_t *status,
                                                       DevCounters *ctr, unsigned long long *units)
{
    const uint64_t nd = phase_count(P, G.nbk);
    note_units(units, nd);  // units: buckets with candidates
    const bool spread = phase_spread(P, nd);
    for (uint64_t t0 = 0; t0 < nd; t0 += (uint64_t)gridDim.x * TPB) {
        const uint64_t j = phase_pos(spread, t0);
        uint32_t s = 0, e = 0;
        uint64_t q = 0;
        if (j < nd) q = phase_dst(P, j, s, e);
        for (unsigned hot = HOT ? __ballot_sync(0xffffffffu, e - s > DST_HOT) : 0u; hot; hot &= hot - 1) {
            const int src = __ffs(hot) - 1;
            const uint32_t hs = __shfl_sync(0xffffffffu, s, src), he = __shfl_sync(0xffffffffu, e, src);
            hot_bucket_insert(bk, __shfl_sync(0xffffffffu, q, src), he - hs, rec + hs, recI + hs, status, ctr);
            if ((int)(threadIdx.x & 31) == src) s = e;
        }
        if (s == e) continue;
        bucket_insert_step<true>(bk, q, e - s, [&](uint32_t i) { return rec[s + i]; }, [&](uint32_t i) { return recI[s + i]; },
                           status, ctr);
    }
}

__global__ void __launch_bounds__(TPB) tcf_bucket_insert(TcfGeom G, uint64_t *bk, PhaseDst P,
                                                         const uint64_t *__restrict__ rec,
                                                         const uint32_t *__restrict__ recI, uint8_t *status,
                                                         DevCounters *ctr, unsigned long long *units)
{
    tcf_bucket_insert_body<false>(G, bk, P, rec, recI, status, ctr, units);
}

// ---------------------------------------------------------------------------
// Bulk delete: per-block matching. For each tag present c times in the block,
// the c smallest (tag, index) candidates with that tag remove one copy each.
// ---------------------------------------------------------------------------
template <int F, bool COOP>
__device__ __forceinline__ void tcf_block_remove_body(TcfGeom G, uint8_t *blocks, uint8_t *fill, PhaseDst P,
                                                      const uint64_t *__restrict__ rec, uint32_t *pend32,
                                                      unsigned *npend, unsigned long long *units)
{
    constexpr int B = Blk<F>::B;
    __shared__ uint64_t s_sink[TPB / 32][SINK_CAP];
    RejSink sink{s_sink[threadIdx.x >> 5], 0u, pend32, nullptr, npend};
    const uint64_t nd = phase_count(P, G.nb);
    if (P.dlist) note_units(units, nd);  // units: blocks with candidates
    const uint32_t lm = Blk<F>::lane_mask(G.vmask);
    const uint64_t stride = (uint64_t)gridDim.x * TPB;
    const bool spread = COOP && phase_spread(P, nd);
    for (uint64_t t0 = COOP ? 0 : blockIdx.x * (uint64_t)TPB + (threadIdx.x & ~31u); t0 < nd; t0 += stride) {
        const uint64_t j = COOP ? phase_pos(spread, t0) : t0 + (threadIdx.x & 31);
        uint32_t s = 0, e = 0, nunm = 0, unm = 0;
        bool fast = false;
        uint64_t r8[8];  // fast path: the candidates, sorted
        // general path: per distinct stored tag, its first slot, the copies,
        // the candidates that matched and the largest matched record
        uint32_t dt[B], dp[B], dc[B], used[B];
        uint64_t thr[B];
        int ndt = 0;
        uint64_t b = 0;
        uint32_t f0 = 0;
        if (j < nd) {
            b = phase_dst(P, j, s, e);
            f0 = fill[b];  // dense phases: b = j, so this load goes out with the offsets'
        }
        if (units && !P.dlist) {
            const unsigned t = __ballot_sync(0xffffffffu, s != e);
            if ((threadIdx.x & 31) == 0 && t) atomicAdd(units, (unsigned long long)__popc(t));
        }
        if (j < nd) {
            if (s != e) {
                Blk<F> blk;
                blk.load(blocks, b);
                int removed = 0;
                if (e - s <= 8) {
                    // few candidates: sort them in registers; each takes the
                    // first remaining copy of its tag, so the block stays sorted
                    fast = true;
                    const uint32_t c = e - s;
#pragma unroll
                    for (int q = 0; q < 8; q++) r8[q] = (uint32_t)q < c ? rec[s + q] : ~0ull;
                    sort_small(r8, c);
#pragma unroll
                    for (int q = 0; q < 8; q++) {
                        if ((uint32_t)q < c) {
                            const uint32_t sm = blk.eq_slots((uint32_t)(r8[q] >> 32), lm);
                            if (sm) {
                                blk.delete_at(__ffs(sm) - 1);
                                removed++;
                            } else {
                                unm |= 1u << q;
                                nunm++;
                            }
                        }
                    }
                    if (removed) {
                        blk.store(blocks, b);
                        fill[b] = (uint8_t)(f0 - removed);
                    }
                } else {
                    uint32_t tags[B];
#pragma unroll
                    for (int p = 0; p < B; p++) tags[p] = blk.tag(p);
                    // copies of a tag are adjacent (sorted by tag, then value)
                    for (int p = 0; p < (int)f0; p++) {
                        const uint32_t mt = tags[p] & ~G.vmask;
                        if (ndt > 0 && dt[ndt - 1] == mt) {
                            dc[ndt - 1]++;
                        } else {
                            dt[ndt] = mt;
                            dp[ndt] = (uint32_t)p;
                            dc[ndt] = 1;
                            ndt++;
                        }
                    }
                    for (int d = 0; d < ndt; d++) {
                        uint64_t a[MAXSEL];
                        int have = 0;
                        uint64_t lo = (uint64_t)dt[d] << 32, hi = lo | 0xffffffffull;
                        each_record<COOP>(rec, s, e, [&](uint64_t r) {
                            if (r >= lo && r <= hi) have = topk_push(a, have, (int)dc[d], r);
                        });
                        used[d] = (uint32_t)have;
                        thr[d] = have ? a[have - 1] : 0;
                    }
                    // rebuild the block without the removed copies (the
                    // smallest values of each tag)
                    uint32_t t_out[B];
                    int o = 0;
                    for (int d = 0; d < ndt; d++) {
                        for (uint32_t c = used[d]; c < dc[d]; c++) t_out[o++] = tags[dp[d] + c];
                        removed += (int)used[d];
                    }
                    for (int p = o; p < B; p++) t_out[p] = 0;
                    if (removed) {
                        blk.pack(t_out);
                        blk.store(blocks, b);
                        fill[b] = (uint8_t)(f0 - removed);
                    }
                    nunm = (e - s) - (uint32_t)removed;
                }
            }
        }
        // unmatched candidates go on
        bool direct;
        uint32_t slot = sink.reserve(nunm, direct);
        if (nunm == 0) continue;
        if (fast) {
#pragma unroll
            for (int q = 0; q < 8; q++)
                if ((unm >> q) & 1u) sink.put(direct, slot, (uint32_t)r8[q]);
        } else {
            each_record<COOP>(rec, s, e, [&](uint64_t r) {
                const uint32_t t = (uint32_t)(r >> 32);
                bool matched = false;
                for (int d = 0; d < ndt; d++)
                    if (dt[d] == t && used[d] > 0 && r <= thr[d]) matched = true;
                if (!matched) sink.put(direct, slot, (uint32_t)r);
            });
        }
    }
    sink.flush();
}

template <int F>
__global__ void __launch_bounds__(TPB) tcf_block_remove(TcfGeom G, uint8_t *blocks, uint8_t *fill, PhaseDst P,
                                                        const uint64_t *__restrict__ rec, uint32_t *pend32,
                                                        unsigned *npend, const unsigned *gate,
                                                        unsigned long long *units)
{
    if (gate && !*gate) return;
    tcf_block_remove_body<F, false>(G, blocks, fill, P, rec, pend32, npend, units);
}

// backing buckets of a remove
__device__ __forceinline__ void tcf_bucket_remove_body(TcfGeom G, uint64_t *bk, PhaseDst P,
                                                       const uint64_t *__restrict__ rec,
                                                       const uint32_t *__restrict__ recI, uint8_t *status,
                                                       DevCounters *ctr, unsigned long long *units)
{
    const uint64_t nd = phase_count(P, G.nbk);
    note_units(units, nd);  // units: buckets with candidates
    const bool spread = phase_spread(P, nd);
    for (uint64_t t0 = 0; t0 < nd; t0 += (uint64_t)gridDim.x * TPB) {
        const uint64_t j = phase_pos(spread, t0);
        if (j >= nd) continue;
        uint32_t s, e;
        const uint64_t q = phase_dst(P, j, s, e);
        if (s == e) continue;
        bucket_remove_step<true>(G, bk, q, e - s, [&](uint32_t i) { return rec[s + i]; },
                           [&](uint32_t i) { return recI[s + i]; }, status, ctr);
    }
}

__global__ void __launch_bounds__(TPB) tcf_bucket_remove(TcfGeom G, uint64_t *bk, PhaseDst P,
                                                         const uint64_t *__restrict__ rec,
                                                         const uint32_t *__restrict__ recI, uint8_t *status,
                                                         DevCounters *ctr, unsigned long long *units)
{
    tcf_bucket_remove_body(G, bk, P, rec, recI, status, ctr, units);
}

// ---------------------------------------------------------------------------
// The later phases of a call in one cooperative launch: what the launches of
// the sparse path do one after another (histogram, segments, scatter and steps
// of the less full block, the other block and the backing buckets), with a
// barrier of the grid in each launch's place, and an end as soon as a phase has
// no candidates. Eleven launches cost about 45 us whatever they have to do.
// ---------------------------------------------------------------------------
// Every CTA of the grid arrives at *bar; thread 0 waits for the n-th round of
// them. False when the wait gave up (the status word then shows a timeout).
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned round, unsigned long long *status)
{
    __shared__ bool s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned want = round * gridDim.x;
        __threadfence();
        atomicAdd(bar, 1u);
        bool ok = false;
        for (uint32_t i = 0; i < SPIN_LIMIT && !ok; i++) {
            unsigned got;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(bar) : "memory");
            ok = got >= want;
        }
        if (!ok) atomicOr(status, ST_TIMEOUT);
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok;
}

// what the phases work on
struct SparseArgs {
    const uint64_t *keys;
    uint64_t n;
    TcfGeom G;
    TcfPrep prep;
    uint8_t *blocks, *fill;
    uint64_t *bk;
    uint32_t *cnt, *off, *tlist, *tcount, *dlist, *pend0, *pend2;
    uint64_t *rec, *pend1, *seg;
    uint8_t *status;
    DevCounters *ctr;
    uint32_t unit_min;  // more candidates than this of the second phase went by unit
    bool first;         // the first phase is taken here too
    const unsigned *uneven;  // set: all phases are taken here, or all but the first
    bool first_done;
};

__device__ __forceinline__ unsigned ld_now(const unsigned *p) { return *(const volatile unsigned *)p; }

// Where a call's phases have got to: the barriers passed, and whether one CTA
// has taken over (a phase had few candidates; the next ones have no more).
struct SparseRun {
    unsigned round;
    bool few;
};
static constexpr int SPARSE_FEW = TPB;  // a candidate, and then a destination, a thread of the first CTA

// the end of a phase's part: its writes are seen by the next
__device__ __forceinline__ bool sparse_next(const SparseArgs &A, SparseRun &run)
{
    if (!run.few) return grid_barrier(&A.ctr->bar, ++run.round, &A.ctr->status);
    __syncthreads();
    return true;
}

// Few candidates, by one CTA: their segments by counting. Over the grid a
// phase of a hundred candidates took 9 to 13 us, all of it barriers and
// latency; most calls have one or two of that size.
template <int SRC, int DST>
__device__ __forceinline__ void few_group(const SparseArgs &A, const void *pend, uint32_t m, uint32_t *recI,
                                          unsigned *touched)
{
    __shared__ uint32_t s_d[SPARSE_FEW];
    const uint32_t j = threadIdx.x;
    uint64_t rec = 0, i = j;
    uint32_t d = 0;
    if (j < m) {
        uint64_t pw = 0;
        if (SRC == SRC_PEND_U32) i = static_cast<const uint32_t *>(pend)[j];
        if (SRC == SRC_PEND_U64) {
            pw = static_cast<const uint64_t *>(pend)[j];
            i = pw & 0xffffffffu;
        }
        const KeyInfo k = key_at<DST>(A.keys, A.prep, i, A.G);
        d = (uint32_t)dest_of(DST, k, pw, A.G, A.fill, A.prep, i);
        s_d[j] = d;
        rec = DST == DST_BUCKET ? (A.prep.bt ? A.prep.e[i] : tcf_entry(k, A.G.f)) : ((uint64_t)k.t << 32) | i;
    }
    __syncthreads();
    if (j >= m) return;
    uint32_t less = 0, before = 0, same = 0;
    for (uint32_t q = 0; q < m; q++) {
        const uint32_t x = s_d[q];
        less += x < d;
        same += x == d;
        before += x == d && q < j;
    }
    A.rec[less + before] = rec;
    if (DST == DST_BUCKET) recI[less + before] = (uint32_t)i;
    if (before) return;
    const unsigned at = atomicAdd(touched, 1u);
    A.dlist[at] = d;
    A.seg[at] = ((uint64_t)less << 32) | same;
}

// Groups the candidates of one phase by the destinations that they touch.
// False in a CTA that is done: no candidates, another CTA has the rest, or a
// barrier gave up.
template <int SRC, int DST>
__device__ __forceinline__ bool sparse_group(const SparseArgs &A, const void *pend, const unsigned *npend, int slot,
                                             uint32_t *recI, SparseRun &run, PhaseDst &P)
{
    DevCounters *c = A.ctr;
    const uint64_t m = SRC == SRC_KEYS ? A.n : (uint64_t)ld_now(npend);  // (the same in every CTA)
    if (m == 0) return false;
    P = PhaseDst{nullptr, A.dlist, A.seg, &c->touched[slot], m};
    if (run.few || m <= SPARSE_FEW) {
        run.few = true;
        P.nrec = 0;  // (the other CTAs' warps are gone)
        if (blockIdx.x != 0) return false;
        few_group<SRC, DST>(A, pend, (uint32_t)m, recI, &c->touched[slot]);
        __syncthreads();
        return true;
    }
    tcf_group_hist_body<SRC, DST, true>(A.keys, A.prep, A.n, pend, npend, A.G, A.fill, A.cnt, A.tlist, A.tcount, nullptr);
    if (!sparse_next(A, run)) return false;
    tcf_alloc_body(npend, A.n, A.tlist, A.tcount, A.cnt, A.off, A.dlist, A.seg, &c->cursor[slot], &c->touched[slot], nullptr);
    if (!sparse_next(A, run)) return false;
    tcf_group_scatter_body<SRC, DST>(A.keys, A.prep, A.n, pend, npend, A.G, A.fill, A.cnt, A.off, A.rec, recI, nullptr);
    return sparse_next(A, run);
}

template <int F>
__global__ void __launch_bounds__(TPB, 4) tcf_sparse_insert_coop(const SparseArgs A)
{
    unsigned *np = A.ctr->pend;
    SparseRun run{0, false};
    PhaseDst P;
    const bool uneven = A.uneven && ld_now(A.uneven), all = A.first || uneven;  // (the same in every CTA)
    if (A.first || (uneven && !A.first_done)) {
        if (!sparse_group<SRC_KEYS, DST_B1>(A, nullptr, nullptr, 0, nullptr, run, P)) return;
        tcf_block_insert_body<F, true>(A.G, A.blocks, A.fill, P, A.rec, 0, A.G.tsc, A.pend0, nullptr, &np[0], A.prep, nullptr);
        if (!sparse_next(A, run)) return;
    }
    if (all || ld_now(&np[0]) <= A.unit_min) {
        if (!sparse_group<SRC_PEND_U32, DST_TARGET>(A, A.pend0, &np[0], 1, nullptr, run, P)) return;
        tcf_block_insert_body<F, true>(A.G, A.blocks, A.fill, P, A.rec, 1, A.G.B, nullptr, A.pend1, &np[1], A.prep, nullptr);
        if (!sparse_next(A, run)) return;
        if (!sparse_group<SRC_PEND_U64, DST_ALT>(A, A.pend1, &np[1], 2, nullptr, run, P)) return;
        tcf_block_insert_body<F, true>(A.G, A.blocks, A.fill, P, A.rec, 2, A.G.B, A.pend2, nullptr, &np[2], A.prep, nullptr);
        if (!sparse_next(A, run)) return;
    }
    if (!sparse_group<SRC_PEND_U32, DST_BUCKET>(A, A.pend2, &np[2], 3, A.pend0, run, P)) return;
    tcf_bucket_insert_body<true>(A.G, A.bk, P, A.rec, A.pend0, A.status, A.ctr, nullptr);
}

template <int F>
__global__ void __launch_bounds__(TPB, 4) tcf_sparse_remove_coop(const SparseArgs A)
{
    unsigned *np = A.ctr->pend;
    SparseRun run{0, false};
    PhaseDst P;
    const bool uneven = A.uneven && ld_now(A.uneven), all = A.first || uneven;  // (the same in every CTA)
    if (A.first || (uneven && !A.first_done)) {
        if (!sparse_group<SRC_KEYS, DST_B1>(A, nullptr, nullptr, 0, nullptr, run, P)) return;
        tcf_block_remove_body<F, true>(A.G, A.blocks, A.fill, P, A.rec, A.pend0, &np[0], nullptr);
        if (!sparse_next(A, run)) return;
    }
    if (all || ld_now(&np[0]) <= A.unit_min) {
        if (!sparse_group<SRC_PEND_U32, DST_B2>(A, A.pend0, &np[0], 1, nullptr, run, P)) return;
        tcf_block_remove_body<F, true>(A.G, A.blocks, A.fill, P, A.rec, A.pend2, &np[2], nullptr);
        if (!sparse_next(A, run)) return;
    }
    if (!sparse_group<SRC_PEND_U32, DST_BUCKET>(A, A.pend2, &np[2], 2, A.pend0, run, P)) return;
    tcf_bucket_remove_body(A.G, A.bk, P, A.rec, A.pend0, A.status, A.ctr, nullptr);
}

// ---------------------------------------------------------------------------
// Small batches: every phase of an insert or remove in one CTA. A phase sorts
// its candidates by (destination, slot, index) in shared memory; the first
// candidate of a block finds the others behind it, already in the order in
// which the block takes them, and does the block's step. The phases are kept
// apart by CTA barriers, as the launches of the general path keep them. Bound
// by latency (four to five dependent loads per phase and the barriers): one
// launch instead of 18 for an insert, 1000 keys into 2^20 slots in 20 us
// instead of 76.
// ---------------------------------------------------------------------------
static constexpr int TS_CAP = 2048;  // keys
static constexpr uint32_t TS_IDX = 11, TS_DST = 27;  // a candidate: dest << 27 | slot << 11 | index
static_assert(TS_CAP == 1 << TS_IDX, "the index fits its field");
static constexpr size_t TS_SMEM = TS_CAP * 16 + TS_CAP * 8 + TS_CAP * 2 + (TS_CAP + 1) * 4;

template <int F, bool DEL>
__global__ void __launch_bounds__(SM_T) tcf_small(const uint64_t *__restrict__ keys, const TcfPrep prep, uint32_t n,
                                                  TcfGeom G, uint8_t *blocks, uint8_t *fill, uint64_t *bk,
                                                  uint8_t *status, DevCounters *ctr)
{
    extern __shared__ __align__(16) uint64_t s_small[];
    __shared__ uint32_t s_warp[32], s_next;
    uint64_t *a = s_small, *left = s_small + TS_CAP;
    uint32_t *b1 = reinterpret_cast<uint32_t *>(left + TS_CAP), *b2 = b1 + TS_CAP;
    uint32_t *cnt = b2 + TS_CAP;
    uint16_t *slot = reinterpret_cast<uint16_t *>(cnt + TS_CAP + 1);
    const uint32_t lm = Blk<F>::lane_mask(G.vmask);
    for (uint32_t i = threadIdx.x; i < n; i += SM_T) {
        const KeyInfo k = key_at<DST_B2>(keys, prep, i, G);
        b1[i] = (uint32_t)k.b1;
        b2[i] = (uint32_t)k.b2;
        slot[i] = (uint16_t)k.t;
        a[i] = (k.b1 << TS_DST) | ((uint64_t)k.t << TS_IDX) | i;
        if (status) status[i] = FILTER_KEY_OK;
    }
    const uint64_t block_scale = ((uint64_t)TS_CAP << 32) / G.nb;  // destinations spread over the sort's buckets
    // insert: shortcut into b1, the less full block, the other; remove: b1, b2
    for (int phase = 0; phase < (DEL ? 2 : 3); phase++) {
        if (threadIdx.x == 0) s_next = 0;
        small_sort<TS_CAP>(a, left, cnt, s_warp, n, [block_scale](uint64_t v) {
            return (uint32_t)(((v >> TS_DST) * block_scale) >> 32);
        });
        for (uint32_t i = threadIdx.x; i < n; i += SM_T) {
            const uint64_t d = a[i] >> TS_DST;
            if (i > 0 && (a[i - 1] >> TS_DST) == d) continue;
            uint32_t e = i + 1;
            while (e < n && (a[e] >> TS_DST) == d) e++;
            const uint32_t f0 = fill[d];
            Blk<F> blk;
            if (DEL) {
                blk.load(blocks, d);
                uint32_t removed = 0;
                for (uint32_t q = i; q < e; q++) {
                    const uint32_t sm = blk.eq_slots((uint32_t)(a[q] >> TS_IDX) & 0xffffu, lm);
                    if (sm) {
                        blk.delete_at(__ffs(sm) - 1);
                        removed++;
                    } else {
                        left[atomicAdd(&s_next, 1u)] = a[q];
                    }
                }
                if (removed) {
                    blk.store(blocks, d);
                    fill[d] = (uint8_t)(f0 - removed);
                }
                continue;
            }
            const uint32_t cap = phase == 0 ? G.tsc : G.B;
            const uint32_t k = cap > f0 ? min(e - i, cap - f0) : 0u;
            if (k) {
                blk.load(blocks, d);
                for (uint32_t q0 = 0; q0 < k; q0 += 8) {
                    const uint32_t kk = min(8u, k - q0);
                    uint64_t r8[8];
#pragma unroll
                    for (uint32_t m = 0; m < 8; m++) r8[m] = m < kk ? ((a[i + q0 + m] >> TS_IDX) & 0xffffu) << 32 : 0;
                    blk.merge_new(f0 + q0, kk, r8);
                }
                blk.store(blocks, d);
                fill[d] = (uint8_t)(f0 + k);
            }
            if (i + k < e) {
                uint32_t pos = atomicAdd(&s_next, e - i - k);
                for (uint32_t q = i + k; q < e; q++) left[pos++] = a[q];
            }
        }
        __syncthreads();  // the blocks and fills of this phase are written
        n = s_next;
        if (n == 0) return;
        for (uint32_t j = threadIdx.x; j < n; j += SM_T) {
            const uint64_t v = left[j];
            const uint32_t i = (uint32_t)v & (TS_CAP - 1);
            uint64_t d;
            if (phase == (DEL ? 1 : 2)) {  // on to the backing buckets
                const KeyInfo k{b1[i], b2[i], slot[i]};
                a[j] = ((prep.bt ? (uint64_t)prep.bucket[i] : tcf_bucket_of(tcf_entry(k, G.f), G)) << TS_DST) | i;
                continue;
            }
            if (DEL) d = b2[i];
            else if (phase == 0) d = fill[b1[i]] <= fill[b2[i]] ? b1[i] : b2[i];
            else d = (v >> TS_DST) == b1[i] ? b2[i] : b1[i];
            a[j] = (d << TS_DST) | (v & ((1ull << TS_DST) - 1ull));
        }
        __syncthreads();
    }
    const uint64_t bucket_scale = ((uint64_t)TS_CAP << 32) / G.nbk;
    small_sort<TS_CAP>(a, left, cnt, s_warp, n, [bucket_scale](uint64_t v) {
        return (uint32_t)(((v >> TS_DST) * bucket_scale) >> 32);
    });
    for (uint32_t i = threadIdx.x; i < n; i += SM_T) {
        const uint64_t d = a[i] >> TS_DST;
        if (i > 0 && (a[i - 1] >> TS_DST) == d) continue;
        uint32_t e = i + 1;
        while (e < n && (a[e] >> TS_DST) == d) e++;
        auto index = [&](uint32_t q) { return (uint32_t)a[i + q] & (TS_CAP - 1); };
        auto entry = [&](uint32_t q) {
            const uint32_t x = index(q);
            return prep.bt ? prep.e[x] : tcf_entry(KeyInfo{b1[x], b2[x], slot[x]}, G.f);
        };
        if (DEL) bucket_remove_step<false>(G, bk, d, e - i, entry, index, status, ctr);
        else bucket_insert_step<false>(bk, d, e - i, entry, index, status, ctr);
    }
}

// ---------------------------------------------------------------------------
// Bulk phases by unit. A phase's candidates are partitioned by the top bits of
// their destination block (one or two passes whose writes are runs, gf_msd.cu)
// into units of two thousand candidates and their stretch of blocks; one CTA
// per unit groups its candidates by block in shared memory, and a thread per
// block that has some takes its step. A candidate is one word: the low bits of its
// block, its slot and its batch index; the partition implies the bits above.
// Against a counting sort by block (a counter, an offset and a scattered
// record per block and key) every global write is a run, nothing is sized by
// the table, and a phase's time goes with its candidates.
// ---------------------------------------------------------------------------
static constexpr int TU_T = 512;             // threads of a unit
static constexpr uint32_t TU_CAP = 3072;     // candidates that a unit holds in shared memory
static constexpr int TU_PER = TU_CAP / TU_T;
static constexpr uint32_t TU_BBITS = 12, TU_BUCKETS = 1u << TU_BBITS;  // buckets they are grouped by: a block or a few
// Candidates of one bucket above which the CTA takes them, one bucket after
// another: 20 us each, where a thread takes 0.2 us a candidate and other buckets go
// beside it (42,000 keys with a hundred copies each on 2^22 blocks: 3.28 ms an
// insert's step and 6.88 a remove's with 64, 0.33 and 0.69 so).
static constexpr uint32_t TU_HOT = 512;
static constexpr uint32_t TU_MANY = 16;  // and above which a remove skips the rest of a tag without copies left
static uint64_t tcf_unit_words(uint64_t max_n);  // scratch words of calls of up to max_n keys
static MsdScratch tu_scratch(uint32_t *base, uint64_t max_n);

// geometry of one phase: 2^k units of 2^lbits blocks each
struct TuGeom {
    uint32_t k, b1, b2;      // unit bits, in one (b2 = 0) or two passes
    uint32_t lbits;          // bits of a block inside its unit
    uint32_t sbits, ibits;   // slot and index bits of a record
};

// where a phase's candidates come from: the call's keys (hashed here, or the
// prepared keys of a group call), or a pending list (rec, idx) of n_dev items
struct TuSrc {
    const uint64_t *keys;
    const uint64_t *rec;     // dest << 16 | slot
    const uint32_t *idx;
    const unsigned *n_dev;   // pending lists: their length on the device,
    uint32_t n_min;          // taken for zero up to this many (the cooperative launch takes them)
    uint64_t n;              // keys: their number; pending lists: an upper bound
};

enum TuSrcKind : int { TU_KEYS = 0, TU_TARGET = 1, TU_SAME = 2 };      // dest: b1; the less full block; the record's
enum TuNext : int { TU_NX_SAME = 0, TU_NX_OTHER = 1, TU_NX_IDX = 2 };  // what a candidate left becomes

__device__ __forceinline__ uint64_t tu_count(const TuSrc &s)
{
    if (!s.n_dev) return s.n;
    const unsigned m = *s.n_dev;
    return m > s.n_min ? m : 0;
}

// the other block of the pair of candidate (b, slot, idx): b1 ^ b2 = g(tag)
// for a single filter; group calls read the prepared pair
__device__ __forceinline__ uint64_t tu_other(uint64_t b, uint32_t slot, uint32_t i, const TcfGeom &G, const TcfPrep &P)
{
    if (P.bt) return (P.bt[i] >> 32) + P.b2[i] - b;
    return b ^ tcf_g(slot >> G.vbits, G.nb);
}

// candidate j: its destination block; rec = its record
template <int SRC>
__device__ __forceinline__ uint64_t tu_item(const TuSrc &s, uint64_t j, const TcfGeom &G, const TcfPrep &P,
                                            const uint8_t *fill, const TuGeom &U, uint64_t &rec)
{
    uint64_t b;
    uint32_t slot, idx = (uint32_t)j;
    if (SRC == TU_KEYS) {
        if (P.bt) {
            const uint64_t v = P.bt[j];
            b = v >> 32;
            slot = (uint32_t)v;
        } else {
            KeyInfo k = tcf_keyinfo(__ldcs(s.keys + j), G);
            if (P.vals) k.t |= P.vals[j] & G.vmask;
            b = k.b1;
            slot = k.t;
        }
    } else {
        const uint64_t r = s.rec[j];
        idx = s.idx[j];
        b = r >> 16;
        slot = (uint32_t)(r & 0xffffu);
        if (SRC == TU_TARGET) {
            const uint64_t b2 = tu_other(b, slot, idx, G, P);
            if (fill[b] > fill[b2]) b = b2;
        }
    }
    rec = (b << (U.sbits + U.ibits)) | ((uint64_t)slot << U.ibits) | idx;  // (bits above 64 are the first pass's)
    return b;
}

template <int SRC>
__global__ void __launch_bounds__(MP_T) tu_hist(const TuSrc s, TcfGeom G, TcfPrep P, const uint8_t *fill, TuGeom U,
                                                MsdScratch M, const unsigned *uneven, unsigned long long *units)
{
    __shared__ uint32_t h[MP_BINS];
    const uint32_t nb = 1u << U.b1, shift = U.lbits + U.b2;
    if (uneven && *uneven) {
        if (blockIdx.x == 0 && threadIdx.x == 0) M.tile1[nb] = M.htile1[nb] = 0;  // nothing for the second pass
        return;
    }
    const uint64_t n = tu_count(s);
    note_units(units, n);
    for (uint32_t b = threadIdx.x; b < nb; b += MP_T) h[b] = 0;
    __syncthreads();
    for (uint64_t base = (uint64_t)blockIdx.x * MP_TILE; base < n; base += (uint64_t)gridDim.x * MP_TILE) {
        uint64_t b[MP_I];
#pragma unroll
        for (int r = 0; r < MP_I; r++) {
            const uint64_t j = base + r * MP_T + threadIdx.x;
            uint64_t rec;
            b[r] = j < n ? tu_item<SRC>(s, j, G, P, fill, U, rec) : 0;
        }
#pragma unroll
        for (int r = 0; r < MP_I; r++)
            if (base + r * MP_T + threadIdx.x < n) atomicAdd(&h[(uint32_t)(b[r] >> shift)], 1u);
    }
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < nb; b += MP_T)
        if (h[b]) atomicAdd(&M.cnt1[b], h[b]);
    hist_end(M, nb, U.b2 > 0);
}

// the first pass: a tile's records to the bins of their blocks' top bits
template <int SRC>
__global__ void __launch_bounds__(MP_T, 3) tu_part(const TuSrc s, TcfGeom G, TcfPrep P, const uint8_t *fill, TuGeom U,
                                                   MsdScratch M, uint64_t *__restrict__ out, const unsigned *uneven,
                                                   unsigned long long *units)
{
    __shared__ PartSmem S;
    if (uneven && *uneven) return;
    const uint64_t n = tu_count(s), base = (uint64_t)blockIdx.x * MP_TILE;
    note_units(units, n);
    if (base >= n) return;
    const uint32_t cnt = n - base < MP_TILE ? (uint32_t)(n - base) : MP_TILE, shift = U.lbits + U.b2;
    const uint32_t nb = 1u << U.b1, rshift = shift + U.sbits + U.ibits;
    const bool whole = rshift + U.b1 <= 64;
    uint64_t v[MP_I];
    uint16_t bin[MP_I];
#pragma unroll
    for (int r = 0; r < MP_I; r++) {
        const uint32_t i = r * MP_T + threadIdx.x;
        if (i < cnt) bin[r] = (uint16_t)(tu_item<SRC>(s, base + i, G, P, fill, U, v[r]) >> shift);
    }
    part_tile<false>(S, v, cnt, nb, [&](uint64_t, int r) { return (uint32_t)bin[r]; }, M.cur1);
#pragma unroll
    for (int r = 0; r < MP_I; r++) {
        const uint32_t i = r * MP_T + threadIdx.x;
        if (i >= cnt) continue;
        const uint64_t x = S.key[i];
        uint32_t b;
        if (whole) {
            b = (uint32_t)(x >> rshift);
        } else {  // the record does not hold its bin's bits: the last bin that starts at or before it
            uint32_t hi = nb;
            b = 0;
            while (hi - b > 1) {
                const uint32_t mid = (b + hi) >> 1;
                if (S.cnt[mid] <= i) b = mid;
                else hi = mid;
            }
        }
        out[S.delta[b] + i] = x;
    }
}

struct TuSmem {
    uint32_t cnt[TU_BUCKETS / 2 + 4];  // per bucket, two to a word: records, then the first position
    uint64_t a[TU_CAP];                // records by bucket
    uint16_t head[TU_CAP], left[TU_CAP];  // buckets with records; positions of the records left
    uint16_t hot[TU_CAP / TU_HOT];
    uint32_t warp[TU_T / 32];
    unsigned long long red[TU_T / 32];
    uint32_t nhead, nleft, nhot, base;
    unsigned long long bytes;
};

// Groups a unit's n records (record r * TU_T + t in thread t) by bucket into
// S.a and lists the buckets that have some in S.head. All threads pass its
// barriers.
__device__ __forceinline__ void tu_group(TuSmem &S, const uint64_t (&key)[TU_PER], uint32_t n, uint32_t shift)
{
    const uint16_t *first = reinterpret_cast<const uint16_t *>(S.cnt);
    for (uint32_t k = threadIdx.x; k < TU_BUCKETS / 8; k += TU_T) reinterpret_cast<uint4 *>(S.cnt)[k] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    uint32_t at[TU_PER];  // bucket << 16 | rank
#pragma unroll
    for (int r = 0; r < TU_PER; r++) {
        if (r * TU_T >= n) break;
        if (r * TU_T + threadIdx.x < n) {
            const uint32_t bk = (uint32_t)(key[r] >> shift), sh = (bk & 1u) * 16u;
            at[r] = (bk << 16) | ((atomicAdd(&S.cnt[bk >> 1], 1u << sh) >> sh) & 0xffffu);  // (no half carries)
        }
    }
    __syncthreads();
    {
        // one scan for the buckets' starts and the places in the list: counts
        // below 2^16 each, so that records and buckets share a word
        uint4 *w = reinterpret_cast<uint4 *>(S.cnt) + threadIdx.x;
        static_assert(TU_BUCKETS / 8 == TU_T, "four words per thread");
        const uint4 y = *w;
        uint32_t x[4] = {y.x, y.y, y.z, y.w}, sum = 0, some = 0;  // some: bit q set where bucket q has records
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint32_t lo = x[q] & 0xffffu, hi = x[q] >> 16;
            some |= (lo ? 1u << (2 * q) : 0u) | (hi ? 2u << (2 * q) : 0u);
            x[q] = sum | ((sum + lo) << 16);
            sum += lo + hi;
        }
        const uint32_t pre = cta_scan<TU_T>(sum | (__popc(some) << 16), S.warp), p2 = (pre & 0xffffu) * 0x00010001u;
        *w = make_uint4(x[0] + p2, x[1] + p2, x[2] + p2, x[3] + p2);
        uint32_t h = pre >> 16;
        if (threadIdx.x == TU_T - 1) {
            S.cnt[TU_BUCKETS / 2] = n;
            S.nhead = h + __popc(some);
        }
        for (; some; some &= some - 1) S.head[h++] = (uint16_t)(threadIdx.x * 8 + __ffs(some) - 1);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < TU_PER; r++) {
        if (r * TU_T >= n) break;
        if (r * TU_T + threadIdx.x < n) S.a[first[at[r] >> 16] + (at[r] & 0xffffu)] = key[r];
    }
    __syncthreads();
}

// smallest over the CTA; S.red is free again after the next barrier
__device__ __forceinline__ uint64_t tu_min(TuSmem &S, uint64_t m)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t y = __shfl_xor_sync(0xffffffffu, m, o);
        m = y < m ? y : m;
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) S.red[threadIdx.x >> 5] = m;
    __syncthreads();
    m = S.red[0];
#pragma unroll
    for (int w = 1; w < TU_T / 32; w++) m = S.red[w] < m ? S.red[w] : m;
    return m;
}

// where a unit's candidates left go
struct TuOut {
    uint64_t *rec;
    uint32_t *idx;
    unsigned *n;
    uint64_t cap;
    unsigned long long *status;
};

template <int NEXT>
__device__ __forceinline__ void tu_leave(const TuOut &O, uint64_t pos, uint64_t b, uint32_t slot, uint32_t i,
                                         const TcfGeom &G, const TcfPrep &P)
{
    if (pos >= O.cap) {  // more left than the pending list holds
        atomicOr(O.status, ST_INTERNAL);
        return;
    }
    O.idx[pos] = i;
    if (NEXT != TU_NX_IDX) O.rec[pos] = ((NEXT == TU_NX_OTHER ? tu_other(b, slot, i, G, P) : b) << 16) | slot;
}

// A block with many candidates (a hot key): the CTA reads them once per stored
// slot, for the next smallest each time. v: c records, some of them the
// block's; lb: the block inside the unit.
template <int F, bool DEL, int NEXT>
__device__ __noinline__ void tu_hot_block(TuSmem &S, const uint64_t *v, uint32_t c, uint64_t b, uint32_t lb,
                                          const TcfGeom &G, const TcfPrep &P, const TuGeom &U, uint8_t *blocks,
                                          uint8_t *fill, uint32_t cap, const TuOut &O)
{
    constexpr int B = Blk<F>::B;
    __shared__ uint32_t s_tag[B];
    __shared__ uint64_t s_thr[B];
    const uint32_t tsh = U.ibits, bsh = U.ibits + U.sbits, smask = (1u << U.sbits) - 1u, lmask = (1u << U.lbits) - 1u;
    const uint64_t rmask = bsh + U.lbits >= 64 ? ~0ull : (1ull << (bsh + U.lbits)) - 1ull;
    const uint32_t f0 = fill[b];
    Blk<F> blk;
    blk.load(blocks, b);
    auto mine = [&](uint64_t x) { return ((uint32_t)(x >> bsh) & lmask) == lb; };
    // the smallest record of the block that `want` accepts and is above `prev`
    auto next = [&](uint64_t prev, bool any, auto want) {
        uint64_t m = ~0ull;
        for (uint32_t i = threadIdx.x; i < c; i += TU_T) {
            const uint64_t x = v[i] & rmask;
            if (mine(x) && (any || x > prev) && want(x) && x < m) m = x;
        }
        return tu_min(S, m);
    };
    uint32_t used = 0;  // entries of s_tag / s_thr (DEL), accepted records
    uint64_t thr = 0;
    if (!DEL) {
        const uint32_t k = cap > f0 ? cap - f0 : 0u;
        for (uint32_t j = 0; j < k; j++) {
            const uint64_t m = next(thr, j == 0, [](uint64_t) { return true; });
            if (m == ~0ull) break;  // (the same in every thread)
            thr = m;
            used++;
            uint64_t r8[8] = {((thr >> tsh) & smask) << 32, 0, 0, 0, 0, 0, 0, 0};
            blk.merge_new(f0 + j, 1, r8);
        }
        if (used && threadIdx.x == 0) {
            blk.store(blocks, b);
            fill[b] = (uint8_t)(f0 + used);
        }
    } else {
        const uint32_t lm = G.vmask;
        Blk<F> old = blk;
        uint32_t removed = 0;
        bool left = true;  // candidates of the current tag
        uint64_t prev = 0;
        for (uint32_t p = 0; p < f0; p++) {  // a stored copy each; copies of a tag are adjacent
            uint32_t t = 0;
#pragma unroll
            for (int q = 0; q < B; q++)
                if (q == (int)p) t = old.tag(q);
            t &= ~lm;
            const bool again = used > 0 && s_tag[used - 1] == t;
            __syncthreads();
            if (!again) {
                left = true;
                if (threadIdx.x == 0) {
                    s_tag[used] = t;
                    s_thr[used] = 0;  // none matched (a record is never 0: tags are at least 2)
                }
                used++;
            }
            if (left) {
                const uint64_t m = next(prev, !again, [&](uint64_t x) { return ((uint32_t)(x >> tsh) & smask) == t; });
                left = m != ~0ull;
                if (left) {
                    prev = m;
                    if (threadIdx.x == 0) s_thr[used - 1] = m;
                    const uint32_t sm = blk.eq_slots(t, Blk<F>::lane_mask(G.vmask));
                    if (sm) blk.delete_at(__ffs(sm) - 1);
                    removed++;
                }
            }
            __syncthreads();
        }
        if (removed && threadIdx.x == 0) {
            blk.store(blocks, b);
            fill[b] = (uint8_t)(f0 - removed);
        }
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < c; i += TU_T) {
        const uint64_t x = v[i] & rmask;
        if (!mine(x)) continue;
        const uint32_t slot = (uint32_t)(x >> tsh) & smask;
        bool took = !DEL && used && x <= thr;
        if (DEL)
            for (uint32_t d = 0; d < used; d++) took |= s_tag[d] == slot && x <= s_thr[d];
        if (!took) tu_leave<NEXT>(O, atomicAdd(O.n, 1u), b, slot, (uint32_t)x & (uint32_t)((1ull << U.ibits) - 1ull), G, P);
    }
    __syncthreads();
}

// Inserts a tag into the sorted tags of a 16-bit block, all lanes less one, so
// that empty ones are the largest: lane i becomes max(lane i - 1, min(lane i,
// tag)). tt: the tag less one in both lanes.
__device__ __forceinline__ void insert_tag16(uint32_t (&w)[8], uint32_t tt)
{
#pragma unroll
    for (int q = 7; q >= 0; q--) {
        const uint32_t below = q ? __funnelshift_l(w[q - 1], w[q], 16) : w[0] << 16;
        uint32_t m;
        asm("min.u16x2 %0, %1, %2;" : "=r"(m) : "r"(w[q]), "r"(tt));
        asm("max.u16x2 %0, %1, %2;" : "=r"(w[q]) : "r"(m), "r"(below));
    }
}

__device__ __forceinline__ void add_lanes16(uint32_t (&w)[8], uint32_t x)
{
#pragma unroll
    for (int q = 0; q < 8; q++) asm("add.u16x2 %0, %0, %1;" : "+r"(w[q]) : "r"(x));
}

// Removes the first lane whose tag part (lm) is tt's from the sorted lanes of a
// 16-bit block (EMPTY ones last): lanes of at least that tag take the next one.
__device__ __forceinline__ bool remove_tag16(uint32_t (&w)[8], uint32_t tt, uint32_t lm)
{
    uint32_t none = 0x00010001u;  // a half is 0 once a lane of it matched
#pragma unroll
    for (int q = 0; q < 8; q++) {
        uint32_t m;
        asm("min.u16x2 %0, %1, %2;" : "=r"(m) : "r"((w[q] & lm) ^ tt), "r"(0x00010001u));
        none &= m;
    }
    if (none == 0x00010001u) return false;
#pragma unroll
    for (int q = 0; q < 8; q++) {
        const uint32_t x = w[q] & lm, next = q < 7 ? __funnelshift_r(w[q], w[q + 1], 16) : w[7] >> 16;
        uint32_t m;
        asm("max.u16x2 %0, %1, %2;" : "=r"(m) : "r"(x), "r"(tt));
        asm("min.u16x2 %0, %1, %2;" : "=r"(m) : "r"(m - x), "r"(0x00010001u));  // 1: below the tag
        m *= 0xffffu;
        w[q] = (w[q] & m) | (next & ~m);
    }
    return true;
}

// The steps of bucket [s, e) of S.a by one thread, block by block in ascending
// order (ONE: a bucket is a block). Insert: the candidates that fit under
// `cap`, smallest first, join the sorted block; their order matters only where
// some do not fit. Remove: each candidate, smallest first, takes the first copy
// of its tag. Those left are listed in S.left. Returns the algorithmic bytes
// (64 per block changed, 32 per block only read, 2 per fill).
template <int F, bool DEL, bool ONE, bool MANY = false>
__device__ __forceinline__ uint32_t tu_bucket(TuSmem &S, uint32_t s, uint32_t e, uint32_t lb, uint64_t b0,
                                              const TcfGeom &G, uint32_t tsh, uint32_t bsh, uint32_t smask,
                                              uint8_t *blocks, uint8_t *fill, uint32_t cap)
{
    uint32_t done = 0, bytes = 0;
    do {
        uint32_t m = e - s;  // the block's candidates
        if (!ONE) {
            uint32_t mn = 0xffffffffu;
            for (uint32_t j = s; j < e; j++) {
                const uint32_t x = (uint32_t)(S.a[j] >> bsh);
                if (done == 0 || x > lb) mn = min(mn, x);
            }
            lb = mn;
            m = 0;
            for (uint32_t j = s; j < e; j++) m += (uint32_t)(S.a[j] >> bsh) == lb;
        }
        done += m;
        const uint64_t b = b0 + lb;
        const uint32_t f0 = min((uint32_t)fill[b], (uint32_t)Blk<F>::B);
        Blk<F> blk;
        blk.load(blocks, b);
        bytes += 34;
        auto mine = [&](uint64_t x) { return ONE || (uint32_t)(x >> bsh) == lb; };
        // the smallest of the block's candidates above prev (or of all)
        auto next = [&](uint64_t prev, bool any) {
            uint64_t q = ~0ull;
            for (uint32_t j = s; j < e; j++) {
                const uint64_t x = S.a[j];
                if (mine(x) && (any || x > prev) && x < q) q = x;
            }
            return q;
        };
        if (!DEL) {
            const uint32_t k = cap > f0 ? min(m, cap - f0) : 0u;
            uint64_t thr = 0;
            if (k) {
                if constexpr (F == 16) {
                    add_lanes16(blk.w, 0xffffffffu);
                    if (k == m) {
                        for (uint32_t j = s; j < e; j++) {
                            const uint64_t x = S.a[j];
                            if (mine(x)) insert_tag16(blk.w, (((uint32_t)(x >> tsh) & smask) - 1) * 0x00010001u);
                        }
                    } else {
                        for (uint32_t at = 0; at < k; at++) {
                            thr = next(thr, at == 0);
                            insert_tag16(blk.w, (((uint32_t)(thr >> tsh) & smask) - 1) * 0x00010001u);
                        }
                    }
                    add_lanes16(blk.w, 0x00010001u);
                } else {
                    for (uint32_t at = 0; at < k; at += 8) {
                        uint64_t r8[8];
#pragma unroll
                        for (uint32_t q = 0; q < 8; q++) {
                            r8[q] = 0;
                            if (at + q < k) {
                                thr = next(thr, at + q == 0);
                                r8[q] = ((thr >> tsh) & smask) << 32;
                            }
                        }
                        blk.merge_new(f0 + at, min(8u, k - at), r8);
                    }
                }
                blk.store(blocks, b);
                fill[b] = (uint8_t)(f0 + k);
                bytes += 32;
            }
            if (k < m) {
                uint32_t pos = atomicAdd(&S.nleft, m - k);
                for (uint32_t j = s; j < e; j++) {
                    const uint64_t x = S.a[j];
                    if (mine(x) && (k == 0 || x > thr)) S.left[pos++] = (uint16_t)j;
                }
            }
        } else {
            uint32_t removed = 0;
            uint64_t prev = 0;
            for (uint32_t q = 0; q < m; q++) {
                prev = e - s == 1 ? S.a[s] : next(prev, q == 0);
                const uint32_t tag = (uint32_t)(prev >> tsh) & smask, lm = Blk<F>::lane_mask(G.vmask);
                bool hit;
                if constexpr (F == 16) {
                    hit = remove_tag16(blk.w, tag * 0x00010001u, lm);
                } else {
                    const uint32_t sm = blk.eq_slots(tag, lm);
                    hit = sm != 0;
                    if (hit) blk.delete_at(__ffs(sm) - 1);
                }
                if (hit) {
                    removed++;
                } else if constexpr (MANY) {  // no copy left: nor for the others of this tag
                    uint64_t last = prev;
                    for (uint32_t j = s; j < e; j++) {
                        const uint64_t x = S.a[j];
                        if (!mine(x) || x < prev || ((uint32_t)(x >> tsh) & smask) != tag) continue;
                        S.left[atomicAdd(&S.nleft, 1u)] = (uint16_t)j;
                        q += x != prev;
                        last = x > last ? x : last;
                    }
                    prev = last;
                } else {
                    uint32_t j = s;
                    while (S.a[j] != prev) j++;
                    S.left[atomicAdd(&S.nleft, 1u)] = (uint16_t)j;
                }
            }
            if (removed) {
                blk.store(blocks, b);
                fill[b] = (uint8_t)(f0 - removed);
                bytes += 32;
            }
        }
    } while (!ONE && done < e - s);
    return bytes;
}

// the candidates that a unit's steps left in S.left, with one reservation
template <int NEXT>
__device__ __forceinline__ void tu_emit(TuSmem &S, const TuOut &O, uint64_t b0, const TcfGeom &G, const TcfPrep &P,
                                        const TuGeom &U)
{
    const uint32_t nleft = S.nleft;
    if (threadIdx.x == 0 && nleft) S.base = atomicAdd(O.n, nleft);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < nleft; i += TU_T) {
        const uint64_t x = S.a[S.left[i]];
        tu_leave<NEXT>(O, (uint64_t)S.base + i, b0 + (x >> (U.ibits + U.sbits)),
                       (uint32_t)(x >> U.ibits) & ((1u << U.sbits) - 1u), (uint32_t)(x & ((1ull << U.ibits) - 1ull)), G, P);
    }
}

// the arguments of a phase's steps (a kernel parameter that functions out of
// line read in place)
struct TuStep {
    TcfGeom G;
    TcfPrep P;
    TuGeom U;
    uint8_t *blocks, *fill;
    const uint32_t *ust;   // the units' first records
    uint32_t nunits, cap;
    const uint64_t *v;     // records by unit
    TuOut O;
    TuSrc src;
    const unsigned *uneven;  // set: no phase goes by unit
    unsigned long long *units;
};

// a remove's steps of a bucket of many candidates
template <int F, bool ONE>
__device__ __noinline__ uint32_t tu_bucket_many(TuSmem &S, uint32_t s, uint32_t e, uint32_t lb, uint64_t b0, const TuStep &A)
{
    const uint32_t tsh = A.U.ibits, bsh = A.U.ibits + A.U.sbits, smask = (1u << A.U.sbits) - 1u;
    return tu_bucket<F, true, ONE, true>(S, s, e, lb, b0, A.G, tsh, bsh, smask, A.blocks, A.fill, A.cap);
}

// the hot buckets in S.hot, by the whole CTA, block by block
template <int F, bool DEL, int NEXT>
__device__ __noinline__ void tu_hot_buckets(TuSmem &S, const TuStep &A, uint64_t b0)
{
    const uint32_t bsh = A.U.ibits + A.U.sbits;
    const uint16_t *first = reinterpret_cast<const uint16_t *>(S.cnt);
    for (uint32_t h = 0; h < S.nhot; h++) {
        const uint32_t bk = S.hot[h], s = first[bk], e = first[bk + 1];
        uint64_t last = 0;
        for (bool any = true;; any = false) {
            uint64_t m = ~0ull;
            for (uint32_t j = s + threadIdx.x; j < e; j += TU_T) {
                const uint64_t x = S.a[j] >> bsh;
                if ((any || x > last) && x < m) m = x;
            }
            last = tu_min(S, m);
            if (last == ~0ull) break;
            tu_hot_block<F, DEL, NEXT>(S, S.a + s, e - s, b0 + last, (uint32_t)last, A.G, A.P, A.U, A.blocks, A.fill, A.cap,
                                       A.O);
        }
    }
    __syncthreads();
}

// A unit with more candidates than fit: ranges of blocks that do, found by
// counting, take the same steps; a block that alone has more goes by the CTA.
template <int F, bool DEL, int NEXT>
__device__ __noinline__ void tu_big_unit(TuSmem &S, const TuStep &A, uint32_t unit)
{
    const TuGeom &U = A.U;
    const uint32_t tsh = U.ibits, bsh = U.ibits + U.sbits, smask = (1u << U.sbits) - 1u, lmask = (1u << U.lbits) - 1u;
    const uint64_t rmask = bsh + U.lbits >= 64 ? ~0ull : (1ull << (bsh + U.lbits)) - 1ull;
    const uint32_t bkshift = bsh + (U.lbits > TU_BBITS ? U.lbits - TU_BBITS : 0u);
    const uint16_t *first = reinterpret_cast<const uint16_t *>(S.cnt);
    const uint64_t b0 = (uint64_t)unit << U.lbits;
    const uint64_t *w = A.v + A.ust[unit];
    const uint32_t all = A.ust[unit + 1] - A.ust[unit], end = 1u << U.lbits;
    uint32_t lo = 0, range = end;
    while (lo < end) {
        uint32_t n = 0;
        while (true) {
            uint32_t m = 0;
            for (uint32_t i = threadIdx.x; i < all; i += TU_T) m += ((uint32_t)(w[i] >> bsh) & lmask) - lo < range;
            const uint32_t before = cta_scan<TU_T>(m, S.warp);
            if (threadIdx.x == TU_T - 1) S.base = before + m;
            __syncthreads();
            n = S.base;
            __syncthreads();
            if (n <= TU_CAP || range == 1) break;
            range >>= 1;
        }
        if (n > TU_CAP) {
            tu_hot_block<F, DEL, NEXT>(S, w, all, b0 + lo, lo, A.G, A.P, U, A.blocks, A.fill, A.cap, A.O);
        } else if (n) {
            if (threadIdx.x == 0) S.base = S.nleft = S.nhot = 0;
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < all; i += TU_T)
                if (((uint32_t)(w[i] >> bsh) & lmask) - lo < range) S.a[atomicAdd(&S.base, 1u)] = w[i] & rmask;
            __syncthreads();
            uint64_t key[TU_PER];
#pragma unroll
            for (int r = 0; r < TU_PER; r++)
                if (r * TU_T + threadIdx.x < n) key[r] = S.a[r * TU_T + threadIdx.x];
            tu_group(S, key, n, bkshift);
            for (uint32_t h = threadIdx.x; h < S.nhead; h += TU_T) {
                const uint32_t bk = S.head[h], s = first[bk], e = first[bk + 1];
                if (e - s > TU_HOT) S.hot[atomicAdd(&S.nhot, 1u)] = (uint16_t)bk;
                else if (DEL && e - s > TU_MANY) tu_bucket_many<F, false>(S, s, e, bk, b0, A);
                else tu_bucket<F, DEL, false>(S, s, e, bk, b0, A.G, tsh, bsh, smask, A.blocks, A.fill, A.cap);
            }
            __syncthreads();
            tu_emit<NEXT>(S, A.O, b0, A.G, A.P, U);
            tu_hot_buckets<F, DEL, NEXT>(S, A, b0);
        }
        lo += range;
        while (range < end && lo % (2 * range) == 0) range <<= 1;  // wider again where it may be
    }
}

// One CTA per unit (staying for more, the next one's records on their way):
// group the candidates by block, then a thread per block with candidates takes
// its step. units: algorithmic bytes (tu_bucket's, 8 per candidate read, 12 per
// candidate left). Bound by instructions and the latency of the blocks' loads:
// 2^22 candidates on 2^22 blocks 81 us, 2^24 on 2^24 291 us (3.7 TB/s of
// algorithmic bytes).
template <int F, bool DEL, int NEXT, bool ONE>
__global__ void __launch_bounds__(TU_T, 3) tcf_unit_step(const __grid_constant__ TuStep A)
{
    if (tu_count(A.src) == 0 || (A.uneven && *A.uneven)) return;
    __shared__ __align__(16) TuSmem S;
    const uint32_t tsh = A.U.ibits, bsh = A.U.ibits + A.U.sbits, smask = (1u << A.U.sbits) - 1u;
    const uint64_t rmask = bsh + A.U.lbits >= 64 ? ~0ull : (1ull << (bsh + A.U.lbits)) - 1ull;
    const uint32_t bkshift = ONE ? bsh : bsh + A.U.lbits - TU_BBITS;
    const uint16_t *first = reinterpret_cast<const uint16_t *>(S.cnt);
    uint64_t key[TU_PER];
    uint32_t u = blockIdx.x, c = 0;
    unsigned long long total = 0;
    auto fetch = [&] {
        const uint32_t s0 = A.ust[u];
        c = A.ust[u + 1] - s0;
        if (c > TU_CAP) return;
#pragma unroll
        for (int r = 0; r < TU_PER; r++) {
            if (r * TU_T >= c) break;
            if (r * TU_T + threadIdx.x < c) key[r] = __ldcs(A.v + s0 + r * TU_T + threadIdx.x) & rmask;
        }
    };
    if (u < A.nunits) fetch();
    while (u < A.nunits) {
        const uint32_t unit = u, n = c;
        const uint64_t b0 = (uint64_t)unit << A.U.lbits;
        u += gridDim.x;
        if (n == 0) {
            if (u < A.nunits) fetch();
            continue;
        }
        __syncthreads();  // everything of the last unit is done
        if (n > TU_CAP) {
            tu_big_unit<F, DEL, NEXT>(S, A, unit);
            if (u < A.nunits) fetch();
            continue;
        }
        if (threadIdx.x == 0) S.nleft = S.nhot = 0;
        tu_group(S, key, n, bkshift);
        if (u < A.nunits) fetch();  // the next unit's records
        const uint32_t heads = S.nhead;
        uint32_t bytes = 0;
        for (uint32_t h = threadIdx.x; h < heads; h += TU_T) {
            const uint32_t bk = S.head[h], s = first[bk], e = first[bk + 1];
            if (e - s > TU_HOT) S.hot[atomicAdd(&S.nhot, 1u)] = (uint16_t)bk;
            else if (DEL && e - s > TU_MANY) bytes += tu_bucket_many<F, ONE>(S, s, e, bk, b0, A);
            else bytes += tu_bucket<F, DEL, ONE>(S, s, e, bk, b0, A.G, tsh, bsh, smask, A.blocks, A.fill, A.cap);
        }
        __syncthreads();
        if (A.units) total += bytes + (threadIdx.x == 0 ? 8ull * n + 12ull * S.nleft : 0ull);
        tu_emit<NEXT>(S, A.O, b0, A.G, A.P, A.U);
        if (S.nhot) tu_hot_buckets<F, DEL, NEXT>(S, A, b0);
    }
    if (A.units) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) total += __shfl_down_sync(0xffffffffu, total, o);
        if ((threadIdx.x & 31) == 0 && total) atomicAdd(A.units, total);
    }
}

// ---------------------------------------------------------------------------
// Point mode (Alg. 1)
// ---------------------------------------------------------------------------
template <int F>
__device__ bool point_put(uint8_t *blocks, uint64_t b, uint32_t t, DevCounters *ctr)
{
    constexpr int B = Blk<F>::B;
    for (int attempt = 0; attempt < 4 * B; attempt++) {
        Blk<F> blk;
        blk.load_l2(blocks, b);
        int s = -1;
#pragma unroll
        for (int p = 0; p < B; p++)
            if (s < 0 && blk.tag(p) < 2) s = p;
        if (s < 0) return false;
        uint32_t seen = blk.tag(s);
        if (F == 16) {
            unsigned short *slot = reinterpret_cast<unsigned short *>(blocks + b * 32) + s;
            if (atomicCAS(slot, (unsigned short)seen, (unsigned short)t) == (unsigned short)seen) return true;
        } else {
            unsigned int *word = reinterpret_cast<unsigned int *>(blocks + b * 32) + (s >> 2);
            unsigned sh = (s & 3) * 8;
            unsigned int cur = blk.w[s >> 2];
            unsigned int want = (cur & ~(0xffu << sh)) | (t << sh);
            if (atomicCAS(word, cur, want) == cur) return true;
        }
    }
    atomicOr(&ctr->status, ST_TIMEOUT);
    return false;
}

template <int F>
__device__ bool point_take(uint8_t *blocks, uint64_t b, uint32_t t, uint32_t vmask, DevCounters *ctr)
{
    constexpr int B = Blk<F>::B;
    for (int attempt = 0; attempt < 4 * B; attempt++) {
        Blk<F> blk;
        blk.load_l2(blocks, b);
        int s = -1;
#pragma unroll
        for (int p = 0; p < B; p++)
            if (s < 0 && (blk.tag(p) & ~vmask) == t) s = p;
        if (s < 0) return false;
        if (F == 16) {
            unsigned short *slot = reinterpret_cast<unsigned short *>(blocks + b * 32) + s;
            const unsigned short seen = (unsigned short)blk.tag(s);
            if (atomicCAS(slot, seen, (unsigned short)1) == seen) return true;
        } else {
            unsigned int *word = reinterpret_cast<unsigned int *>(blocks + b * 32) + (s >> 2);
            unsigned sh = (s & 3) * 8;
            unsigned int cur = blk.w[s >> 2];
            unsigned int want = (cur & ~(0xffu << sh)) | (1u << sh);
            if (atomicCAS(word, cur, want) == cur) return true;
        }
    }
    atomicOr(&ctr->status, ST_TIMEOUT);
    return false;
}

template <int F>
__global__ void __launch_bounds__(TPB) tcf_point_insert(const uint64_t *__restrict__ keys,
                                                        const uint8_t *__restrict__ vals, uint64_t n, TcfGeom G,
                                                        uint8_t *blocks, uint64_t *bk, uint8_t *status,
                                                        DevCounters *ctr)
{
    for (uint64_t i = blockIdx.x * (uint64_t)TPB + threadIdx.x; i < n; i += (uint64_t)gridDim.x * TPB) {
        KeyInfo k = tcf_keyinfo(keys[i], G);
        if (vals) k.t |= vals[i] & G.vmask;
        Blk<F> x;
        x.load_l2(blocks, k.b1);
        int f1 = x.live();
        bool done = false;
        if (f1 < (int)G.tsc) done = point_put<F>(blocks, k.b1, k.t, ctr);  // shortcut (Sec. 4.1)
        if (!done) {
            Blk<F> y;
            y.load_l2(blocks, k.b2);
            x.load_l2(blocks, k.b1);
            uint64_t first = x.live() <= y.live() ? k.b1 : k.b2;
            done = point_put<F>(blocks, first, k.t, ctr) ||
                   point_put<F>(blocks, first == k.b1 ? k.b2 : k.b1, k.t, ctr);
        }
        if (!done) {
            uint64_t e = tcf_entry(k, G.f);
            unsigned long long *p =
                reinterpret_cast<unsigned long long *>(bk + tcf_bucket_of(e, G) * BK_W);
            for (int s = 0; s < (int)BK_W && !done; s++)
                if (atomicCAS(p + s, 0ull, (unsigned long long)e) == 0ull) done = true;
            if (done) atomicAdd(&ctr->backing, 1ull);
        }
        if (!done) {
            if (status) status[i] = FILTER_KEY_FULL;
            atomicAdd(&ctr->failed, 1ull);
            atomicOr(&ctr->status, ST_FULL);
        } else if (status) {
            status[i] = FILTER_KEY_OK;
        }
    }
}

template <int F>
__global__ void __launch_bounds__(TPB) tcf_point_remove(const uint64_t *__restrict__ keys, uint64_t n, TcfGeom G,
                                                        uint8_t *blocks, uint64_t *bk, uint8_t *status,
                                                        DevCounters *ctr)
{
    for (uint64_t i = blockIdx.x * (uint64_t)TPB + threadIdx.x; i < n; i += (uint64_t)gridDim.x * TPB) {
        KeyInfo k = tcf_keyinfo(keys[i], G);
        bool done = point_take<F>(blocks, k.b1, k.t, G.vmask, ctr) || point_take<F>(blocks, k.b2, k.t, G.vmask, ctr);
        if (!done) {
            const uint64_t e = tcf_entry(k, G.f), em = ~(uint64_t)G.vmask;
            unsigned long long *p =
                reinterpret_cast<unsigned long long *>(bk + tcf_bucket_of(e, G) * BK_W);
            for (int s = 0; s < (int)BK_W && !done; s++) {
                const unsigned long long v = __ldcg(p + s);
                if ((v & em) == e && atomicCAS(p + s, v, 0ull) == v) done = true;
            }
            if (done) atomicAdd(&ctr->backing, (unsigned long long)-1ll);
        }
        if (status) status[i] = done ? FILTER_KEY_OK : FILTER_KEY_NOT_FOUND;
    }
}

// fill bytes and backing count from the table image (after import)
template <int F>
__global__ void tcf_refill(TcfGeom G, const uint8_t *blocks, uint8_t *fill)
{
    for (uint64_t b = blockIdx.x * (uint64_t)TPB + threadIdx.x; b < G.nb; b += (uint64_t)gridDim.x * TPB) {
        Blk<F> x;
        x.load(blocks, b);
        fill[b] = (uint8_t)x.nonzero();
    }
}

__global__ void tcf_count_backing(TcfGeom G, const uint64_t *bk, DevCounters *ctr)
{
    unsigned long long c = 0;
    for (uint64_t j = blockIdx.x * (uint64_t)TPB + threadIdx.x; j < G.nbk * BK_W; j += (uint64_t)gridDim.x * TPB)
        c += bk[j] != 0;
    if (c) atomicAdd(&ctr->backing, c);
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
int tcf_setup(filter *F, uint64_t &table_bytes, uint64_t &scratch_bytes, bool plan_only)
{
    const filter_config &c = F->cfg;
    if (c.tag_bits != 8 && c.tag_bits != 12 && c.tag_bits != 16) return FILTER_ERR_ARG;
    if (c.value_bits > c.tag_bits / 2 || c.value_bits > 7) return FILTER_ERR_ARG;
    if (c.mode != FILTER_MODE_BULK && c.mode != FILTER_MODE_POINT) return FILTER_ERR_ARG;
    const uint32_t B = c.block_slots ? c.block_slots : 256 / c.tag_bits;
    TcfState &T = F->tcf;
    T.G.f = c.tag_bits;
    T.G.B = B;
    if (tcf_custom(T.G) && (!tcf_geom_supported(c.tag_bits, B) || c.mode != FILTER_MODE_BULK || c.value_bits))
        return FILTER_ERR_ARG;
    // nb: the largest power of two with nb B <= 2^log2_slots
    uint32_t lb = 0;
    while ((1ull << lb) < B) lb++;  // ceil(log2 B)
    if (c.log2_slots < lb + 1 || c.log2_slots > lb + 32) return FILTER_ERR_ARG;
    T.mode = c.mode;
    T.G.bbytes = (c.tag_bits * B + 255) / 256 * 32;
    T.G.tsc = 3 * B / 4;
    T.G.tmask = (1u << (c.tag_bits - c.value_bits)) - 1u;
    T.G.vbits = c.value_bits;
    T.G.vmask = (1u << c.value_bits) - 1u;
    T.G.nb = 1ull << (c.log2_slots - lb);
    T.G.seed = c.hash_seed;
    const uint64_t N = T.G.nb * B;
    uint64_t cap = (N + 99) / 100;
    T.G.nbk = (cap + BK_W - 1) / BK_W;
    if (T.G.nbk < 8) T.G.nbk = 8;
    const uint64_t M = c.max_batch ? c.max_batch : 1;
    if (M > 0xffffffffull) return FILTER_ERR_ARG;
    const uint64_t groups = (T.G.nb > T.G.nbk ? T.G.nb : T.G.nbk) + 1;
    // every buffer is listed once: the same list sizes the arena (plan) and
    // carves it (allocation); the table comes first
    uint64_t bytes = 0;
    Arena &A = F->arena;
    auto piece = [&](auto *&ptr, uint64_t count) {
        using T_ = typename std::remove_reference<decltype(*ptr)>::type;
        const uint64_t b = (count * sizeof(T_) + 255) & ~255ull;
        bytes += b;
        if (!plan_only) ptr = A.take<T_>(count);
    };
    piece(T.blocks, T.G.nb * T.G.bbytes);
    piece(T.bk, T.G.nbk * BK_W);
    piece(T.fill, T.G.nb);
    table_bytes = bytes;
    piece(T.cnt, groups);
    piece(T.off, groups);
    piece(T.rec, M);
    piece(T.pend0, M);
    piece(T.pend1, M);
    piece(T.pend2, M);
    piece(T.tlist, M);
    piece(T.tcount, (uint64_t)sm_count() * 8);
    piece(T.dlist, M);
    piece(T.seg, M);
    piece(T.tcur, tcf_unit_words(M));
    piece(T.pb, M);
    piece(T.pbi, M);
    piece(F->scan_tmp, scan_tmp_words(groups));
    scratch_bytes = bytes - table_bytes;
    return FILTER_OK;
}

int tcf_clear(filter *F, cudaStream_t st)
{
    TcfState &T = F->tcf;
    const uint64_t groups = (T.G.nb > T.G.nbk ? T.G.nb : T.G.nbk) + 1;
    GF_CUDA(cudaMemsetAsync(T.blocks, 0, T.G.nb * T.G.bbytes, st));
    GF_CUDA(cudaMemsetAsync(T.bk, 0, T.G.nbk * BK_W * 8, st));
    GF_CUDA(cudaMemsetAsync(T.fill, 0, T.G.nb, st));
    GF_CUDA(cudaMemsetAsync(T.cnt, 0, groups * 4, st));
    GF_CUDA(cudaMemsetAsync(T.tcur, 0, tu_scratch(nullptr, F->cfg.max_batch).zero_words * 4, st));
    GF_CUDA(cudaMemsetAsync(F->ctr, 0, sizeof(DevCounters), st));
    return FILTER_OK;
}

// Everything one bulk call touches: a filter's own table, or for a group the
// concatenated arrays of all members (G.nb and G.nbk are then the totals)
// with the keys prepared per member.
struct TcfBulk {
    TcfGeom G;
    uint8_t *blocks;
    uint64_t *bk;
    uint8_t *fill;
    uint32_t *cnt, *off;
    uint64_t *rec;
    uint32_t *pend0;
    uint64_t *pend1;
    uint32_t *pend2;
    uint32_t *tlist, *tcount, *dlist;
    uint64_t *seg;
    uint64_t max_n;  // entries of every per-key scratch list (max_batch)
    uint32_t tile_target;  // unit path: most candidates per unit on average
    uint32_t *tcur;  // unit phases: the partition's scratch
    uint64_t *pb;    // unit phases: the second pending list
    uint32_t *pbi;
    uint64_t *scan_tmp;
    DevCounters *ctr;
    TcfPrep prep;
    unsigned *uneven;  // unit path: where the call's keys turned out too uneven for it (null: not asked)
};

static TcfBulk bulk_of(const TcfState &T, uint64_t *scan_tmp, DevCounters *ctr, const TcfPrep &prep, uint64_t max_n,
                       const filter_tuning &tune)
{
    TcfBulk W;
    W.max_n = max_n;
    W.tile_target = tcf_tile_target(tune);
    W.G = T.G;
    W.blocks = T.blocks;
    W.bk = T.bk;
    W.fill = T.fill;
    W.cnt = T.cnt;
    W.off = T.off;
    W.rec = T.rec;
    W.pend0 = T.pend0;
    W.pend1 = T.pend1;
    W.pend2 = T.pend2;
    W.tlist = T.tlist;
    W.tcount = T.tcount;
    W.dlist = T.dlist;
    W.seg = T.seg;
    W.tcur = T.tcur;
    W.pb = T.pb;
    W.pbi = T.pbi;
    W.scan_tmp = scan_tmp;
    W.ctr = ctr;
    W.prep = prep;
    W.uneven = nullptr;
    return W;
}

// CTAs of the grouping launches of a phase (the same for histogram and
// segment allocation, whose chunks must agree)
static int group_grid(uint64_t n) { return grid_for(n, TPB, 8); }

// Groups one phase's candidates by destination. The first phase of a call
// (all keys, most blocks hit) is dense: per-destination counts, an exclusive
// scan over all destinations, then the scatter. Later phases see few
// candidates and are sparse: only the touched destinations get a segment and
// a list entry (slot: the phase's counters), so their per-destination kernel
// visits those alone. `recI` (bucket phases) receives the batch indices. gate: a
// word on the device without which the kernels do nothing (null: always).
template <int SRC, int DST>
static PhaseDst group_phase(const TcfBulk &T, const uint64_t *keys, uint64_t n, const void *pend,
                            const unsigned *npend, int slot, uint32_t *recI, cudaStream_t st,
                            const unsigned *gate = nullptr)
{
    const TcfGeom G = T.G;
    const int gk = group_grid(n);
    constexpr bool SPARSE = SRC != SRC_KEYS;
    const uint64_t ndst = (DST == DST_BUCKET ? G.nbk : G.nb);
    PhaseDst P{nullptr, nullptr, nullptr, nullptr};
    {
        gf::TraceScope ts_(SPARSE ? "tcf_group_hist_sparse" : "tcf_group_hist", n, st, SPARSE);
        tcf_group_hist<SRC, DST, SPARSE><<<gk, TPB, 0, st>>>(keys, T.prep, n, pend, npend, G, T.fill, T.cnt, T.tlist,
                                                             T.tcount, gate, ts_.units());
    }
    if (SPARSE) {
        gf::TraceScope ts_("tcf_alloc", 0, st, true);
        tcf_alloc<<<gk, TPB, 0, st>>>(npend, n, T.tlist, T.tcount, T.cnt, T.off, T.dlist, T.seg, &T.ctr->cursor[slot],
                                      &T.ctr->touched[slot], ts_.units());
        P.dlist = T.dlist;
        P.seg = T.seg;
        P.nlist = &T.ctr->touched[slot];
    } else {
        exclusive_scan_u32(T.cnt, T.off, ndst + 1, T.scan_tmp, T.ctr, st, gate);
        P.off = T.off;
    }
    {
        gf::TraceScope ts_(SPARSE ? "tcf_group_scatter_sparse" : "tcf_group_scatter", n, st, SPARSE);
        tcf_group_scatter<SRC, DST><<<gk, TPB, 0, st>>>(keys, T.prep, n, pend, npend, G, T.fill, T.cnt, T.off, T.rec,
                                                        recI, gate, ts_.units());
    }
    return P;
}

// per-destination grid: dense phases visit every destination, sparse ones at
// most one per candidate
static int dst_grid(const PhaseDst &P, uint64_t n, uint64_t ndst)
{
    return grid_for(P.dlist ? (n < ndst ? n : ndst) : ndst, TPB, 8);
}

// ---------------------------------------------------------------------------
// Other block geometries (Sec. 4.1: blocks sized up to a cache line and
// beyond; Sec. 4.2: the bulk TCF's 128-slot blocks; Sec. 4: 12-bit tags that
// straddle word boundaries). A block is B slots of F bits packed
// little-endian into whole 32-byte sectors (gf_packed.cuh); the phases and
// their grouping are the ones above, only the per-block steps and the query
// read and write packed slots.
//
// A block's step is shared by 4, 8 or 16 lanes: its words and candidates go
// through shared memory, each candidate ranks itself among the others and finds
// its slot by binary search, and a bit map of the new (or removed) slots tells
// each lane what its slots of the new block hold. Bound by instructions; a
// thread per block kept the candidate and tag lists (up to 4 KB) in local
// memory. 128 slots of 16 bits, 2^22 slots: the block steps of removing half in
// four batches 1822 us with threads, 153 with the lanes; of eight inserts to
// 90 % 398 and 212 us.
// ---------------------------------------------------------------------------
template <int F, int B>
struct GBlk : Packed<F, B> {
    using Packed<F, B>::w;
    static constexpr int WORDS = Packed<F, B>::WORDS;
    static constexpr int BYTES = WORDS * 4;
    static_assert(BYTES % 32 == 0, "whole sectors");
    static constexpr int LANES = B <= 32 ? 4 : (B <= 64 ? 8 : 16);  // that share a block's step
    static constexpr uint32_t CAND = 8 * LANES;                      // candidates the step stages

    __device__ __forceinline__ void load(const uint8_t *blocks, uint64_t b, bool ro)
    {
        const uint4 *p = reinterpret_cast<const uint4 *>(blocks + b * BYTES);
#pragma unroll
        for (int k = 0; k < WORDS / 4; k++) {
            const uint4 v = ro ? __ldg(p + k) : p[k];
            w[4 * k] = v.x;
            w[4 * k + 1] = v.y;
            w[4 * k + 2] = v.z;
            w[4 * k + 3] = v.w;
        }
    }
    __device__ __forceinline__ void store(uint8_t *blocks, uint64_t b) const
    {
        uint4 *p = reinterpret_cast<uint4 *>(blocks + b * BYTES);
#pragma unroll
        for (int k = 0; k < WORDS / 4; k++) p[k] = make_uint4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
    }
    // some slot holds tag t (t >= 2; the bits past the last slot are 0)
    __device__ __forceinline__ bool has(uint32_t t) const
    {
        if constexpr (F == 16 || F == 8) {
            const uint32_t tt = F == 16 ? (t | (t << 16)) : t * 0x01010101u;
            uint32_t m = 0;
#pragma unroll
            for (int k = 0; k < WORDS; k++) m |= F == 16 ? __vcmpeq2(w[k], tt) : __vcmpeq4(w[k], tt);
            return m != 0;
        } else {
            for (int s = 0; s < B; s++)
                if (this->get(s) == t) return true;
            return false;
        }
    }
};

// entries of the ascending v[0 .. n) below t
template <class Get>
__device__ __forceinline__ uint32_t count_below(uint32_t n, uint32_t t, Get v)
{
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (v(mid) < t) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The steps of a block with more candidates than its lanes stage (a hot key),
// by one thread: insert returns the largest accepted record; remove passes the
// unmatched on itself
template <int F, int B>
__device__ __noinline__ uint64_t gblock_insert_many(uint8_t *blocks, uint64_t b, uint32_t f0, uint32_t k,
                                                    const uint64_t *rec, uint32_t cnt)
{
    uint64_t a[B];
    int have = 0;
    for (uint32_t q = 0; q < cnt; q++) have = topk_push(a, have, (int)k, rec[q]);
    uint32_t nv[B];
    for (uint32_t q = 0; q < k; q++) nv[q] = (uint32_t)(a[q] >> 32);
    GBlk<F, B> blk;
    blk.load(blocks, b, false);
    blk.merge_sorted((int)f0, nv, (int)k);
    blk.store(blocks, b);
    return a[k - 1];
}

template <int F, int B>
__device__ __noinline__ uint32_t gblock_remove_many(uint8_t *blocks, uint64_t b, uint32_t f0, const uint64_t *rec,
                                                    uint32_t cnt, uint32_t *pend32, unsigned *npend)
{
    uint32_t dt[B], dc[B], used[B], removed = 0;
    uint64_t thr[B];
    int ndt = 0;
    GBlk<F, B> blk;
    blk.load(blocks, b, false);
    for (int p = 0; p < (int)f0; p++) {  // copies of a tag are adjacent
        const uint32_t t = blk.get(p);
        if (ndt > 0 && dt[ndt - 1] == t) {
            dc[ndt - 1]++;
        } else {
            dt[ndt] = t;
            dc[ndt] = 1;
            ndt++;
        }
    }
    for (int d = 0; d < ndt; d++) {
        uint64_t a[B];
        int have = 0;
        const uint64_t lo = (uint64_t)dt[d] << 32, hi = lo | 0xffffffffull;
        for (uint32_t q = 0; q < cnt; q++)
            if (rec[q] >= lo && rec[q] <= hi) have = topk_push(a, have, (int)dc[d], rec[q]);
        used[d] = (uint32_t)have;
        thr[d] = have ? a[have - 1] : 0;
        removed += (uint32_t)have;
    }
    if (removed) {
        GBlk<F, B> out;
        out.clear();
        int o = 0;
        for (int d = 0; d < ndt; d++)
            for (uint32_t c = used[d]; c < dc[d]; c++) out.set(o++, dt[d]);
        out.store(blocks, b);
    }
    if (removed < cnt) {
        uint32_t slot = atomicAdd(npend, cnt - removed);
        for (uint32_t q = 0; q < cnt; q++) {
            const uint32_t t = (uint32_t)(rec[q] >> 32);
            bool matched = false;
            for (int d = 0; d < ndt; d++)
                if (dt[d] == t && used[d] > 0 && rec[q] <= thr[d]) matched = true;
            if (!matched) pend32[slot++] = (uint32_t)rec[q];
        }
    }
    return f0 - removed;
}

// One phase over its blocks. Insert (DEL = false): the k smallest (tag, index)
// candidates that fit under `cap` join the block; rejects go on as in
// tcf_block_insert. Remove: per tag, the smallest candidates take one copy
// each; the unmatched go on.
template <int F, int B, bool DEL>
__global__ void __launch_bounds__(TPB) tcf_gblock_step(TcfGeom G, uint8_t *blocks, uint8_t *fill, PhaseDst P,
                                                       const uint64_t *__restrict__ rec, int phase, uint32_t cap,
                                                       uint32_t *pend32, uint64_t *pend64, unsigned *npend,
                                                       unsigned long long *units)
{
    using Blk = GBlk<F, B>;
    constexpr int L = Blk::LANES, NG = TPB / L, RM = (B + 31) / 32;
    constexpr uint32_t CAND = Blk::CAND;
    constexpr int S = (B + L - 1) / L;  // slots per lane: gl, gl + L, ..
    __shared__ uint64_t s_rec[NG][CAND];
    __shared__ __align__(16) Blk s_blk[NG];
    constexpr bool BYTEWISE = F == 8 || F == 16;  // the new block's slots are its words
    using Slot = typename std::conditional<F == 8, uint8_t, uint16_t>::type;
    __shared__ uint16_t s_new[NG][B];
    __shared__ __align__(16) Slot s_out[NG][BYTEWISE ? Blk::BYTES / sizeof(Slot) : B];
    __shared__ uint32_t s_map[NG][RM];  // insert: the new slots; remove: the removed ones
    const int gl = threadIdx.x % L, g = threadIdx.x / L;
    const uint64_t nd = phase_count(P, G.nb);
    if (P.dlist) note_units(units, nd);  // units: blocks with candidates
    const uint64_t stride = (uint64_t)gridDim.x * NG;
    auto old = [&](uint32_t i) -> uint32_t {
        if constexpr (F == 16) return reinterpret_cast<const uint16_t *>(s_blk[g].w)[i];
        else if constexpr (F == 8) return reinterpret_cast<const uint8_t *>(s_blk[g].w)[i];
        else return s_blk[g].get((int)i);
    };
    auto fresh = [&](uint32_t i) { return (uint32_t)s_new[g][i]; };
    if (BYTEWISE)
        for (int i = B + gl; i < Blk::BYTES / (int)sizeof(Slot); i += L) s_out[g][i] = 0;  // past the last slot
    // whole warps step together: a warp's lanes all reach its barriers
    for (uint64_t j0 = blockIdx.x * (uint64_t)NG + (threadIdx.x & ~31u) / L; j0 < nd; j0 += stride) {
        const uint64_t j = j0 + (threadIdx.x & 31) / L;
        uint32_t s = 0, e = 0, f0 = 0, k = 0;
        uint64_t b = 0;
        if (j < nd) b = phase_dst(P, j, s, e);
        const uint32_t cnt = e - s;
        const bool staged = cnt > 0 && cnt <= CAND;
        uint64_t r[8];
        uint32_t left = 0;  // bit u: candidate gl + u L goes on
        if (cnt) f0 = fill[b];
        if (staged) {
#pragma unroll
            for (int u = 0; u < 8; u++) {
                if (u * L >= (int)cnt) break;
                const uint32_t q = gl + u * L;
                r[u] = q < cnt ? rec[s + q] : ~0ull;
                if (q < cnt) s_rec[g][q] = r[u];
            }
            for (int w = gl; w < Blk::WORDS / 4; w += L)
                reinterpret_cast<uint4 *>(s_blk[g].w)[w] = reinterpret_cast<const uint4 *>(blocks + b * Blk::BYTES)[w];
            for (int w = gl; w < RM; w += L) s_map[g][w] = 0;
        }
        if (!DEL) k = cap > f0 ? min(cnt, cap - f0) : 0u;
        __syncwarp();
        if (staged) {
#pragma unroll
            for (int u = 0; u < 8; u++) {
                if (u * L >= (int)cnt) break;
                uint32_t rank = 0;  // smaller candidates (DEL: of the same tag)
                for (uint32_t i = 0; i < cnt; i++) {
                    const uint64_t x = s_rec[g][i];
                    rank += x < r[u] && (!DEL || (x >> 32) == (r[u] >> 32));
                }
                if (gl + u * L >= (int)cnt) continue;
                const uint32_t tag = (uint32_t)(r[u] >> 32);
                if (!DEL) {
                    if (rank < k) s_new[g][rank] = (uint16_t)tag;
                    else left |= 1u << u;
                } else {
                    const uint32_t at = count_below(f0, tag, old) + rank;
                    if (at < f0 && old(at) == tag) atomicOr(&s_map[g][at >> 5], 1u << (at & 31));
                    else left |= 1u << u;
                }
            }
        }
        __syncwarp();
        if (!DEL && staged) {
            // an accepted tag lands behind the old ones up to it and the accepted before it
            for (uint32_t i = gl; i < k; i += L) {
                const uint32_t at = i + count_below(f0, fresh(i) + 1, old);
                atomicOr(&s_map[g][at >> 5], 1u << (at & 31));
            }
        }
        __syncwarp();
        uint32_t f1 = f0;  // the new fill
        if (staged) {
            uint32_t map[RM], pre[RM + 1];
            pre[0] = 0;
#pragma unroll
            for (int w = 0; w < RM; w++) {
                map[w] = s_map[g][w];
                pre[w + 1] = pre[w] + __popc(map[w]);
            }
            f1 = DEL ? f0 - pre[RM] : f0 + k;
#pragma unroll
            for (int u = 0; u < S; u++) {
                const int w = u * L / 32;  // the slots of one u share a map word
                const uint32_t i = gl + u * L, m = map[w] >> ((u * L) % 32);
                if (i >= (uint32_t)B) break;
                const uint32_t before = pre[w] + __popc(map[w] & ((1u << (i & 31)) - 1u));
                if (!DEL) {
                    s_out[g][i] = (Slot)(i >= f1 ? 0u : ((m >> gl) & 1u) ? fresh(before) : old(i - before));
                } else {
                    if (i < f0 && !((m >> gl) & 1u)) s_out[g][i - before] = (Slot)old(i);
                    if (i >= f1) s_out[g][i] = 0;
                }
            }
        }
        __syncwarp();
        if (staged && f1 != f0) {
            for (int w = gl; w < Blk::WORDS; w += L) {
                uint32_t x = 0;
                if constexpr (BYTEWISE) {
                    x = reinterpret_cast<const uint32_t *>(s_out[g])[w];
                } else {
                    for (int i = 32 * w / F; i < B && F * i < 32 * (w + 1); i++) {
                        const int o = F * i - 32 * w;
                        x |= o >= 0 ? (uint32_t)s_out[g][i] << o : (uint32_t)s_out[g][i] >> -o;
                    }
                }
                reinterpret_cast<uint32_t *>(blocks + b * Blk::BYTES)[w] = x;
            }
            if (gl == 0) fill[b] = (uint8_t)f1;
        }
        uint64_t thr = 0;
        const bool many = cnt > CAND && gl == 0;
        uint32_t nleft = __popc(left);
        if (many) {
            if (DEL) {
                f1 = gblock_remove_many<F, B>(blocks, b, f0, rec + s, cnt, pend32, npend);
            } else if (k) {
                thr = gblock_insert_many<F, B>(blocks, b, f0, k, rec + s, cnt);
                f1 = f0 + k;
            }
            if (f1 != f0) fill[b] = (uint8_t)f1;
            if (!DEL) nleft = cnt - k;
        }
        uint32_t slot = warp_reserve(npend, nleft);
        auto pass_on = [&](uint64_t x) {
            if (!DEL && phase == 1) pend64[slot++] = ((b ^ tcf_g((uint32_t)(x >> 32), G.nb)) << 32) | (uint32_t)x;  // the other block
            else pend32[slot++] = (uint32_t)x;
        };
#pragma unroll
        for (int u = 0; u < 8; u++)
            if ((left >> u) & 1u) pass_on(r[u]);
        if (many && !DEL)
            for (uint32_t q = s; q < e; q++)
                if (k == 0 || rec[q] > thr) pass_on(rec[q]);
        __syncwarp();  // the group's shared memory is free again
    }
}

// The insert of blocks of up to 21 slots, a thread each: a block gets a
// candidate or two, too few for lanes to share (2^24 slots filled to 90 %:
// blocks of 8 slots 2.43 ms by threads, 3.45 by lanes; 21 slots of 12 bits
// 2.44 and 3.18; 32 slots of 16 bits 1.99 and 1.96)
template <int F, int B>
__global__ void __launch_bounds__(TPB) tcf_gblock_insert(TcfGeom G, uint8_t *blocks, uint8_t *fill, PhaseDst P,
                                                         const uint64_t *__restrict__ rec, int phase, uint32_t cap,
                                                         uint32_t *pend32, uint64_t *pend64, unsigned *npend,
                                                         unsigned long long *units)
{
    const uint64_t nd = phase_count(P, G.nb);
    if (P.dlist) note_units(units, nd);  // units: blocks with candidates
    const uint64_t stride = (uint64_t)gridDim.x * TPB;
    for (uint64_t j0 = blockIdx.x * (uint64_t)TPB + (threadIdx.x & ~31u); j0 < nd; j0 += stride) {
        const uint64_t j = j0 + (threadIdx.x & 31);
        uint32_t s = 0, e = 0, k = 0;
        uint64_t b = 0, thr = 0;  // records <= thr are accepted
        if (j < nd) {
            b = phase_dst(P, j, s, e);
            if (s != e) {
                const uint32_t f0 = fill[b];
                k = cap > f0 ? min(e - s, cap - f0) : 0u;
                if (k > 0) {
                    // the k smallest (tag, index) candidates, merged into the sorted block
                    uint64_t a[B];
                    int have = 0;
                    for (uint32_t q = s; q < e; q++) have = topk_push(a, have, (int)k, rec[q]);
                    thr = a[k - 1];
                    uint32_t nv[B];
                    for (uint32_t q = 0; q < k; q++) nv[q] = (uint32_t)(a[q] >> 32);
                    GBlk<F, B> blk;
                    blk.load(blocks, b, false);
                    blk.merge_sorted((int)f0, nv, (int)k);
                    blk.store(blocks, b);
                    fill[b] = (uint8_t)(f0 + k);
                }
            }
        }
        const uint32_t nrej = (e - s) - k;
        uint32_t slot = warp_reserve(npend, nrej);
        if (nrej == 0) continue;
        for (uint32_t q = s; q < e; q++) {
            const uint64_t r = rec[q];
            if (k > 0 && r <= thr) continue;
            const uint32_t i = (uint32_t)r;
            if (phase == 1) pend64[slot++] = ((b ^ tcf_g((uint32_t)(r >> 32), G.nb)) << 32) | i;  // the other block
            else pend32[slot++] = i;
        }
    }
}

// A thread per key reads a 32-byte block; a wider one is read by one lane per
// 16 bytes, so that a load instruction covers whole lines (128 slots of 16
// bits: 32 lines a load with a thread per key, 2 this way; 1.5e7 queries of
// 2^24 slots 1.33 and 0.76 ms). The second block only for keys not in the
// first.
template <int F, int B>
__global__ void __launch_bounds__(TPB) tcf_gquery_kernel(const uint64_t *__restrict__ keys, uint64_t n, TcfGeom G,
                                                         const uint8_t *__restrict__ blocks,
                                                         const uint64_t *__restrict__ bk, const DevCounters *ctr,
                                                         uint8_t *__restrict__ out)
{
    constexpr int L = GBlk<F, B>::BYTES / 16, KW = 32 / L;  // lanes per block, keys of one load
    const bool backing = ctr->backing != 0;
    const int lane = threadIdx.x & 31;
    for (uint64_t i0 = blockIdx.x * (uint64_t)TPB + (threadIdx.x & ~31u); i0 < n; i0 += (uint64_t)gridDim.x * TPB) {
        const uint64_t i = i0 + lane;
        KeyInfo k{0, 0, 0};
        if (i < n) k = tcf_keyinfo(__ldcs(keys + i), G);
        bool hit = false;
        if constexpr (L == 2) {
            GBlk<F, B> x;
            if (i < n) {
                x.load(blocks, k.b1, true);
                hit = x.has(k.t);
                if (!hit) {
                    x.load(blocks, k.b2, true);
                    hit = x.has(k.t);
                }
            }
        } else {
            static_assert(F == 16 || F == 8, "wide blocks of whole bytes");
            const uint4 *base = reinterpret_cast<const uint4 *>(blocks) + lane % L;
            for (int side = 0; side < 2; side++) {
                if (!__any_sync(0xffffffffu, !hit && i < n)) break;
                constexpr int U = L < 8 ? L : 8;  // loads in flight
                for (int r0 = 0; r0 < L; r0 += U) {
                    uint4 v[U];
                    uint32_t t[U];
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        const int src = (r0 + u) * KW + lane / L;
                        const uint32_t b = __shfl_sync(0xffffffffu, (uint32_t)(side ? k.b2 : k.b1), src);  // nb <= 2^32
                        t[u] = __shfl_sync(0xffffffffu, hit ? 0u : k.t, src);
                        const bool want = t[u] != 0;
                        t[u] = F == 16 ? (t[u] | (t[u] << 16)) : t[u] * 0x01010101u;
                        v[u] = want ? __ldg(base + (uint64_t)b * L) : make_uint4(0, 0, 0, 0);
                    }
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        const uint32_t m = F == 16 ? __vcmpeq2(v[u].x, t[u]) | __vcmpeq2(v[u].y, t[u]) |
                                                         __vcmpeq2(v[u].z, t[u]) | __vcmpeq2(v[u].w, t[u])
                                                   : __vcmpeq4(v[u].x, t[u]) | __vcmpeq4(v[u].y, t[u]) |
                                                         __vcmpeq4(v[u].z, t[u]) | __vcmpeq4(v[u].w, t[u]);
                        const unsigned any = __ballot_sync(0xffffffffu, m != 0);
                        if (lane / KW == r0 + u && !hit && k.t) hit = ((any >> (lane % KW * L)) & ((1u << L) - 1u)) != 0;
                    }
                }
            }
        }
        if (i >= n) continue;
        if (!hit && backing) {
            const uint64_t e = tcf_entry(k, G.f);
            const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(bk + tcf_bucket_of(e, G) * BK_W);
#pragma unroll
            for (int s = 0; s < 4; s++) {
                const ulonglong2 v = __ldg(p + s);
                hit |= (v.x == e) | (v.y == e);
            }
        }
        __stcs(out + i, (uint8_t)(hit ? 1 : 0));
    }
}

// one phase's per-block steps of a packed geometry
template <int F, int B, bool DEL>
static void gblock_phase(const TcfBulk &T, const PhaseDst &P, uint64_t n, int phase, uint32_t cap, uint32_t *pend32,
                         uint64_t *pend64, unsigned *npend, unsigned long long *units, cudaStream_t st)
{
    const uint64_t nd = P.dlist && n < T.G.nb ? n : T.G.nb;
    if constexpr (!DEL && B <= 21)
        tcf_gblock_insert<F, B><<<grid_for(nd, TPB, 8), TPB, 0, st>>>(T.G, T.blocks, T.fill, P, T.rec, phase, cap, pend32,
                                                                       pend64, npend, units);
    else
        tcf_gblock_step<F, B, DEL><<<grid_for(nd * GBlk<F, B>::LANES, TPB, 8), TPB, 0, st>>>(
            T.G, T.blocks, T.fill, P, T.rec, phase, cap, pend32, pend64, npend, units);
}

template <int F, int GB = 0>
static void tcf_sparse_insert(const TcfBulk &T, const uint64_t *keys, uint64_t n, uint8_t *status, cudaStream_t st);
template <int F, int GB = 0>
static void tcf_sparse_remove(const TcfBulk &T, const uint64_t *keys, uint64_t n, uint8_t *status, cudaStream_t st);

// Of an uneven call, the first phase over every block instead of the touched
// ones? As in tcf_few_keys; only on large tables, where the five launches that an
// even call then passes through (24 us) count for little: 2^24 keys in a quarter
// of 1024 members of 2^18 slots, an insert 1015 us by touched blocks, 901 so.
static bool uneven_dense(const TcfBulk &T, uint64_t n) { return T.uneven && T.G.nb > (1ull << 22) && n > T.G.nb / 2; }

// the later phases in one launch; at most four CTAs per SM, which its launch
// bounds keep resident together (fewer where the stream has a part of the SMs)
template <int F, bool DEL>
static void tcf_sparse_coop(const TcfBulk &T, const uint64_t *keys, uint64_t n, uint8_t *status, uint32_t unit_min,
                            bool first, cudaStream_t st)
{
    SparseArgs A{keys, n, T.G, T.prep, T.blocks, T.fill, T.bk, T.cnt, T.off, T.tlist, T.tcount, T.dlist, T.pend0, T.pend2,
                 T.rec, T.pend1, T.seg, status, T.ctr, unit_min, first, T.uneven, uneven_dense(T, n)};
    void *args[] = {&A};
    gf::TraceScope ts_(DEL ? "tcf_sparse_remove" : "tcf_sparse_insert", n, st);
    const void *kernel = DEL ? (const void *)tcf_sparse_remove_coop<F> : (const void *)tcf_sparse_insert_coop<F>;
    coop_launch(
        grid_for(n, TPB * 2, 4), cudaErrorCooperativeLaunchTooLarge,
        [&](int g) { return cudaLaunchCooperativeKernel(kernel, dim3(g), dim3(TPB), args, 0, st); },
        [] { cudaGetLastError(); });
}

// the first phase over every block: a shortcut into b1 (A), or removes from it (1)
template <int F, bool DEL, int GB = 0>
static void first_by_block(const TcfBulk &T, const uint64_t *keys, uint64_t n, cudaStream_t st,
                           const unsigned *gate = nullptr)
{
    const TcfGeom G = T.G;
    unsigned *np = T.ctr->pend;
    const PhaseDst P = group_phase<SRC_KEYS, DST_B1>(T, keys, n, nullptr, nullptr, 0, nullptr, st, gate);
    gf::TraceScope ts_(DEL ? "tcf_block_remove" : "tcf_block_insert", 0, st, true);
    if constexpr (GB != 0)
        gblock_phase<F, GB, DEL>(T, P, n, 0, DEL ? 0 : G.tsc, T.pend0, nullptr, &np[0], ts_.units(), st);
    else if constexpr (DEL)
        tcf_block_remove<F><<<dst_grid(P, n, G.nb), TPB, 0, st>>>(G, T.blocks, T.fill, P, T.rec, T.pend0, &np[0], gate,
                                                                   ts_.units());
    else
        tcf_block_insert<F><<<dst_grid(P, n, G.nb), TPB, 0, st>>>(G, T.blocks, T.fill, P, T.rec, 0, G.tsc, T.pend0, nullptr,
                                                                   &np[0], T.prep, gate, ts_.units());
}

// The per-block counting-sort path: each phase groups its candidates by
// destination block (counts, scan, scatter) and one thread per block takes
// its step. Its scratch (a counter and an offset per block, a record per
// candidate) stays in the L2 for moderate tables and batches.
template <int F, int GB = 0>  // GB: slots of a packed block of another geometry
static void tcf_bulk_insert(const TcfBulk &T, const uint64_t *keys, uint64_t n, uint8_t *status, cudaStream_t st)
{
    const TcfGeom G = T.G;
    DevCounters *ctr = T.ctr;
    unsigned *np = ctr->pend;
    cudaMemsetAsync(np, 0, CALL_WORDS_BYTES, st);
    if constexpr (GB == 0)
        if (tcf_few_keys(G.nb, n)) return tcf_sparse_coop<F, false>(T, keys, n, status, 0xffffffffu, true, st);
    first_by_block<F, false, GB>(T, keys, n, st);
    if constexpr (GB == 0)
        if (G.nb >= TCF_COOP_MIN_BLOCKS) return tcf_sparse_coop<F, false>(T, keys, n, status, 0xffffffffu, false, st);
    tcf_sparse_insert<F, GB>(T, keys, n, status, st);
}

// phases B to D of an insert, whose candidates T.pend0 lists by index: a
// counting sort over the blocks that they touch
template <int F, int GB>
static void tcf_sparse_insert(const TcfBulk &T, const uint64_t *keys, uint64_t n, uint8_t *status, cudaStream_t st)
{
    const TcfGeom G = T.G;
    DevCounters *ctr = T.ctr;
    unsigned *np = ctr->pend;
    // B: the less full of b1, b2 under the post-A fills
    PhaseDst P = group_phase<SRC_PEND_U32, DST_TARGET>(T, keys, n, T.pend0, &np[0], 1, nullptr, st);
    {
        gf::TraceScope ts_("tcf_block_insert_sparse", 0, st, true);
        if constexpr (GB == 0)
            tcf_block_insert<F><<<dst_grid(P, n, G.nb), TPB, 0, st>>>(G, T.blocks, T.fill, P, T.rec, 1, G.B, nullptr,
                                                                       T.pend1, &np[1], T.prep, nullptr, ts_.units());
        else
            gblock_phase<F, GB, false>(T, P, n, 1, G.B, nullptr, T.pend1, &np[1], ts_.units(), st);
    }
    // C: the other block
    P = group_phase<SRC_PEND_U64, DST_ALT>(T, keys, n, T.pend1, &np[1], 2, nullptr, st);
    {
        gf::TraceScope ts_("tcf_block_insert_sparse", 0, st, true);
        if constexpr (GB == 0)
            tcf_block_insert<F><<<dst_grid(P, n, G.nb), TPB, 0, st>>>(G, T.blocks, T.fill, P, T.rec, 2, G.B, T.pend2,
                                                                       nullptr, &np[2], T.prep, nullptr, ts_.units());
        else
            gblock_phase<F, GB, false>(T, P, n, 2, G.B, T.pend2, nullptr, &np[2], ts_.units(), st);
    }
    // D: backing buckets
    P = group_phase<SRC_PEND_U32, DST_BUCKET>(T, keys, n, T.pend2, &np[2], 3, T.pend0, st);
    {
        gf::TraceScope ts_("tcf_bucket_insert", 0, st, true);
        tcf_bucket_insert<<<dst_grid(P, n, G.nbk), TPB, 0, st>>>(G, T.bk, P, T.rec, T.pend0, status, ctr, ts_.units());
    }
}

template <int F, int GB = 0>
static void tcf_bulk_remove(const TcfBulk &T, const uint64_t *keys, uint64_t n, uint8_t *status, cudaStream_t st)
{
    const TcfGeom G = T.G;
    DevCounters *ctr = T.ctr;
    unsigned *np = ctr->pend;
    cudaMemsetAsync(np, 0, CALL_WORDS_BYTES, st);
    if constexpr (GB == 0)
        if (tcf_few_keys(G.nb, n)) return tcf_sparse_coop<F, true>(T, keys, n, status, 0xffffffffu, true, st);
    first_by_block<F, true, GB>(T, keys, n, st);
    if constexpr (GB == 0)
        if (G.nb >= TCF_COOP_MIN_BLOCKS) return tcf_sparse_coop<F, true>(T, keys, n, status, 0xffffffffu, false, st);
    tcf_sparse_remove<F, GB>(T, keys, n, status, st);
}

// phases 2 and 3 of a remove, likewise
template <int F, int GB>
static void tcf_sparse_remove(const TcfBulk &T, const uint64_t *keys, uint64_t n, uint8_t *status, cudaStream_t st)
{
    const TcfGeom G = T.G;
    DevCounters *ctr = T.ctr;
    unsigned *np = ctr->pend;
    // 2: secondary block
    PhaseDst P = group_phase<SRC_PEND_U32, DST_B2>(T, keys, n, T.pend0, &np[0], 1, nullptr, st);
    {
        gf::TraceScope ts_("tcf_block_remove_sparse", 0, st, true);
        if constexpr (GB == 0)
            tcf_block_remove<F><<<dst_grid(P, n, G.nb), TPB, 0, st>>>(G, T.blocks, T.fill, P, T.rec, T.pend2, &np[2],
                                                                       nullptr, ts_.units());
        else
            gblock_phase<F, GB, true>(T, P, n, 0, 0, T.pend2, nullptr, &np[2], ts_.units(), st);
    }
    // 3: backing bucket; what is left is not found
    P = group_phase<SRC_PEND_U32, DST_BUCKET>(T, keys, n, T.pend2, &np[2], 2, T.pend0, st);
    {
        gf::TraceScope ts_("tcf_bucket_remove", 0, st, true);
        tcf_bucket_remove<<<dst_grid(P, n, G.nbk), TPB, 0, st>>>(G, T.bk, P, T.rec, T.pend0, status, ctr, ts_.units());
    }
}


// the packed geometries (f, B) that have kernels
#define GF_TCF_GEOMS(X) X(16, 8) X(16, 32) X(16, 64) X(16, 128) X(12, 21) X(8, 64)

bool tcf_geom_supported(uint32_t f, uint32_t B)
{
#define GF_GEOM_IS(FF, BB) \
    if (f == FF && B == BB) return true;
    GF_TCF_GEOMS(GF_GEOM_IS)
#undef GF_GEOM_IS
    return false;
}

static void tcf_custom_bulk(const TcfBulk &W, const uint64_t *keys, uint64_t n, uint8_t *status, bool del,
                            cudaStream_t st)
{
#define GF_GEOM_BULK(FF, BB)                                      \
    if (W.G.f == FF && W.G.B == BB) {                             \
        if (del) tcf_bulk_remove<FF, BB>(W, keys, n, status, st); \
        else tcf_bulk_insert<FF, BB>(W, keys, n, status, st);     \
        return;                                                   \
    }
    GF_TCF_GEOMS(GF_GEOM_BULK)
#undef GF_GEOM_BULK
}

// ---------------------------------------------------------------------------
// Unit phases: host side
// ---------------------------------------------------------------------------
// units of at most `target` candidates on average (2048: a uniform phase's
// largest unit is far below what a CTA holds), one pass up to 2^9 of them
static TuGeom tu_geom(const TcfGeom &G, uint64_t n, uint32_t target)
{
    TuGeom U;
    uint32_t lgnb = 0;
    while ((1ull << lgnb) < G.nb) lgnb++;
    U.k = 0;
    while (U.k < lgnb && U.k < 18 && (n >> U.k) > target) U.k++;
    U.b1 = U.k > 9 ? (U.k + 1) / 2 : U.k;
    U.b2 = U.k - U.b1;
    U.lbits = lgnb - U.k;
    U.sbits = G.f;
    U.ibits = 1;
    while ((1ull << U.ibits) < n) U.ibits++;
    return U;
}

// the record holds what the first pass does not imply
static bool tu_takes(const TcfGeom &G, uint64_t n, uint32_t target)
{
    const TuGeom U = tu_geom(G, n, target);
    return n <= (1ull << 28) && U.lbits <= 31 && U.lbits + U.b2 + U.sbits + U.ibits <= 64;
}

// The partition's scratch for calls of up to max_n keys: one layout for all of
// them, so that the counts, zero between phases, stay where they are.
static MsdScratch tu_scratch(uint32_t *base, uint64_t max_n)
{
    uint32_t k = 0;
    while (k < 18 && (max_n >> k) > 128) k++;  // the smallest target
    return msd_scratch(base, max_n, k, true, false, false);
}
static uint64_t tcf_unit_words(uint64_t max_n) { return tu_scratch(nullptr, max_n).words; }

// one phase: partition the candidates (n: at most as many), step every unit
template <int F, bool DEL, int SRC, int NEXT>
static void tu_phase(const TcfBulk &T, const TuSrc &src, uint64_t n, uint32_t cap, uint64_t *orec, uint32_t *oidx,
                     unsigned *nout, cudaStream_t st)
{
    const TuGeom U = tu_geom(T.G, n, T.tile_target);
    const MsdScratch M = tu_scratch(T.tcur, T.max_n);
    const bool keys = SRC == TU_KEYS;
    const unsigned *uneven = keys ? T.uneven : nullptr;  // (the later phases have no candidates then)
    const bool known = keys && !uneven;  // the number of candidates
    const uint32_t nb1 = 1u << U.b1;
    const uint64_t tiles = (n + MP_TILE - 1) / MP_TILE;
    {
        gf::TraceScope ts_(keys ? "tcf_tile_hist" : "tcf_tile_hist_pend", known ? n : 0, st, !known);
        tu_hist<SRC><<<grid_for(tiles * MP_T, MP_T, 4), MP_T, 0, st>>>(src, T.G, T.prep, T.fill, U, M, uneven, ts_.units());
    }
    {
        gf::TraceScope ts_(keys ? "tcf_tile_part" : "tcf_tile_part_pend", known ? n : 0, st, !known);
        tu_part<SRC><<<(unsigned)tiles, MP_T, 0, st>>>(src, T.G, T.prep, T.fill, U, M, T.rec, uneven, ts_.units());
    }
    if (U.b2)
        msd_second_pass(M, T.rec, T.seg, n, nb1, U.lbits + U.sbits + U.ibits, U.b2, "tcf_tile_hist2", "tcf_tile_part2", st);
    gf::TraceScope ts_(DEL ? "tcf_tile_remove" : "tcf_tile_insert", 0, st, true);
    const TuStep A{T.G, T.prep, U, T.blocks, T.fill, U.b2 ? M.st2 : M.st1, 1u << U.k, cap, U.b2 ? T.seg : T.rec,
                   TuOut{orec, oidx, nout, T.max_n, &T.ctr->status}, src, uneven, ts_.units()};
    const int g = grid_for((uint64_t)TU_T << U.k, TU_T, 3);
    if (U.lbits <= TU_BBITS) tcf_unit_step<F, DEL, NEXT, true><<<g, TU_T, 0, st>>>(A);
    else tcf_unit_step<F, DEL, NEXT, false><<<g, TU_T, 0, st>>>(A);
}

// Candidates of the first phase of all keys up to which the later phases go by
// touched destinations, in one cooperative launch: their counters and records
// stay in the L2 up to 2^22 blocks, whatever their number; on larger tables
// more than one key in sixteen goes by unit (2^28 slots, 2^24 keys at 90 %
// load: 1.41 ms by destination, 0.64 by unit; on the first batches 0.02 and
// 0.13).
static uint32_t tu_unit_min(const TcfBulk &T, uint64_t n)
{
    return T.G.nb > (1ull << 22) ? (uint32_t)(n / 16) : 0xffffffffu;
}

template <int F>
static void tcf_unit_insert(const TcfBulk &T, const uint64_t *keys, uint64_t n, uint8_t *status, cudaStream_t st)
{
    const TcfGeom G = T.G;
    unsigned *np = T.ctr->pend;
    const uint32_t unit_min = tu_unit_min(T, n);
    if (!T.uneven) cudaMemsetAsync(np, 0, CALL_WORDS_BYTES, st);
    // A: shortcut into b1 while fill < 3B/4; rejects keep b1
    tu_phase<F, false, TU_KEYS, TU_NX_SAME>(T, TuSrc{keys, nullptr, nullptr, nullptr, 0, n}, n, G.tsc, T.pend1, T.pend0,
                                            &np[0], st);
    if (unit_min != 0xffffffffu) {
        // B: the less full of b1, b2 under the post-A fills; rejects go to the other block
        tu_phase<F, false, TU_TARGET, TU_NX_OTHER>(T, TuSrc{nullptr, T.pend1, T.pend0, &np[0], unit_min, n}, n, G.B, T.pb,
                                                   T.pbi, &np[1], st);
        // C: the other block; rejects go to the backing buckets by index
        tu_phase<F, false, TU_SAME, TU_NX_IDX>(T, TuSrc{nullptr, T.pb, T.pbi, &np[1], 0, n}, n, G.B, nullptr, T.pend2,
                                               &np[2], st);
    }
    if (uneven_dense(T, n)) first_by_block<F, false>(T, keys, n, st, T.uneven);
    // B and C of fewer candidates, and D: backing buckets
    tcf_sparse_coop<F, false>(T, keys, n, status, unit_min, false, st);
}

template <int F>
static void tcf_unit_remove(const TcfBulk &T, const uint64_t *keys, uint64_t n, uint8_t *status, cudaStream_t st)
{
    unsigned *np = T.ctr->pend;
    const uint32_t unit_min = tu_unit_min(T, n);
    if (!T.uneven) cudaMemsetAsync(np, 0, CALL_WORDS_BYTES, st);
    // 1: primary block; misses go on to the secondary block
    tu_phase<F, true, TU_KEYS, TU_NX_OTHER>(T, TuSrc{keys, nullptr, nullptr, nullptr, 0, n}, n, 0, T.pend1, T.pend0, &np[0],
                                            st);
    // 2: secondary block; misses go to the backing buckets by index
    if (unit_min != 0xffffffffu)
        tu_phase<F, true, TU_SAME, TU_NX_IDX>(T, TuSrc{nullptr, T.pend1, T.pend0, &np[0], unit_min, n}, n, 0, nullptr,
                                              T.pend2, &np[2], st);
    if (uneven_dense(T, n)) first_by_block<F, true>(T, keys, n, st, T.uneven);
    // 2 of fewer candidates, and 3: backing bucket; what is left is not found
    tcf_sparse_coop<F, true>(T, keys, n, status, unit_min, false, st);
}

// Batches that one CTA takes whole (32-byte blocks); false for the others.
// Insert + remove with statuses on 2^20 slots at 88 % load, one CTA against the
// general path: 256 keys 29 / 140, 1000 keys 36 / 143, 2048 keys 48 / 143 us.
template <bool DEL>
static bool tcf_small_call(const TcfBulk &W, const uint64_t *keys, uint64_t n, uint8_t *status, cudaStream_t st)
{
    if (n > TS_CAP || tcf_custom(W.G)) return false;
    auto *kernel = W.G.f == 16 ? tcf_small<16, DEL> : tcf_small<8, DEL>;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TS_SMEM);
    gf::TraceScope ts_(DEL ? "tcf_small_remove" : "tcf_small_insert", n, st);
    kernel<<<1, SM_T, TS_SMEM, st>>>(keys, W.prep, (uint32_t)n, W.G, W.blocks, W.fill, W.bk, status, W.ctr);
    return true;
}

int tcf_insert(filter *F, const uint64_t *keys, const uint8_t *vals, uint64_t n, uint8_t *status, cudaStream_t st)
{
    if (n == 0) return FILTER_OK;
    TcfState &T = F->tcf;
    const TcfBulk W = bulk_of(T, F->scan_tmp, F->ctr, TcfPrep{nullptr, nullptr, nullptr, nullptr, vals}, F->cfg.max_batch,
                               F->tune);
    if (T.mode == FILTER_MODE_BULK && tcf_small_call<false>(W, keys, n, status, st)) {
        GF_CUDA(cudaGetLastError());
        return FILTER_OK;
    }
    if (status) GF_CUDA(cudaMemsetAsync(status, 0, n, st));
    if (T.mode == FILTER_MODE_POINT) {
        const int g = grid_for(n, TPB, 16);
        {
            gf::TraceScope ts_("tcf_point_insert", n, st);
            if (T.G.f == 16) tcf_point_insert<16><<<g, TPB, 0, st>>>(keys, vals, n, T.G, T.blocks, T.bk, status, F->ctr);
            else tcf_point_insert<8><<<g, TPB, 0, st>>>(keys, vals, n, T.G, T.blocks, T.bk, status, F->ctr);
        }
    } else {
        const bool tiled = !tcf_custom(T.G) && tcf_tiled(F->tune, T.G.nb, n, false) && tu_takes(T.G, n, tcf_tile_target(F->tune));
        if (tcf_custom(T.G)) tcf_custom_bulk(W, keys, n, status, false, st);
        else if (T.G.f == 16) tiled ? tcf_unit_insert<16>(W, keys, n, status, st) : tcf_bulk_insert<16>(W, keys, n, status, st);
        else tiled ? tcf_unit_insert<8>(W, keys, n, status, st) : tcf_bulk_insert<8>(W, keys, n, status, st);
    }
    GF_CUDA(cudaGetLastError());
    return FILTER_OK;
}

int tcf_remove(filter *F, const uint64_t *keys, uint64_t n, uint8_t *status, cudaStream_t st)
{
    if (n == 0) return FILTER_OK;
    TcfState &T = F->tcf;
    const TcfBulk W = bulk_of(T, F->scan_tmp, F->ctr, TcfPrep{nullptr, nullptr, nullptr, nullptr}, F->cfg.max_batch, F->tune);
    if (T.mode == FILTER_MODE_BULK && tcf_small_call<true>(W, keys, n, status, st)) {
        GF_CUDA(cudaGetLastError());
        return FILTER_OK;
    }
    if (status) GF_CUDA(cudaMemsetAsync(status, 0, n, st));
    if (T.mode == FILTER_MODE_POINT) {
        const int g = grid_for(n, TPB, 16);
        {
            gf::TraceScope ts_("tcf_point_remove", n, st);
            if (T.G.f == 16) tcf_point_remove<16><<<g, TPB, 0, st>>>(keys, n, T.G, T.blocks, T.bk, status, F->ctr);
            else tcf_point_remove<8><<<g, TPB, 0, st>>>(keys, n, T.G, T.blocks, T.bk, status, F->ctr);
        }
    } else {
        const bool tiled = !tcf_custom(T.G) && tcf_tiled(F->tune, T.G.nb, n, true) && tu_takes(T.G, n, tcf_tile_target(F->tune));
        if (tcf_custom(T.G)) tcf_custom_bulk(W, keys, n, status, true, st);
        else if (T.G.f == 16) tiled ? tcf_unit_remove<16>(W, keys, n, status, st) : tcf_bulk_remove<16>(W, keys, n, status, st);
        else tiled ? tcf_unit_remove<8>(W, keys, n, status, st) : tcf_bulk_remove<8>(W, keys, n, status, st);
    }
    GF_CUDA(cudaGetLastError());
    return FILTER_OK;
}

int tcf_query(filter *F, const uint64_t *keys, uint64_t n, uint8_t *found, bool values, cudaStream_t st)
{
    if (n == 0) return FILTER_OK;
    TcfState &T = F->tcf;
    const int g = grid_for(n, TPB, 16);
    if (values) {
        gf::TraceScope ts_("tcf_query_values_kernel", n, st);
        if (T.G.f == 16) tcf_query_kernel<16, true><<<g, TPB, 0, st>>>(keys, n, T.G, T.blocks, T.bk, F->ctr, found);
        else tcf_query_kernel<8, true><<<g, TPB, 0, st>>>(keys, n, T.G, T.blocks, T.bk, F->ctr, found);
    } else if (tcf_custom(T.G)) {
        gf::TraceScope ts_("tcf_gquery_kernel", n, st);
#define GF_GEOM_QUERY(FF, BB)                                                                                   \
    if (T.G.f == FF && T.G.B == BB) tcf_gquery_kernel<FF, BB><<<g, TPB, 0, st>>>(keys, n, T.G, T.blocks, T.bk, \
                                                                                F->ctr, found);
        GF_TCF_GEOMS(GF_GEOM_QUERY)
#undef GF_GEOM_QUERY
    } else {
        gf::TraceScope ts_("tcf_query_kernel", n, st);
        if (T.G.f == 16) tcf_query_kernel<16, false><<<g, TPB, 0, st>>>(keys, n, T.G, T.blocks, T.bk, F->ctr, found);
        else tcf_query_kernel<8, false><<<g, TPB, 0, st>>>(keys, n, T.G, T.blocks, T.bk, F->ctr, found);
    }
    GF_CUDA(cudaGetLastError());
    return FILTER_OK;
}

uint64_t tcf_image_bytes(const filter *F) { return F->tcf.G.nb * F->tcf.G.bbytes + F->tcf.G.nbk * BK_W * 8; }

int tcf_copy_image(filter *F, void *host, bool to_host, cudaStream_t st)
{
    TcfState &T = F->tcf;
    char *h = static_cast<char *>(host);
    const uint64_t nbB = T.G.nb * T.G.bbytes, bkB = T.G.nbk * BK_W * 8;
    if (to_host) {
        GF_CUDA(cudaMemcpyAsync(h, T.blocks, nbB, cudaMemcpyDeviceToHost, st));
        GF_CUDA(cudaMemcpyAsync(h + nbB, T.bk, bkB, cudaMemcpyDeviceToHost, st));
    } else {
        GF_CUDA(cudaMemcpyAsync(T.blocks, h, nbB, cudaMemcpyHostToDevice, st));
        GF_CUDA(cudaMemcpyAsync(T.bk, h + nbB, bkB, cudaMemcpyHostToDevice, st));
        const int g = grid_for(T.G.nb, TPB, 8);
        {
            gf::TraceScope ts_("tcf_refill", T.G.nb, st);
            if (T.G.f == 16) tcf_refill<16><<<g, TPB, 0, st>>>(T.G, T.blocks, T.fill);
            else tcf_refill<8><<<g, TPB, 0, st>>>(T.G, T.blocks, T.fill);
        }
        GF_CUDA(cudaMemsetAsync(&F->ctr->backing, 0, 8, st));
        {
            gf::TraceScope ts_("tcf_count_backing", T.G.nbk * BK_W, st);
            tcf_count_backing<<<grid_for(T.G.nbk * BK_W, TPB, 4), TPB, 0, st>>>(T.G, T.bk, F->ctr);
        }
    }
    GF_CUDA(cudaStreamSynchronize(st));
    return FILTER_OK;
}

// ---------------------------------------------------------------------------
// Filter groups: every member's keys in one set of launches. A member's keys
// are hashed with its own geometry, then every phase runs over the
// concatenated blocks and buckets of all members. Candidates of one block
// all belong to its member and keep their batch order, so each member ends
// up exactly as a standalone filter given the same keys.
// ---------------------------------------------------------------------------
__device__ __forceinline__ TcfGeom member_geom(const TcfMember &M, uint32_t f)
{
    TcfGeom G;
    G.nb = M.nb;
    G.nbk = M.nbk;
    G.seed = M.seed;
    G.f = f;
    G.B = 256 / f;
    G.tsc = 3 * G.B / 4;
    G.tmask = (1u << f) - 1u;
    return G;
}

// Units are equal stretches of a group's blocks, and a call may bring its keys
// to a few members only: one CTA would then read a unit of many thousand
// candidates once for every range that it holds. A member's keys spread evenly
// over its blocks, so the offsets tell. With a unit of more keys than a CTA holds
// (less some five deviations) the partition is left out (its kernels return at
// once), and the cooperative launch takes all phases by touched blocks. An
// insert and a remove in us by unit / so, in 1024 members of 2^18 slots: 2^20 keys
// in 8 of them 121400 + 167900 / 185 + 256, 2^22 in a quarter 872 + 1080 / 413 +
// 420, 2^24 in a half 923 + 1179 / 873 + 1067; in all of them, by unit, 755 + 932.
static constexpr uint64_t TU_UNEVEN = TU_CAP - 256;

// the keys of the blocks below b, as the members' shares of blocks say
__device__ __forceinline__ uint64_t keys_below(uint64_t b, const uint64_t *__restrict__ off, uint32_t nmem,
                                               const TcfMember *__restrict__ mem)
{
    uint32_t lo = 0, hi = nmem;  // the last member that starts at or before b
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (mem[mid].block0 <= b) lo = mid;
        else hi = mid;
    }
    const uint64_t in = b - mem[lo].block0, nb = mem[lo].nb, c = off[lo + 1] - off[lo];
    return off[lo] + (in < nb ? in * c / nb : c);
}

// uneven: set when some unit of 2^lbits blocks has too many keys (null: not asked)
__global__ void __launch_bounds__(TPB) tcf_group_prep(const uint64_t *__restrict__ keys, uint64_t n,
                                                      const uint64_t *__restrict__ off, uint32_t nmem,
                                                      const TcfMember *__restrict__ mem, uint32_t f, TcfPrep out,
                                                      uint64_t nunits, uint32_t lbits, unsigned *uneven)
{
    if (uneven)
        for (uint64_t u = blockIdx.x * (uint64_t)TPB + threadIdx.x; u < nunits; u += (uint64_t)gridDim.x * TPB)
            if (keys_below((u + 1) << lbits, off, nmem, mem) - keys_below(u << lbits, off, nmem, mem) > TU_UNEVEN) *uneven = 1;
    MemberCursor c(off, nmem, n);
    uint32_t cm = 0xffffffffu;
    TcfMember M;
    TcfGeom G;
    for (; c.valid(); c.next(off)) {
        if (c.m != cm) {
            cm = c.m;
            M = mem[cm];
            G = member_geom(M, f);
        }
        const KeyInfo k = tcf_keyinfo(__ldcs(keys + c.i), G);
        const uint64_t e = tcf_entry(k, f);
        out.bt[c.i] = ((M.block0 + k.b1) << 32) | k.t;
        out.b2[c.i] = (uint32_t)(M.block0 + k.b2);
        out.bucket[c.i] = (uint32_t)(M.bucket0 + tcf_bucket(e, M.nbk));
        out.e[c.i] = e;
    }
}

template <int F>
__global__ void __launch_bounds__(TPB) tcf_group_query_kernel(const uint64_t *__restrict__ keys, uint64_t n,
                                                              const uint64_t *__restrict__ off, uint32_t nmem,
                                                              const TcfMember *__restrict__ mem,
                                                              const uint8_t *__restrict__ blocks,
                                                              const uint64_t *__restrict__ bk,
                                                              const DevCounters *ctr, uint8_t *__restrict__ out)
{
    const bool backing = ctr->backing != 0;
    MemberCursor c(off, nmem, n);
    uint32_t cm = 0xffffffffu;
    TcfMember M;
    TcfGeom G;
    for (; c.valid(); c.next(off)) {
        if (c.m != cm) {
            cm = c.m;
            M = mem[cm];
            G = member_geom(M, F);
        }
        const KeyInfo k = tcf_keyinfo(__ldcs(keys + c.i), G);
        Blk<F> x, y;
        x.load_ro(blocks, M.block0 + k.b1);
        y.load_ro(blocks, M.block0 + k.b2);
        bool hit = x.has(k.t, 0xffffffffu) || y.has(k.t, 0xffffffffu);  // group members carry no values
        if (!hit && backing) {
            const uint64_t e = tcf_entry(k, F);
            const ulonglong2 *p =
                reinterpret_cast<const ulonglong2 *>(bk + (M.bucket0 + tcf_bucket(e, M.nbk)) * BK_W);
#pragma unroll
            for (int s = 0; s < 4; s++) {
                ulonglong2 v = __ldg(p + s);
                hit |= (v.x == e) | (v.y == e);
            }
        }
        __stcs(out + c.i, (uint8_t)(hit ? 1 : 0));
    }
}

int tcf_group_setup(filter_group *GR, const filter_config *cfgs, uint64_t &bytes_out, bool plan_only)
{
    const uint32_t n = GR->n;
    const uint32_t f = cfgs[0].tag_bits;
    const uint64_t M = GR->max_total ? GR->max_total : 1;
    if (M > 0xffffffffull) return FILTER_ERR_ARG;
    std::vector<TcfMember> tm(n);
    uint64_t nb_tot = 0, nbk_tot = 0;
    for (uint32_t m = 0; m < n; m++) {
        const filter_config &c = cfgs[m];
        if (c.kind != FILTER_TCF || c.tag_bits != f || c.mode != FILTER_MODE_BULK || c.value_bits || c.block_slots ||
            (f != 8 && f != 16))
            return FILTER_ERR_ARG;  // members: 32-byte blocks of 8- or 16-bit tags
        filter V;
        V.cfg = c;
        V.cfg.max_batch = M;
        uint64_t tb = 0, sb = 0;
        int rc = tcf_setup(&V, tb, sb, true);  // geometry only
        if (rc != FILTER_OK) return rc;
        tm[m].nb = V.tcf.G.nb;
        tm[m].nbk = V.tcf.G.nbk;
        tm[m].seed = V.tcf.G.seed;
        tm[m].block0 = nb_tot;
        tm[m].bucket0 = nbk_tot;
        nb_tot += V.tcf.G.nb;
        nbk_tot += V.tcf.G.nbk;
    }
    if (nb_tot > 0xffffffffull || nbk_tot > 0xffffffffull) return FILTER_ERR_ARG;  // 32-bit indices
    TcfState &T = GR->tcf;
    T.mode = FILTER_MODE_BULK;
    T.G.f = f;
    T.G.B = 256 / f;
    T.G.tsc = 3 * T.G.B / 4;
    T.G.tmask = (1u << f) - 1u;
    T.G.nb = nb_tot;
    T.G.nbk = nbk_tot;
    T.G.seed = 0;
    const uint64_t groups = (nb_tot > nbk_tot ? nb_tot : nbk_tot) + 1;
    uint64_t bytes = 0;
    Arena &A = GR->arena;
    auto piece = [&](auto *&ptr, uint64_t count) {
        using T_ = typename std::remove_reference<decltype(*ptr)>::type;
        bytes += (count * sizeof(T_) + 255) & ~255ull;
        if (!plan_only) ptr = A.take<T_>(count);
    };
    piece(T.blocks, nb_tot * 32);
    piece(T.bk, nbk_tot * BK_W);
    piece(T.fill, nb_tot);
    piece(T.cnt, groups);
    piece(T.off, groups);
    piece(T.rec, M);
    piece(T.pend0, M);
    piece(T.pend1, M);
    piece(T.pend2, M);
    piece(T.tlist, M);
    piece(T.tcount, (uint64_t)sm_count() * 8);
    piece(T.dlist, M);
    piece(T.seg, M);
    piece(T.tcur, tcf_unit_words(M));
    piece(T.pb, M);
    piece(T.pbi, M);
    piece(GR->prep.bt, M);
    piece(GR->prep.b2, M);
    piece(GR->prep.bucket, M);
    piece(GR->prep.e, M);
    piece(GR->d_tmem, (uint64_t)n);
    piece(GR->scan_tmp, scan_tmp_words(groups));
    bytes_out = bytes;
    if (plan_only) return FILTER_OK;
    if (!T.blocks || !T.bk || !T.fill || !T.cnt || !T.off || !T.rec || !T.pend0 || !T.pend1 || !T.pend2 ||
        !T.tlist || !T.tcount || !T.dlist || !T.seg || !T.tcur || !T.pb || !T.pbi || !GR->prep.bt || !GR->prep.b2 || !GR->prep.bucket ||
        !GR->prep.e || !GR->d_tmem || !GR->scan_tmp)
        return FILTER_ERR_INTERNAL;
    GF_CUDA(cudaMemcpy(GR->d_tmem, tm.data(), n * sizeof(TcfMember), cudaMemcpyHostToDevice));
    // host views of the members: their slices of the group's arrays
    for (uint32_t m = 0; m < n; m++) {
        filter &V = GR->members[m];
        V.cfg = cfgs[m];
        V.cfg.max_batch = M;
        uint64_t tb = 0, sb = 0;
        tcf_setup(&V, tb, sb, true);
        TcfState &S = V.tcf;
        S.blocks = T.blocks + tm[m].block0 * 32;
        S.bk = T.bk + tm[m].bucket0 * BK_W;
        S.fill = T.fill + tm[m].block0;
        S.cnt = T.cnt;
        S.off = T.off;
        S.rec = T.rec;
        S.pend0 = T.pend0;
        S.pend1 = T.pend1;
        S.pend2 = T.pend2;
        S.tlist = T.tlist;
        S.tcount = T.tcount;
        S.dlist = T.dlist;
        S.seg = T.seg;
        S.tcur = T.tcur;
        S.pb = T.pb;
        S.pbi = T.pbi;
        V.ctr = GR->ctr;
        V.scan_tmp = GR->scan_tmp;
        V.arena.base = GR->arena.base;  // marks the view valid; the group owns the memory
        V.device = GR->device;
    }
    return FILTER_OK;
}

int tcf_group_clear(filter_group *GR, cudaStream_t st)
{
    TcfState &T = GR->tcf;
    const uint64_t groups = (T.G.nb > T.G.nbk ? T.G.nb : T.G.nbk) + 1;
    GF_CUDA(cudaMemsetAsync(T.blocks, 0, T.G.nb * T.G.bbytes, st));
    GF_CUDA(cudaMemsetAsync(T.bk, 0, T.G.nbk * BK_W * 8, st));
    GF_CUDA(cudaMemsetAsync(T.fill, 0, T.G.nb, st));
    GF_CUDA(cudaMemsetAsync(T.cnt, 0, groups * 4, st));
    GF_CUDA(cudaMemsetAsync(T.tcur, 0, tu_scratch(nullptr, GR->max_total).zero_words * 4, st));
    GF_CUDA(cudaMemsetAsync(GR->ctr, 0, sizeof(DevCounters), st));
    return FILTER_OK;
}

int tcf_group_op(filter_group *GR, int op, const uint64_t *off, const uint64_t *keys, uint64_t n, uint8_t *out,
                 cudaStream_t st)
{
    if (n == 0) return FILTER_OK;
    TcfState &T = GR->tcf;
    if (op == GROUP_QUERY) {
        const int g = grid_for(n, TPB, 16);
        gf::TraceScope ts_("tcf_group_query_kernel", n, st);
        if (T.G.f == 16)
            tcf_group_query_kernel<16><<<g, TPB, 0, st>>>(keys, n, off, GR->n, GR->d_tmem, T.blocks, T.bk, GR->ctr, out);
        else
            tcf_group_query_kernel<8><<<g, TPB, 0, st>>>(keys, n, off, GR->n, GR->d_tmem, T.blocks, T.bk, GR->ctr, out);
        GF_CUDA(cudaGetLastError());
        return FILTER_OK;
    }
    TcfBulk W = bulk_of(T, GR->scan_tmp, GR->ctr, GR->prep, GR->max_total, GR->tune);
    const bool tiled = n > TS_CAP && tcf_tiled(GR->tune, T.G.nb, n, op != GROUP_INSERT) && tu_takes(T.G, n, W.tile_target);
    const TuGeom U = tu_geom(T.G, n, W.tile_target);
    if (tiled && GR->tune.tcf_path == FILTER_TCF_PATH_AUTO) {
        W.uneven = &GR->ctr->uneven;
        GF_CUDA(cudaMemsetAsync(GR->ctr->pend, 0, CALL_WORDS_BYTES, st));
    }
    {
        gf::TraceScope ts_("tcf_group_prep", n, st);
        tcf_group_prep<<<grid_for(n, TPB, 8), TPB, 0, st>>>(keys, n, off, GR->n, GR->d_tmem, T.G.f, GR->prep, 1ull << U.k,
                                                            U.lbits, W.uneven);
    }
    if (op == GROUP_INSERT ? tcf_small_call<false>(W, nullptr, n, out, st) : tcf_small_call<true>(W, nullptr, n, out, st)) {
        GF_CUDA(cudaGetLastError());
        return FILTER_OK;
    }
    if (out) GF_CUDA(cudaMemsetAsync(out, 0, n, st));
    if (op == GROUP_INSERT) {
        if (T.G.f == 16) tiled ? tcf_unit_insert<16>(W, nullptr, n, out, st) : tcf_bulk_insert<16>(W, nullptr, n, out, st);
        else tiled ? tcf_unit_insert<8>(W, nullptr, n, out, st) : tcf_bulk_insert<8>(W, nullptr, n, out, st);
    } else {
        if (T.G.f == 16) tiled ? tcf_unit_remove<16>(W, nullptr, n, out, st) : tcf_bulk_remove<16>(W, nullptr, n, out, st);
        else tiled ? tcf_unit_remove<8>(W, nullptr, n, out, st) : tcf_bulk_remove<8>(W, nullptr, n, out, st);
    }
    GF_CUDA(cudaGetLastError());
    return FILTER_OK;
}

}  // namespace gf
