// Sort and reduce of a large batch's fingerprints (paper Sec. 5.3 "Sorting
// hashes", Sec. 5.4 map-reduce): the distinct values in ascending order with
// the number of copies before each, from the most significant bits down.
//
// Fingerprints are hashes, so their top k bits cut a batch into units of a
// thousand or two keys each. One or two partition passes by those bits (the
// order inside a bin is free, so a key takes its place with one shared-memory
// atomic and a tile its room in a bin with one global one: no per-tile count
// matrix, no scan over it, no ranking by ballots), then one CTA per unit sorts
// it in shared memory and writes its groups behind those of the units before.
// 2.4e8 36-bit keys move 8 (histogram) + 16 + 8 + 16 bytes each in the passes
// and 8 in the last one; the least-significant-digit sort of gf_prims.cu, which
// serves batches that carry values, moves 16 + 4 * 16 + 3 * 8, and 8 in the
// reduction. Zipf keys: 8.35 ms there, 5.14 ms here (histograms 0.47 + 0.29,
// passes 0.97 + 1.07, hot units 0.38, units 1.95).
//
// Skew: the copies of a key all fall into one unit. A unit of more than MU_CAP
// keys goes through a hash table in shared memory (its distinct values are
// few) before the others are sorted, and one of more than MS_CHUNK keys is
// squeezed to (value, copies) pairs before that, chunk by chunk. Where the
// distinct values do not fit the table, the values are not spread as hashes are
// (a stretch of a filter's enumeration put into another of its geometry): the
// units are then given up, and the caller sorts by digits, whatever the values.
#include "gf_internal.cuh"

namespace gf {

static constexpr int MU_T = 256;                // threads of a unit, a chunk or an oversized unit
static constexpr uint32_t MU_CAP = 2560;        // keys that a unit sorts in shared memory
static constexpr uint32_t MU_BBITS = 12, MU_BUCKETS = 1u << MU_BBITS;  // buckets of that sort
static constexpr uint32_t MU_HOT = 8;           // keys of one bucket above which a warp takes them
static constexpr uint32_t MT_CAP = 4096;        // hash table: home slots
static constexpr uint32_t MT_PAD = 256;         // and slots past the last one
static constexpr uint32_t MT_PROBES = 192;      // hash table: longest probe
static constexpr uint32_t MS_CHUNK = 16384;     // keys of a squeezed chunk
static constexpr uint32_t EMPTY = 0xffffffffu;  // (values below have at most 31 bits)

static_assert(MP_BINS <= MP_T, "a thread per bin");

MsdScratch msd_scratch(uint32_t *base, uint64_t n, uint32_t k, bool two, bool lookback, bool big)
{
    MsdScratch s;
    uint64_t at = 0;
    auto take = [&](uint64_t words) {
        uint32_t *p = base ? base + at : nullptr;
        at += (words + 3) & ~3ull;
        return p;
    };
    const uint64_t units = 1ull << k, chunks = 2 * (n / MS_CHUNK) + 2;
    s.cnt1 = take(MP_BINS);
    s.misc = take(5);
    s.look = reinterpret_cast<uint64_t *>(take(lookback ? 2 * units : 0));
    s.cnt2 = take(two ? units : 0);
    s.zero_words = at;
    s.st1 = take(MP_BINS + 1);
    s.cur1 = take(MP_BINS);
    s.tile1 = take(MP_BINS + 1);
    s.htile1 = take(MP_BINS + 1);
    s.st2 = take(two ? units + 1 : 0);
    s.cur2 = take(two ? units : 0);
    s.chunk0 = s.distinct = s.big = s.chunk_unit = s.chunk_cnt = nullptr;
    if (big) {
        s.chunk0 = take(units);
        s.distinct = take(units);
        s.big = take(n / MU_CAP + 1);
        s.chunk_unit = take(chunks);
        s.chunk_cnt = take(chunks);
    }
    s.big_cap = MU_CAP;
    s.chunk = MS_CHUNK;
    s.words = at;
    return s;
}

// ---------------------------------------------------------------------------
// Histograms
// ---------------------------------------------------------------------------
// keys per first-pass bin (fingerprint >> shift), one shared histogram per CTA
__global__ void __launch_bounds__(MP_T) msd_hist1(const uint64_t *__restrict__ keys, uint64_t n, PHash H,
                                                  uint32_t shift, uint32_t nb, MsdScratch s, bool two, uint32_t *m_out)
{
    __shared__ uint32_t h[MP_BINS];
    if (blockIdx.x == 0 && threadIdx.x == 0) *m_out = 0;  // (the units count into it)
    for (uint32_t b = threadIdx.x; b < nb; b += MP_T) h[b] = 0;
    __syncthreads();
    const uint64_t step = (uint64_t)gridDim.x * MP_TILE;
    for (uint64_t base = (uint64_t)blockIdx.x * MP_TILE; base < n; base += step) {
        uint64_t v[MP_I];
#pragma unroll
        for (int r = 0; r < MP_I; r++) {
            const uint64_t i = base + r * MP_T + threadIdx.x;
            if (i < n) v[r] = __ldcs(keys + i);
        }
#pragma unroll
        for (int r = 0; r < MP_I; r++) {
            const uint64_t i = base + r * MP_T + threadIdx.x;
            if (i < n) atomicAdd(&h[(uint32_t)(fingerprint(v[r], H) >> shift)], 1u);
        }
    }
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < nb; b += MP_T)
        if (h[b]) atomicAdd(&s.cnt1[b], h[b]);
    hist_end(s, nb, two);
}

// the bin whose tiles hold tile t, or nb past the last tile
__device__ __forceinline__ uint32_t bin_of_tile(const uint32_t *__restrict__ first, uint32_t nb, uint32_t t)
{
    if (t >= first[nb]) return nb;
    uint32_t lo = 0, hi = nb;  // first[lo] <= t < first[hi]
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (first[mid] <= t) lo = mid;
        else hi = mid;
    }
    return lo;
}

// keys per unit: every CTA counts MH_TILE keys of one first-pass bin
__global__ void __launch_bounds__(MP_T) msd_hist2(const uint64_t *__restrict__ v, MsdScratch s, uint32_t nb1,
                                                  uint32_t shift, uint32_t bits2, unsigned long long *units)
{
    __shared__ uint32_t h[MP_BINS];
    if (units && blockIdx.x == 0 && threadIdx.x == 0) *units = s.st1[nb1];  // (a phase may have fewer than its bound)
    const uint32_t j = bin_of_tile(s.htile1, nb1, blockIdx.x), nb = 1u << bits2;
    if (j == nb1) return;
    for (uint32_t b = threadIdx.x; b < nb; b += MP_T) h[b] = 0;
    __syncthreads();
    const uint32_t i0 = s.st1[j] + (blockIdx.x - s.htile1[j]) * MH_TILE, end = min(i0 + MH_TILE, s.st1[j + 1]);
    for (uint32_t base = i0; base < end; base += MP_TILE) {
        uint64_t x[MP_I];
#pragma unroll
        for (int r = 0; r < MP_I; r++) {
            const uint32_t i = base + r * MP_T + threadIdx.x;
            if (i < end) x[r] = __ldcs(v + i);
        }
#pragma unroll
        for (int r = 0; r < MP_I; r++) {
            const uint32_t i = base + r * MP_T + threadIdx.x, d = i < end ? (uint32_t)(x[r] >> shift) & (nb - 1) : nb;
            // a hot unit: a warp's keys in one bin are one update
            const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
            if (__all_sync(0xffffffffu, d == d0)) {
                if (d0 < nb && (threadIdx.x & 31) == 0) atomicAdd(&h[d0], 32u);
            } else if (d < nb) {
                atomicAdd(&h[d], 1u);
            }
        }
    }
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < nb; b += MP_T)
        if (h[b]) atomicAdd(&s.cnt2[(j << bits2) + b], h[b]);
}

// starts and cursors of the units of first-pass bin blockIdx.x; the counts are
// left at zero
__global__ void __launch_bounds__(MP_BINS) msd_scan2(MsdScratch s, uint32_t nb1, uint32_t bits2)
{
    __shared__ uint32_t s_warp[MP_BINS / 32];
    const uint32_t j = blockIdx.x, b = threadIdx.x, u = (j << bits2) + b;
    const uint32_t c = b < (1u << bits2) ? s.cnt2[u] : 0u;
    const uint32_t st = s.st1[j] + cta_scan<MP_BINS>(c, s_warp);
    if (b >= (1u << bits2)) return;
    s.cnt2[u] = 0;
    s.st2[u] = s.cur2[u] = st;
    if (u == (nb1 << bits2) - 1) s.st2[u + 1] = st + c;
    list_big(s, u, c);
}

// ---------------------------------------------------------------------------
// A partition pass. FIRST: tiles of the batch, whose keys are hashed; else
// tiles of a first-pass bin, whose values go to its units. Bound by the
// shared-memory pipe (80 % busy with the rank atomics and the staging; 16 bytes
// a key at 4.4 TB/s); 48 warps per SM.
// ---------------------------------------------------------------------------
template <bool FIRST>
__global__ void __launch_bounds__(MP_T, 3) msd_part(const uint64_t *__restrict__ in, uint32_t n, PHash H, MsdScratch s,
                                                    uint32_t nb1, uint32_t shift, uint32_t bits,
                                                    uint64_t *__restrict__ out, unsigned long long *units)
{
    __shared__ PartSmem S;
    if (!FIRST && units && blockIdx.x == 0 && threadIdx.x == 0) *units = s.st1[nb1];
    const uint32_t nb = 1u << bits;
    uint32_t base, end;
    uint32_t *cur;
    if (FIRST) {
        base = blockIdx.x * MP_TILE;
        end = n;
        cur = s.cur1;
    } else {
        const uint32_t j = bin_of_tile(s.tile1, nb1, blockIdx.x);
        if (j == nb1) return;
        base = s.st1[j] + (blockIdx.x - s.tile1[j]) * MP_TILE;
        end = s.st1[j + 1];
        cur = s.cur2 + ((uint64_t)j << bits);
    }
    const uint32_t cnt = end - base < MP_TILE ? end - base : MP_TILE;
    uint64_t v[MP_I];
#pragma unroll
    for (int r = 0; r < MP_I; r++) {
        const uint32_t i = r * MP_T + threadIdx.x;
        v[r] = i < cnt ? __ldcs(in + base + i) : 0ull;
    }
    if (FIRST)
#pragma unroll
        for (int r = 0; r < MP_I; r++) v[r] = fingerprint(v[r], H);
    part_tile<!FIRST>(S, v, cnt, nb, [=](uint64_t x, int) { return (uint32_t)(x >> shift) & (nb - 1); }, cur);
#pragma unroll
    for (int r = 0; r < MP_I; r++) {
        const uint32_t i = r * MP_T + threadIdx.x;
        if (i < cnt) {
            const uint64_t x = S.key[i];
            __stcs(out + (S.delta[(uint32_t)(x >> shift) & (nb - 1)] + i), x);
        }
    }
}

void msd_second_pass(const MsdScratch &s, const uint64_t *in, uint64_t *out, uint64_t n, uint32_t nb1, uint32_t shift,
                     uint32_t bits2, const char *hist_name, const char *part_name, cudaStream_t st)
{
    {
        TraceScope ts_(hist_name, 0, st, true);
        msd_hist2<<<(unsigned)((n + MH_TILE - 1) / MH_TILE) + nb1, MP_T, 0, st>>>(in, s, nb1, shift, bits2, ts_.units());
    }
    {
        TraceScope ts_("msd_scan2", (uint64_t)nb1 << bits2, st);
        msd_scan2<<<nb1, MP_BINS, 0, st>>>(s, nb1, bits2);
    }
    TraceScope ts_(part_name, 0, st, true);
    msd_part<false><<<(unsigned)((n + MP_TILE - 1) / MP_TILE) + nb1, MP_T, 0, st>>>(in, (uint32_t)n, PHash{}, s, nb1,
                                                                                         shift, bits2, out, ts_.units());
}

// ---------------------------------------------------------------------------
// Hash table of (value, copies), order-preserving: a value's home slot are its
// top bits, probes go up, nothing wraps. So the distinct values lie in order up
// to permutations inside a cluster of slots without a gap.
// ---------------------------------------------------------------------------
struct Table {
    uint32_t *key, *cnt;  // MT_CAP + MT_PAD each
    uint32_t *over;       // set when a value found no slot
    uint32_t shift;       // home slot of v: v >> shift

    __device__ __forceinline__ void add(uint32_t v, uint32_t w) const
    {
        uint32_t p = v >> shift;
        for (uint32_t t = 0; t < MT_PROBES && p < MT_CAP + MT_PAD; t++, p++) {
            uint32_t x = key[p];
            if (x == EMPTY) x = atomicCAS(&key[p], EMPTY, v);
            if (x == EMPTY || x == v) {
                atomicAdd(&cnt[p], w);
                return;
            }
            if (t % 16 == 15 && full()) return;
        }
        *over = 1;
    }
    // some value found no slot (while others are added)
    __device__ __forceinline__ bool full() const { return *(const volatile uint32_t *)over; }
    __device__ __forceinline__ void clear() const
    {
        for (uint32_t p = threadIdx.x; p < MT_CAP + MT_PAD; p += MU_T) {
            key[p] = EMPTY;
            cnt[p] = 0;
        }
        if (threadIdx.x == 0) *over = 0;
    }
};

// a thread's stream of values, runs of one value added once
struct RunCache {
    uint32_t v = EMPTY, w = 0;
    __device__ __forceinline__ void push(const Table &T, uint32_t x, uint32_t copies)
    {
        if (x != v) {
            flush(T);
            v = x;
            w = 0;
        }
        w += copies;
    }
    __device__ __forceinline__ void flush(const Table &T)
    {
        if (w) T.add(v, w);
    }
};

// Squeezes the chunks of the units above MS_CHUNK keys to pairs (copies << 32
// | low value bits), in place: copies of a hot key and a few distinct others. A
// chunk with more of them than the table takes gives the units up.
__global__ void __launch_bounds__(MU_T) msd_squeeze(uint64_t *v, MsdScratch s, const uint32_t *__restrict__ st,
                                                    uint32_t rbits)
{
    __shared__ uint32_t t_key[MT_CAP + MT_PAD], t_cnt[MT_CAP + MT_PAD], s_over, s_n;
    const uint32_t mask = (1u << rbits) - 1u;
    const Table T{t_key, t_cnt, &s_over, rbits > 12 ? rbits - 12 : 0u};
    static_assert(MT_CAP == 1u << 12, "12 bits of home slot");
    for (uint32_t c = blockIdx.x; c < s.misc[1]; c += gridDim.x) {
        const uint32_t u = s.chunk_unit[c], i0 = st[u] + (c - s.chunk0[u]) * MS_CHUNK;
        const uint32_t end = min(i0 + MS_CHUNK, st[u + 1]);
        T.clear();
        if (threadIdx.x == 0) s_n = 0;
        if (__syncthreads_or(s.misc[4])) return;
        RunCache run;
        for (uint32_t base = i0; base < end && !T.full(); base += 8 * MU_T) {
            uint64_t x[8];
#pragma unroll
            for (int r = 0; r < 8; r++) {
                const uint32_t i = base + r * MU_T + threadIdx.x;
                if (i < end) x[r] = v[i];
            }
#pragma unroll
            for (int r = 0; r < 8; r++)
                if (base + r * MU_T + threadIdx.x < end) run.push(T, (uint32_t)x[r] & mask, 1u);
        }
        run.flush(T);
        __syncthreads();
        if (s_over) {
            if (threadIdx.x == 0) s.misc[4] = 1;
            return;
        }
        for (uint32_t p = threadIdx.x; p < MT_CAP + MT_PAD; p += MU_T)
            if (t_key[p] != EMPTY) v[i0 + atomicAdd(&s_n, 1u)] = ((uint64_t)t_cnt[p] << 32) | t_key[p];
        __syncthreads();
        if (threadIdx.x == 0) s.chunk_cnt[c] = s_n;
        __syncthreads();
    }
}

// Oversized units, a CTA each: every (value, copies) through the hash table.
// The distinct values are left in order in `spare` as pairs, their number in
// distinct[u]. They have a launch of their own because a slow unit would hold
// up the look-back of all that follow it. A unit with more distinct values than
// the table takes gives the units up: another round over its keys for each part
// of them grows with the square of their number (2^16 keys spread over one unit
// of 2^28 slots, an insert 95 ms by such rounds, 0.32 given up and sorted by digits).
__global__ void __launch_bounds__(MU_T) msd_big(const uint64_t *__restrict__ v, MsdScratch s,
                                                const uint32_t *__restrict__ st, uint32_t rbits, uint64_t *spare)
{
    __shared__ uint32_t t_key[MT_CAP + MT_PAD], t_cnt[MT_CAP + MT_PAD], s_over, s_warp[MU_T / 32];
    const uint32_t mask = (1u << rbits) - 1u;
    const Table T{t_key, t_cnt, &s_over, rbits > 12 ? rbits - 12 : 0u};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint32_t k = blockIdx.x; k < s.misc[2]; k += gridDim.x) {
        const uint32_t u = s.big[k], s0 = st[u], c = st[u + 1] - s0;
        const bool squeezed = c > MS_CHUNK;
        const uint32_t nch = (c + MS_CHUNK - 1) / MS_CHUNK, ch0 = squeezed ? s.chunk0[u] : 0u;
        // threads per chunk: few when the chunks are many, and hold little each
        uint32_t per = MU_T;
        while (per > 4 && (MU_T / per) < nch) per >>= 1;
        T.clear();
        if (__syncthreads_or(s.misc[4])) return;
        RunCache run;
        for (uint32_t ch = threadIdx.x / per; ch < nch; ch += MU_T / per) {
            const uint64_t *p = v + s0 + ch * MS_CHUNK;
            const uint32_t m = squeezed ? s.chunk_cnt[ch0 + ch] : c;
            for (uint32_t i = threadIdx.x % per; i < m && !T.full(); i += 8 * per) {
                uint64_t x[8];
#pragma unroll
                for (int r = 0; r < 8; r++)
                    if (i + r * per < m) x[r] = p[i + r * per];
#pragma unroll
                for (int r = 0; r < 8; r++)
                    if (i + r * per < m) run.push(T, (uint32_t)x[r] & mask, squeezed ? (uint32_t)(x[r] >> 32) : 1u);
            }
        }
        run.flush(T);
        __syncthreads();
        if (s_over) {
            if (threadIdx.x == 0) s.misc[4] = 1;
            return;
        }
        // occupied slots below each warp's stretch of the table
        constexpr uint32_t SPAN = (MT_CAP + MT_PAD) / (MU_T / 32);
        static_assert(SPAN % 32 == 0, "whole warps of slots");
        uint32_t mine = 0;
        for (uint32_t q = 0; q < SPAN; q += 32)
            mine += __popc(__ballot_sync(0xffffffffu, t_key[warp * SPAN + q + lane] != EMPTY));
        if (lane == 0) s_warp[warp] = mine;
        __syncthreads();
        uint32_t pre = 0, total = 0;
        for (int w = 0; w < MU_T / 32; w++) {
            if (w < warp) pre += s_warp[w];
            total += s_warp[w];
        }
        for (uint32_t q = 0; q < SPAN; q += 32) {
            const uint32_t p = warp * SPAN + q + lane, x = t_key[p];
            const unsigned occ = __ballot_sync(0xffffffffu, x != EMPTY);
            if (x != EMPTY) {
                uint32_t r = pre + __popc(occ & ((1u << lane) - 1u));
                for (uint32_t j = p; j > 0 && t_key[j - 1] != EMPTY; j--) r -= t_key[j - 1] > x;
                for (uint32_t j = p + 1; j < MT_CAP + MT_PAD && t_key[j] != EMPTY; j++) r += t_key[j] < x;
                spare[s0 + r] = ((uint64_t)t_cnt[p] << 32) | x;
            }
            pre += __popc(occ);
        }
        if (threadIdx.x == 0) s.distinct[u] = total;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Units
// ---------------------------------------------------------------------------
static constexpr int MU_PER = MU_CAP / MU_T;  // keys per thread
static_assert(MU_CAP % MU_T == 0 && MU_CAP < 65536, "whole keys per thread, positions of 16 bits");

struct UnitSmem {
    uint32_t cnt[MU_BUCKETS / 2 + 4];  // per bucket, two to a word: keys, then the first position
    uint32_t a[MU_CAP], b[MU_CAP];     // keys by bucket, sorted keys
    uint32_t hot[MU_CAP / MU_HOT];
    uint32_t warp[MU_T / 32], warp2[MU_T / 32];
    uint32_t next, prefix, nhot, sum;
};

// A unit's keys, sorted into S.b (all threads pass its barriers). A key's
// bucket are its top bits; there are two buckets for a key, each key ranks
// itself among its bucket's few; a bucket of more than MU_HOT keys (copies of
// a hot key) is sorted by a warp, value by value.
__device__ __forceinline__ void unit_sort(UnitSmem &S, const uint32_t (&key)[MU_PER], uint32_t c, uint32_t bs)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint16_t *first = reinterpret_cast<const uint16_t *>(S.cnt);
    uint32_t at[(MU_PER + 1) / 2];  // two ranks to a register
    for (uint32_t k = threadIdx.x; k < MU_BUCKETS / 8; k += MU_T) reinterpret_cast<uint4 *>(S.cnt)[k] = make_uint4(0, 0, 0, 0);
    if (threadIdx.x == 0) S.nhot = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < MU_PER; r++) {
        if (r * MU_T >= c) break;
        if (r * MU_T + threadIdx.x < c) {
            const uint32_t bk = key[r] >> bs, sh = (bk & 1u) * 16u;
            const uint32_t rank = (atomicAdd(&S.cnt[bk >> 1], 1u << sh) >> sh) & 0xffffu;  // (no half carries)
            at[r / 2] = r & 1 ? at[r / 2] | (rank << 16) : rank;
        }
    }
    __syncthreads();
    {
        constexpr int WPT = MU_BUCKETS / 2 / MU_T;  // words per thread
        uint32_t x[WPT], sum = 0;
        uint4 *w = reinterpret_cast<uint4 *>(S.cnt) + threadIdx.x * (WPT / 4);
#pragma unroll
        for (int q = 0; q < WPT / 4; q++) {
            const uint4 y = w[q];
            x[4 * q] = y.x;
            x[4 * q + 1] = y.y;
            x[4 * q + 2] = y.z;
            x[4 * q + 3] = y.w;
        }
#pragma unroll
        for (int q = 0; q < WPT; q++) {
            const uint32_t lo = x[q] & 0xffffu, hi = x[q] >> 16;
            if (lo > MU_HOT) S.hot[atomicAdd(&S.nhot, 1u)] = 2 * (threadIdx.x * WPT + q);
            if (hi > MU_HOT) S.hot[atomicAdd(&S.nhot, 1u)] = 2 * (threadIdx.x * WPT + q) + 1;
            x[q] = sum | ((sum + lo) << 16);
            sum += lo + hi;
        }
        const uint32_t pre = cta_scan<MU_T>(sum, S.warp) * 0x00010001u;
#pragma unroll
        for (int q = 0; q < WPT / 4; q++)
            w[q] = make_uint4(x[4 * q] + pre, x[4 * q + 1] + pre, x[4 * q + 2] + pre, x[4 * q + 3] + pre);
        if (threadIdx.x == 0) S.cnt[MU_BUCKETS / 2] = c;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < MU_PER; r++) {
        if (r * MU_T >= c) break;
        if (r * MU_T + threadIdx.x < c) S.a[first[key[r] >> bs] + ((at[r / 2] >> (r & 1 ? 16 : 0)) & 0xffffu)] = key[r];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < MU_PER; r++) {
        if (r * MU_T >= c) break;
        if (r * MU_T + threadIdx.x >= c) break;
        const uint32_t bk = key[r] >> bs, s = first[bk], e = first[bk + 1];
        const uint32_t me = s + ((at[r / 2] >> (r & 1 ? 16 : 0)) & 0xffffu);
        if (e - s > MU_HOT) continue;
        uint32_t p = s;
        if (e - s > 1)
            for (uint32_t j = s; j < e; j++) {
                const uint32_t x = S.a[j];
                p += x < key[r] || (x == key[r] && j < me);
            }
        S.b[p] = key[r];
    }
    for (uint32_t h = warp; h < S.nhot; h += MU_T / 32) {
        const uint32_t s = first[S.hot[h]], e = first[S.hot[h] + 1];
        // per pass: the copies of the last smallest value, and the next one
        uint32_t o = s, val = EMPTY;
        while (true) {
            uint32_t q = 0, mn = EMPTY;
#pragma unroll 4
            for (uint32_t j = s + lane; j < e; j += 32) {
                const uint32_t x = S.a[j];
                q += x == val;
                if (val == EMPTY || x > val) mn = min(mn, x);
            }
            q = __reduce_add_sync(0xffffffffu, q);
            mn = __reduce_min_sync(0xffffffffu, mn);
            for (uint32_t j = o + lane; j < o + q; j += 32) S.b[j] = val;
            o += q;
            if (o >= e) break;
            val = mn;
        }
    }
    __syncthreads();
}

// The groups of every unit. ORDERED: one after another, each unit's behind
// those of the units before it (look-back in ticket order). Else each unit's
// where its keys were, from st[u] on, with a start behind its last group:
// consumers that know their unit need no more, and nobody waits for a slow
// unit (2.4e8 uniform keys 2.67 ms ordered, 2.25 ms in place; Zipf keys, whose
// units differ, 4.36 and 1.97 ms). CTAs stay and fetch the next unit's keys
// while this one's groups are written. v: the keys by unit; pairs: the
// oversized units' groups. Bound by instructions and the barriers between the
// steps. Nothing is done, and *m_out stays 0, when the units were given up.
template <bool ORDERED>
__global__ void __launch_bounds__(MU_T, 6) msd_units(const uint64_t *__restrict__ v, MsdScratch s,
                                                     const uint32_t *__restrict__ st, uint32_t units, uint32_t rbits,
                                                     const uint64_t *__restrict__ pairs, uint64_t *__restrict__ uniq,
                                                     uint32_t *__restrict__ start, uint32_t *m_out,
                                                     unsigned long long *status)
{
    __shared__ __align__(16) UnitSmem S;
    if (s.misc[4]) return;
    const uint32_t mask = (1u << rbits) - 1u, bs = rbits > MU_BBITS ? rbits - MU_BBITS : 0u;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long *look = reinterpret_cast<unsigned long long *>(s.look);
    uint32_t u = blockIdx.x, s0 = 0, c = 0, groups = 0;
    if (ORDERED) {
        if (threadIdx.x == 0) S.next = atomicAdd(&s.misc[0], 1u);
        __syncthreads();
        u = S.next;
    }
    uint32_t key[MU_PER];
    auto fetch = [&] {
        s0 = st[u];
        c = st[u + 1] - s0;
        if (c > MU_CAP) return;
#pragma unroll
        for (int r = 0; r < MU_PER; r++) {
            if (r * MU_T >= c) break;
            if (r * MU_T + threadIdx.x < c) key[r] = (uint32_t)__ldcs(v + s0 + r * MU_T + threadIdx.x) & mask;
        }
    };
    if (u < units) fetch();
    while (u < units) {
        const uint64_t top = (uint64_t)u << rbits;
        const uint32_t unit = u, i0 = s0, n = c;
        __syncthreads();  // every thread has read S.next, and is done with the last unit
        if (ORDERED && threadIdx.x == 0) S.next = atomicAdd(&s.misc[0], 1u);
        uint32_t total = 0, pre = 0;
        uint32_t firsts[MU_PER];  // runs of equal keys: warp w looks at positions [w * span, (w + 1) * span)
        const uint32_t span = (n + MU_T - 1) / MU_T * 32;
        if (n > MU_CAP) {
            total = s.distinct[unit];
        } else {
            unit_sort(S, key, n, bs);
            uint32_t mine = 0;
#pragma unroll
            for (int q = 0; q < MU_PER; q++) {
                if (q * 32 >= span) break;
                const uint32_t i = warp * span + q * 32 + lane;
                firsts[q] = __ballot_sync(0xffffffffu, i < n && (i == 0 || S.b[i] != S.b[i - 1]));
                mine += __popc(firsts[q]);
            }
            if (lane == 0) S.warp2[warp] = mine;
            __syncthreads();
#pragma unroll
            for (int w = 0; w < MU_T / 32; w++) {
                if (w < warp) pre += S.warp2[w];
                total += S.warp2[w];
            }
        }
        uint32_t g0 = i0;
        if (ORDERED) {
            if (warp == 0) {
                const uint32_t prefix = lookback_prefix(look, unit, total, status);
                if (lane == 0) S.prefix = prefix;
            }
            __syncthreads();
            g0 = S.prefix;
            u = S.next;
        } else {
            if (threadIdx.x == 0) s.distinct[unit] = total;
            groups += total;
            u += gridDim.x;
        }
        if (u < units) fetch();  // the next unit's keys, needed after this one's groups
        if (n > MU_CAP) {
            uint32_t at = i0;
            for (uint32_t base = 0; base < total; base += MU_T) {
                const uint32_t i = base + threadIdx.x;
                const uint64_t x = i < total ? pairs[i0 + i] : 0ull;
                const uint32_t w = (uint32_t)(x >> 32), before = cta_scan<MU_T>(w, S.warp);
                if (threadIdx.x == MU_T - 1) S.sum = before + w;
                if (i < total) {
                    uniq[g0 + i] = top | (uint32_t)x;
                    start[g0 + i] = at + before;
                }
                __syncthreads();
                at += S.sum;
            }
        } else {
            uint32_t g = g0 + pre;
#pragma unroll
            for (int q = 0; q < MU_PER; q++) {
                if (q * 32 >= span) break;
                if ((firsts[q] >> lane) & 1u) {
                    const uint32_t i = warp * span + q * 32 + lane, at = g + __popc(firsts[q] & ((1u << lane) - 1u));
                    uniq[at] = top | S.b[i];
                    start[at] = i0 + i;
                }
                g += __popc(firsts[q]);
            }
        }
        if (threadIdx.x == 0 && (ORDERED ? unit == units - 1 : total < n || unit == units - 1)) {
            start[g0 + total] = i0 + n;
            if (ORDERED) *m_out = g0 + total;
        }
    }
    if (!ORDERED && threadIdx.x == 0 && groups) atomicAdd(m_out, groups);
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
bool msd_groups(const uint64_t *keys, uint64_t n, const PHash &H, uint32_t bits, uint32_t max_k, uint64_t *buf_a,
                uint64_t *buf_b, uint64_t *uniq, uint32_t *start, uint32_t *m_out, uint32_t *tmp, uint64_t tmp_words,
                DevCounters *ctr, cudaStream_t st, MsdUnits *units_out)
{
    if (n < 2048 || n >= (1ull << 30)) return false;
    // units of 1024 to 2048 keys on average: what a CTA sorts is eleven deviations
    // above the mean of a uniform batch's units
    uint32_t k = 1;
    while (k < bits && (n >> k) > 2048) k++;
    const bool ordered = units_out == nullptr;
    if (!ordered && k > max_k) {  // units at least as wide as asked for: means up to six deviations below the cap still fit
        if (k > max_k + 1 || (n >> max_k) > MU_CAP - 6 * 45) return false;
        k = max_k;
    }
    const bool two = k > 9;
    const uint32_t b1 = two ? (k + 1) / 2 : k, b2 = k - b1, rbits = bits - k;
    if (k == 0 || k > 18 || rbits > 31) return false;
    const MsdScratch s = msd_scratch(tmp, n, k, two, ordered, true);
    if (s.words > tmp_words) return false;
    const uint32_t units = 1u << k;
    uint64_t *const v = two ? buf_b : buf_a, *const pairs = two ? buf_a : buf_b;
    cudaMemsetAsync(tmp, 0, s.zero_words * 4, st);
    const unsigned tiles = (unsigned)((n + MP_TILE - 1) / MP_TILE);
    {
        TraceScope ts_("msd_hist1", n, st);
        const int g = grid_for(tiles * (uint64_t)MP_T, MP_T, 4);
        msd_hist1<<<g, MP_T, 0, st>>>(keys, n, H, bits - b1, 1u << b1, s, two, m_out);
    }
    {
        TraceScope ts_("msd_part", n, st);
        msd_part<true><<<tiles, MP_T, 0, st>>>(keys, (uint32_t)n, H, s, 0, bits - b1, b1, buf_a, nullptr);
    }
    if (two) msd_second_pass(s, buf_a, buf_b, n, 1u << b1, rbits, b2, "msd_hist2", "msd_part2", st);
    const uint32_t *ust = two ? s.st2 : s.st1;
    if (n > MS_CHUNK) {
        TraceScope ts_("msd_squeeze", 0, st);
        msd_squeeze<<<grid_for(n / MS_CHUNK * MU_T, MU_T, 6), MU_T, 0, st>>>(v, s, ust, rbits);
    }
    {
        TraceScope ts_("msd_big", 0, st);
        msd_big<<<grid_for(n / MU_CAP * MU_T, MU_T, 6), MU_T, 0, st>>>(v, s, ust, rbits, pairs);
    }
    TraceScope ts_("msd_units", n, st);
    const int g = grid_for((uint64_t)units * MU_T, MU_T, 6);
    if (ordered) {
        msd_units<true><<<g, MU_T, 0, st>>>(v, s, ust, units, rbits, pairs, uniq, start, m_out, &ctr->status);
    } else {
        msd_units<false><<<g, MU_T, 0, st>>>(v, s, ust, units, rbits, pairs, uniq, start, m_out, &ctr->status);
        *units_out = MsdUnits{ust, s.distinct, k};
    }
    return true;
}

}  // namespace gf
