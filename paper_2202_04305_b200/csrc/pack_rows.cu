// sp_pack for matrices with a compressed inner level and moderate segments (rows of CSR and DCSR, columns of
// CSC and DCSC): no sort by key, the entries pass through memory twice.
//
//   1. k_rows_count      (where slots of kCap records would not follow the entries) entries per bucket, a bucket being
//                        a range of outer indices, and where every bucket begins
//   2. k_rows_partition  (k_rows_partition_tiles from kSmall entries on) range check; entries to their buckets, in any order
//   3. k_rows_build      a block per bucket: entries per outer index, order inside every segment, and
//                        everything the bucket contributes to the storage, written in order
//   4. k_rows_outer      (compressed outer level) the buckets' lists of stored outer indices, joined
//   5. k_rows_close_up   (duplicate coordinates only) the buckets' entries moved together
//
// Buckets hold about kAverage entries and at most kCap.  Random accesses are what a GPU is slow at (about 140 G
// single-lane accesses/s here, hit or miss): this way an entry costs at most one, its 16-byte store in step 2; every
// other scattered access stays in shared memory.  Sizes are known beforehand (a compressed outer level's are
// bounded), so the one read-back comes at the end.  Duplicate coordinates are found and their values summed, in input
// order, inside the bucket's block; what it stores then ends short of its place, and step 5 closes the gaps, in
// arrays of the right size: 5 M entries with one coordinate repeated 270 us, four times each 385, by radix 330
// and 416; 10,486 entries 62 and 99.  A bucket that overflows (long or very uneven segments) is found on the device
// too; the kernels after that return and the caller takes the radix path.
//
// Without step 1 a bucket has a slot of kCap records, 2.5 times what it holds on average and 16 times in small inputs; it
// runs where slots would take more than 16 records an entry, the rows being many more than the entries, and makes
// the scratch 16 bytes an entry then (1,000 entries in 8 M rows: 0.1 MB, 336 MB in slots).  For all inputs it would cost 3 us
// of 40 and more (300,000 entries 43.5 us against 40.0, 1 M 67 against 64, 5 M 198 against 192).
#include "common.cuh"

#include <stddef.h>

#include <algorithm>

namespace {

constexpr int kCThreads = 1024, kCBlocks = 148; // of k_rows_count
constexpr int kThreads = 512;                   // of k_rows_partition
constexpr int kBThreads = 512;                  // of k_rows_build and k_rows_outer
constexpr int kWarps = kBThreads / 32;
// Entries a bucket can hold: a block orders them in shared memory, two blocks to an SM.  With 4096, 5 M uniform entries
// took 188 us against 196, but power-law rows (mean 16, deviation 54) overflow such buckets and take the radix path: 3.2 M
// of them 279 us against 150, a conversion of 2 M 190 against 123.
constexpr int kCap = 5120;
constexpr int kIpt = kCap / kBThreads;          // ... per thread of k_rows_build
constexpr int kAverage = 2048;                  // entries per bucket aimed at
constexpr int kAverageSmall = 320;               // ... of a small input, for more blocks
// Entries below which an input counts as small: buckets of kAverageSmall entries, stored from where they were read.  60,000
// entries in rows of 16 and of 100: 36.4 and 38 us, the other way 38 and 39; 80,000: 40.2 and 43.2, 39.5 and 39.4;
// 200,000: 51.5 and 56.4, 39.3 and 39.7; 299,999: 60.6 and 67.9, 40.0 and 40.5.
constexpr int64_t kSmall = 80000;
constexpr int kWidth = 2048;                    // outer indices of a bucket
constexpr int kMaxBuckets = 4096;
constexpr int kDense = 24;                      // mean compares per entry above which segments are cut into bins

// What the device reports, straight into the caller's pinned words: one word per event, then the number of
// non-empty outer indices; the last is where the number of duplicates is read back to.  `stop` is the device's own copy: later blocks and kernels return once it is set.
enum { kErrRange = 0, kErrDup, kErrLong, kOuterCount, kLost };
__device__ __forceinline__ void report(int what, uint32_t* stop, unsigned long long* host) {
    *static_cast<volatile unsigned long long*>(host + what) = 1;
    *static_cast<volatile uint32_t*>(stop) = 1;
}

// Where bucket b's records begin, its slot being the b-th of `slot` records (0: buckets side by side, ends in cursor).
__device__ __forceinline__ uint32_t records_of(uint32_t b, uint32_t slot, const uint32_t* cursor) {
    return slot ? b * slot : b ? cursor[b - 1] : 0u;
}

// Value (low, high word) and 64 bits: the low kOffBits of the outer coordinate, which tell a bucket's apart, the
// entry's number in the input, the inner coordinate in its inner_bits (low, high word).
using Rec = uint4;
constexpr int kOffBits = 11, kOffShift = 64 - kOffBits;
static_assert(1 << kOffBits == kWidth, "a bucket's outer indices differ in their low bits");
__device__ __forceinline__ Rec make_rec(double v, uint32_t outer, uint32_t number, uint32_t inner, int inner_bits) {
    return make_uint4((uint32_t)__double2loint(v), (uint32_t)__double2hiint(v), __funnelshift_lc(0u, number, inner_bits) | inner,
                      outer << (kOffShift - 32) | __funnelshift_lc(number, 0u, inner_bits));
}

// Outer index o lies in bucket o * scale / 2^32; bucket b begins at the first o that the formula gives b for.
__host__ __device__ __forceinline__ int64_t bucket_begin(int64_t b, uint32_t scale, int64_t no) {
    const int64_t o = (int64_t)((((uint64_t)b << 32) + scale - 1) / scale);
    return o < no ? o : no;
}

// Whether some block has reported an error, the same answer for all threads of a block.
__device__ __forceinline__ bool stopped(const uint32_t* stop) {
    return __syncthreads_or(threadIdx.x == 0 && __ldcg(stop) != 0) != 0;
}

// Exclusive scan over a block of WARPS warps of one counter per thread.
template <int WARPS = kWarps>
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* s_w, uint32_t* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    uint32_t pre = 0, tot = 0;
#pragma unroll
    for (int i = 0; i < WARPS; ++i) {
        const uint32_t s = s_w[i];
        if (i < w) pre += s;
        tot += s;
    }
    __syncthreads();
    *total = tot;
    return incl - v + pre;
}

// In-place exclusive scan of s[0 .. n), n <= PER * kBThreads; s[n] = the total.
template <int PER>
__device__ __forceinline__ void scan_shared(uint32_t* s, int n, uint32_t* s_w) {
    const int i0 = threadIdx.x * PER;
    uint32_t v[PER], mine = 0, tot;
#pragma unroll
    for (int i = 0; i < PER; ++i) { v[i] = i0 + i < n ? s[i0 + i] : 0u; mine += v[i]; }
    uint32_t at = block_scan(mine, s_w, &tot);
#pragma unroll
    for (int i = 0; i < PER; ++i)
        if (i0 + i < n) { s[i0 + i] = at; at += v[i]; }
    if (threadIdx.x == 0) s[n] = tot;
    __syncthreads();
}

// Entries per bucket, in shared memory per block and then added up in cursor (cleared before), and, by the last block,
// where the buckets begin: cursor[b], which the partition advances to where bucket b ends.  Few blocks, since each
// adds up to kMaxBuckets counters.
template <typename CT>
__global__ void __launch_bounds__(kCThreads)
k_rows_count(const CT* __restrict__ oc, int64_t n, int64_t no, uint32_t scale, int nb, uint32_t* cursor, uint32_t* stop, uint32_t* ticket,
             unsigned long long* host) {
    constexpr int kU = 16, kPerB = kMaxBuckets / kCThreads;
    __shared__ uint32_t s_hist[kMaxBuckets];
    __shared__ uint32_t s_w[kCThreads / 32];
    __shared__ bool s_last;
    sp_release_next_kernel();                       // it ranks its entries before it waits for the cursors
    const int t = threadIdx.x;
    for (int b = t; b < nb; b += kCThreads) s_hist[b] = 0u;
    __syncthreads();
    for (int64_t base = (int64_t)blockIdx.x * (kCThreads * kU); base < n; base += (int64_t)gridDim.x * (kCThreads * kU)) {
        CT o[kU];
#pragma unroll
        for (int i = 0; i < kU; ++i) o[i] = base + i * kCThreads + t < n ? oc[base + i * kCThreads + t] : (CT)-1;
#pragma unroll
        for (int i = 0; i < kU; ++i)                // the partition reports what is out of range
            if (o[i] >= 0 && (int64_t)o[i] < no) atomicAdd(&s_hist[__umulhi((uint32_t)o[i], scale)], 1u);
    }
    __syncthreads();
    for (int b = t; b < nb; b += kCThreads)
        if (s_hist[b]) atomicAdd(cursor + b, s_hist[b]);
    __threadfence();
    __syncthreads();
    if (t == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int b = t; b < nb; b += kCThreads) s_hist[b] = __ldcg(cursor + b);
    __syncthreads();
    uint32_t k[kPerB], mine = 0, tot;
    bool full = false;
#pragma unroll
    for (int q = 0; q < kPerB; ++q) {
        const int b = t * kPerB + q;
        k[q] = b < nb ? s_hist[b] : 0u;
        full |= k[q] > (uint32_t)kCap;
        mine += k[q];
    }
    uint32_t at = block_scan<kCThreads / 32>(mine, s_w, &tot);
#pragma unroll
    for (int q = 0; q < kPerB; ++q) {
        const int b = t * kPerB + q;
        if (b < nb) cursor[b] = at;
        at += k[q];
    }
    if (__syncthreads_or(full) && t == 0) report(kErrLong, stop, host);
}

// A block sends a tile of kThreads * PER entries to their buckets: ranks inside the tile by shared-memory
// atomics, the tile's place in every bucket by one atomic on the bucket's cursor.
template <typename CT, int PER>
__global__ void __launch_bounds__(kThreads, 2)
k_rows_partition(const CT* __restrict__ oc, const CT* __restrict__ ic, const double* __restrict__ vals, int64_t n, int64_t no, int64_t ni,
                 uint32_t scale, int inner_bits, int nb, uint32_t slot, uint32_t* cursor, Rec* __restrict__ rec, uint32_t* stop, unsigned long long* host) {
    extern __shared__ uint32_t s_hist[];
    const int t = threadIdx.x;
    for (int b = t; b < nb; b += kThreads) s_hist[b] = 0u;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * (kThreads * PER) + t;
    CT o[PER], c[PER];
    uint32_t r[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int64_t e = base + i * kThreads;
        o[i] = e < n ? oc[e] : (CT)0;
        c[i] = e < n ? ic[e] : (CT)0;
    }
    bool bad = false;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        if (o[i] < 0 || (int64_t)o[i] >= no || c[i] < 0 || (int64_t)c[i] >= ni) { bad = true; o[i] = 0; }
        r[i] = base + i * kThreads < n ? atomicAdd(&s_hist[__umulhi((uint32_t)o[i], scale)], 1u) : 0u;
    }
    bad = __syncthreads_or(bad) != 0;
    sp_wait_for_previous_kernel();
    if (stopped(stop)) return;
    if (bad) {
        if (t == 0) report(kErrRange, stop, host);
        return;
    }
    // all cursors of a thread at once: one wait, not one per bucket
    constexpr int kPerB = kMaxBuckets / kThreads;
    uint32_t k[kPerB], at[kPerB];
#pragma unroll
    for (int q = 0; q < kPerB; ++q) {
        const int b = t + q * kThreads;
        k[q] = b < nb ? s_hist[b] : 0u;
        at[q] = k[q] ? atomicAdd(cursor + b, k[q]) : 0u;
    }
    bool full = false;
#pragma unroll
    for (int q = 0; q < kPerB; ++q)
        if (k[q]) {
            const uint32_t b = t + q * kThreads;
            full |= slot && at[q] + k[q] > slot;
            s_hist[b] = at[q] + b * slot;
        }
    if (__syncthreads_or(full)) {
        if (t == 0) report(kErrLong, stop, host);
        return;
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int64_t e = base + i * kThreads;
        if (e < n) {
            const uint32_t b = __umulhi((uint32_t)o[i], scale);
            const double v = vals[e];
            rec[s_hist[b] + r[i]] = make_rec(v, (uint32_t)o[i], (uint32_t)e, (uint32_t)c[i], inner_bits);
        }
    }
}

// The same for large inputs, the tile being put in order by bucket in shared memory first: a bucket's entries then
// leave side by side and one store instruction touches fewer lines, and the values, requested with the coordinates,
// are no longer waited for at the end.  5 M entries: pack 190 us (196 with the present kCap), 205 with every entry stored from where it was
// read; 1.5 M with 64-bit coordinates (convert) 98 against 106; 2.5 M 128 against 146.  Tiles of 4096 entries spill
// (188, 102), 1024 threads with 6 entries each 190, 98, 8 entries 192, 102, three blocks per SM 204, 103.
constexpr int kTIpt = 6, kTTile = kThreads * kTIpt;
struct TileShared {
    Rec rec[kTTile];
    uint32_t to[kTTile];                        // where an entry goes among the records
    uint32_t counters[2 * kMaxBuckets];         // of as many buckets as there are: shared memory not taken is L1 for the loads
    static constexpr size_t bytes(int nb) { return offsetof(TileShared, counters) + 2 * (size_t)nb * sizeof(uint32_t); }
};

template <typename CT>
__global__ void __launch_bounds__(kThreads, 2)
k_rows_partition_tiles(const CT* __restrict__ oc, const CT* __restrict__ ic, const double* __restrict__ vals, int64_t n, int64_t no, int64_t ni,
                       uint32_t scale, int inner_bits, int nb, uint32_t slot, uint32_t* cursor, Rec* __restrict__ rec, uint32_t* stop, unsigned long long* host) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    TileShared& s = *reinterpret_cast<TileShared*>(s_raw);
    uint32_t* const s_count = s.counters;           // entries of the tile per bucket, then where they begin in rec
    uint32_t* const s_shift = s.counters + nb;      // place of the bucket's entries of this tile among the records minus place in rec
    __shared__ uint32_t s_w[kThreads / 32];
    const int t = threadIdx.x;
    for (int b = t; b < nb; b += kThreads) s_count[b] = 0u;
    const int64_t base = (int64_t)blockIdx.x * kTTile;
    const int cnt = (int)(n - base < kTTile ? n - base : kTTile);
    uint32_t o[kTIpt], c[kTIpt], r[kTIpt];
    double v[kTIpt];
    bool bad = false;
    CT oo[kTIpt], cc[kTIpt];
#pragma unroll
    for (int i = 0; i < kTIpt; ++i) {
        const int j = i * kThreads + t;
        oo[i] = j < cnt ? oc[base + j] : (CT)0;
        cc[i] = j < cnt ? ic[base + j] : (CT)0;
        v[i] = j < cnt ? vals[base + j] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kTIpt; ++i) {
        const bool out = oo[i] < 0 || (int64_t)oo[i] >= no || cc[i] < 0 || (int64_t)cc[i] >= ni;
        bad |= out;
        o[i] = out ? 0u : (uint32_t)oo[i];
        c[i] = (uint32_t)cc[i];
        r[i] = i * kThreads + t < cnt ? atomicAdd(&s_count[__umulhi(o[i], scale)], 1u) : 0u;
    }
    bad = __syncthreads_or(bad) != 0;
    sp_wait_for_previous_kernel();
    if (stopped(stop)) return;
    if (bad) {
        if (t == 0) report(kErrRange, stop, host);
        return;
    }
    // all cursors of a thread at once: one wait, not one per bucket
    constexpr int kPerB = (kMaxBuckets + kThreads - 1) / kThreads;
    uint32_t at[kPerB], mine = 0;
#pragma unroll
    for (int q = 0; q < kPerB; ++q) {
        const int b = t + q * kThreads;
        const uint32_t k = b < nb ? s_count[b] : 0u;
        at[q] = k ? atomicAdd(cursor + b, k) : 0u;
        mine += k;
    }
    const int lane = t & 31, w = t >> 5;
    uint32_t incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += u;
    }
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    uint32_t from = incl - mine;
#pragma unroll
    for (int i = 0; i < kThreads / 32; ++i) from += i < w ? s_w[i] : 0u;
    bool full = false;
#pragma unroll
    for (int q = 0; q < kPerB; ++q) {
        const int b = t + q * kThreads;
        const uint32_t k = b < nb ? s_count[b] : 0u;    // read again: registers
        if (k) {
            full |= slot && at[q] + k > slot;
            s_count[b] = from;
            s_shift[b] = at[q] + (uint32_t)b * slot - from;
            from += k;
        }
    }
    if (__syncthreads_or(full)) {
        if (t == 0) report(kErrLong, stop, host);
        return;
    }
#pragma unroll
    for (int i = 0; i < kTIpt; ++i)
        if (i * kThreads + t < cnt) {
            const uint32_t b = __umulhi(o[i], scale), at = s_count[b] + r[i];
            s.rec[at] = make_rec(v[i], o[i], blockIdx.x * (uint32_t)kTTile + i * kThreads + t, c[i], inner_bits);
            s.to[at] = s_shift[b] + at;
        }
    __syncthreads();
#pragma unroll 4
    for (int j = t; j < cnt; j += kThreads) {
        rec[s.to[j]] = s.rec[j];
    }
}

struct BuildShared {
    uint32_t count[kWidth + 1];                 // entries, then starts, of the bucket's outer indices
    uint32_t crd[kCap];
    union {
        double val[kCap];
        struct { uint32_t lo[kWidth], hi[kWidth]; };        // smallest and largest coordinate of a segment
        struct { double unused[kCap / 2]; uint32_t bin[kCap]; };
        struct { uint32_t times[kCap], number[kCap]; };     // of equal coordinates, at their place: how many, and which in the input
    };
    uint32_t bin_end;                           // bin[kCap] when the bucket is full
    uint32_t w[kWarps];
    uint32_t compares, places;                  // sums over the block
    uint16_t seg[kCap];                         // outer offsets of the entries, in order
};
static_assert(sizeof(uint32_t) * 2 * kWidth <= sizeof(double) * kCap / 2, "lo and hi lie before bin");

// The place of an entry is the start of its segment plus the number of smaller coordinates in it, counted over
// shared memory.  Where segments are long (more than kDense compares per entry on average) they are first
// cut into as many bins as they have entries, evenly between their smallest and largest coordinate, and only
// the entries of one bin are compared.  first[b]: the entries before bucket b; lost[b]: the duplicates in it; *total: in all.
template <typename P, typename I, bool DBL>
__global__ void __launch_bounds__(kBThreads, 2)
k_rows_build(Rec* rec, const uint32_t* cursor, int64_t n, int64_t no, uint32_t scale, int inner_bits, int nb, uint32_t slot, uint32_t* stop, uint32_t* __restrict__ first, uint32_t* lost,
             uint32_t* total, unsigned long long* host,
             P* __restrict__ pos1, I* __restrict__ crd, double* __restrict__ val, uint32_t* __restrict__ seg_out, uint32_t* __restrict__ outer_count) {
    sp_wait_for_previous_kernel();
    if (stopped(stop)) return;
    extern __shared__ __align__(16) unsigned char s_raw[];
    BuildShared& s = *reinterpret_cast<BuildShared*>(s_raw);
    const int t = threadIdx.x, b = blockIdx.x;
    const uint32_t place = records_of(b, slot, cursor);
    const int cnt = (int)(slot ? cursor[b] : cursor[b] - place);
    const uint32_t lo = (uint32_t)bucket_begin(b, scale, no);
    const int width = (int)((b + 1 < nb ? bucket_begin(b + 1, scale, no) : no) - lo);
    // entries of this thread, requested first; the values are fetched again at the end (registers)
    const Rec* mine = rec + place + t;
    const uint32_t inner_mask = inner_bits < 32 ? (1u << inner_bits) - 1u : ~0u;
    uint32_t c[kIpt], qr[kIpt];                 // inner coordinate; outer offset << 16 | rank, later the place
#pragma unroll
    for (int i = 0; i < kIpt; ++i) {
        c[i] = qr[i] = 0u;
        if (i * kBThreads + t < cnt) {
            const Rec x = mine[i * kBThreads];
            c[i] = x.z & inner_mask;
            qr[i] = ((x.w >> (kOffShift - 32)) - lo) & (kWidth - 1);
        }
    }
    for (int q = t; q < width; q += kBThreads) { s.count[q] = 0u; s.lo[q] = ~0u; s.hi[q] = 0u; }
    if (t == 0) s.compares = s.places = 0u;
    uint32_t before = 0, base = place;          // base: entries in the buckets before
    if (slot) {
        for (int q = t; q < b; q += kBThreads) before += cursor[q];
        block_scan(before, s.w, &base);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kIpt; ++i)
        if (i * kBThreads + t < cnt) qr[i] = qr[i] << 16 | atomicAdd(&s.count[qr[i]], 1u);
    __syncthreads();
    uint32_t sq = 0;                            // mean number of compares without bins
    constexpr int kPerW = kWidth / kBThreads;
#pragma unroll
    for (int i = 0; i < kPerW; ++i) {
        const int q = t * kPerW + i;
        const uint32_t k = q < width ? s.count[q] : 0u;
        sq += k * k;                            // at most kCap^2 in all
    }
    sq = __reduce_add_sync(0xffffffffu, sq);
    if (sp_lane() == 0) atomicAdd(&s.compares, sq);
    scan_shared<kPerW>(s.count, width, s.w);    // (also the barrier after that)
    const bool bins = s.compares > (uint32_t)kDense * (uint32_t)cnt;
    if (!DBL) {
        for (int q = t; q < width; q += kBThreads) pos1[lo + q] = (P)(base + s.count[q]);
        if (b == nb - 1 && t == 0) pos1[no] = (P)n;
    }
    // place of coordinate c among s.crd[j .. e), and the sum of the thread's places
    uint32_t sum = 0;
    auto place_of = [&](int j, int e, uint32_t cc) {
        uint32_t at = (uint32_t)j;
        for (; j + 1 < e; j += 2) {
            const uint32_t c0 = s.crd[j], c1 = s.crd[j + 1];
            at += c0 < cc;
            at += c1 < cc;
        }
        if (j < e) at += s.crd[j] < cc;
        sum += at;
        return at;
    };
    uint32_t to[kIpt];                          // outer offset << 16 | place
    if (!bins) {
#pragma unroll
        for (int i = 0; i < kIpt; ++i)
            if (i * kBThreads + t < cnt) s.crd[s.count[qr[i] >> 16] + (qr[i] & 0xffffu)] = c[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kIpt; ++i)
            if (i * kBThreads + t < cnt) {
                const uint32_t q = qr[i] >> 16;
                to[i] = q << 16 | place_of((int)s.count[q], (int)s.count[q + 1], c[i]);
            }
    } else {
#pragma unroll
        for (int i = 0; i < kIpt; ++i)
            if (i * kBThreads + t < cnt) {
                atomicMin(&s.lo[qr[i] >> 16], c[i]);
                atomicMax(&s.hi[qr[i] >> 16], c[i]);
            }
        for (int j = t; j < cnt; j += kBThreads) s.bin[j] = 0u;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kIpt; ++i)
            if (i * kBThreads + t < cnt) {
                const uint32_t q = qr[i] >> 16, first = s.count[q], len = s.count[q + 1] - first, c0 = s.lo[q];
                // not decreasing in the coordinate: the factor is the segment's, and rounding keeps the order
                const uint32_t k = (uint32_t)((float)(c[i] - c0) * ((float)len / ((float)(s.hi[q] - c0) + 1.0f)));
                const uint32_t g = first + (k < len ? k : len - 1u);
                to[i] = g << 16 | atomicAdd(&s.bin[g], 1u);
            }
        __syncthreads();
        scan_shared<kIpt>(s.bin, cnt, s.w);     // the total lands in bin[cnt], which is bin_end for a full bucket
#pragma unroll
        for (int i = 0; i < kIpt; ++i)
            if (i * kBThreads + t < cnt) s.crd[s.bin[to[i] >> 16] + (to[i] & 0xffffu)] = c[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kIpt; ++i)
            if (i * kBThreads + t < cnt) {
                const uint32_t g = to[i] >> 16;
                to[i] = (qr[i] & 0xffff0000u) | place_of((int)s.bin[g], (int)s.bin[g + 1], c[i]);
            }
    }
    // Distinct coordinates take the places 0 .. cnt - 1; of equal ones all get the lowest, so the sum falls short.
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (sp_lane() == 0) atomicAdd(&s.places, sum);
    __syncthreads();                            // coordinates and bins are dead from here on
    const bool dups = s.places != (uint32_t)(cnt * (cnt - 1) / 2);
    if (dups) {                                 // equal ones take successive places in the order of the input
        for (int j = t; j < cnt; j += kBThreads) s.times[j] = 0u;
        __syncthreads();
        auto number_of = [&](int j) {
            const uint2 k = reinterpret_cast<const uint2*>(rec + place + j)[1];
            return (uint32_t)((((uint64_t)k.y << 32 | k.x) << kOffBits) >> (kOffBits + inner_bits));
        };
#pragma unroll
        for (int i = 0; i < kIpt; ++i) s.crd[i * kBThreads + t] = to[i];       // kept there: the loops are not unrolled
#pragma unroll 1
        for (int j = t; j < cnt; j += kBThreads) {
            const uint32_t p = s.crd[j] & 0xffffu;
            s.number[p + atomicAdd(&s.times[p], 1u)] = number_of(j);
        }
        __syncthreads();
#pragma unroll 1
        for (int j = t; j < cnt; j += kBThreads) {
            const uint32_t p = s.crd[j] & 0xffffu, number = number_of(j);
            uint32_t smaller = 0;
            for (uint32_t k = 0; k < s.times[p]; ++k) smaller += s.number[p + k] < number;
            s.crd[j] += smaller;
        }
#pragma unroll
        for (int i = 0; i < kIpt; ++i) to[i] = s.crd[i * kBThreads + t];
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < kIpt; ++i)
        if (i * kBThreads + t < cnt) {
            const uint2 v = *reinterpret_cast<const uint2*>(mine + i * kBThreads);
            const uint32_t p = to[i] & 0xffffu;
            s.crd[p] = c[i];
            s.val[p] = __hiloint2double((int)v.y, (int)v.x);
            if (seg_out || dups) s.seg[p] = (uint16_t)(to[i] >> 16);
        }
    __syncthreads();
    uint32_t distinct = (uint32_t)cnt;
    if (!dups) {
        for (int j = t; j < cnt; j += kBThreads) {
            crd[base + j] = (I)s.crd[j];
            val[base + j] = s.val[j];
            if (seg_out) seg_out[base + j] = lo + s.seg[j];
        }
    } else {
        // the first of equal ones adds the others up and is stored; each thread takes kIpt adjacent entries
        const int j0 = t * kIpt;
        uint32_t heads = 0;
#pragma unroll 1
        for (int j = j0; j < j0 + kIpt && j < cnt; ++j)
            if (j == 0 || s.crd[j] != s.crd[j - 1] || s.seg[j] != s.seg[j - 1]) heads |= 1u << (j - j0);
        const uint32_t stored = block_scan(__popc(heads), s.w, &distinct);
        uint32_t at = base + stored;
#pragma unroll 1
        for (int j = j0; j < j0 + kIpt && j < cnt; ++j)
            if (heads >> (j - j0) & 1u) {
                double sum = s.val[j];
                for (int k = j + 1; k < cnt && s.crd[k] == s.crd[j] && s.seg[k] == s.seg[j]; ++k) sum += s.val[k];
                crd[at] = (I)s.crd[j];
                val[at] = sum;
                if (seg_out) seg_out[at] = lo + s.seg[j];
                ++at;
            }
        __syncthreads();
        at = stored;                            // from here on crd[j] is the number of entries stored before entry j
#pragma unroll 1
        for (int j = j0; j < j0 + kIpt && j < cnt; ++j) {
            s.crd[j] = at;
            at += heads >> (j - j0) & 1u;
        }
        __syncthreads();
        for (int q = t; q <= width; q += kBThreads) {
            const uint32_t j = s.count[q];
            s.count[q] = j < (uint32_t)cnt ? s.crd[j] : distinct;
            if (!DBL && q < width) pos1[lo + q] = (P)(base + s.count[q]);
        }
        __syncthreads();
        if (t == 0) {
            atomicAdd(total, (uint32_t)cnt - distinct);
            *static_cast<volatile unsigned long long*>(host + kErrDup) = 1;
        }
    }
    if (t == 0) { first[b] = base; lost[b] = (uint32_t)cnt - distinct; }
    if (DBL) {                                  // the stored indices and their first entries, in order, where the records were
        uint32_t filled = 0, all;
#pragma unroll
        for (int i = 0; i < kPerW; ++i) {
            const int q = t * kPerW + i;
            filled += q < width && s.count[q + 1] != s.count[q];
        }
        uint32_t k = block_scan(filled, s.w, &all);
#pragma unroll
        for (int i = 0; i < kPerW; ++i) {
            const int q = t * kPerW + i;
            if (q < width && s.count[q + 1] != s.count[q])
                *reinterpret_cast<uint2*>(rec + place + k++) = make_uint2(lo + q, base + s.count[q]);
        }
        if (t == 0) outer_count[b] = all;
    }
}

// After duplicates: the entries that every bucket stored, moved to where they belong; first and lost as k_rows_build left them.
template <typename P, typename I, bool DBL>
__global__ void __launch_bounds__(kBThreads)
k_rows_close_up(const uint32_t* __restrict__ first, const uint32_t* __restrict__ lost, int64_t n, int64_t stored, int64_t no, uint32_t scale, int nb,
                const P* __restrict__ pos1, const I* __restrict__ crd, const double* __restrict__ val, const uint32_t* __restrict__ seg,
                P* __restrict__ pos1_out, I* __restrict__ crd_out, double* __restrict__ val_out, uint32_t* __restrict__ seg_out) {
    __shared__ uint32_t s_w[kWarps];
    const int t = threadIdx.x, b = blockIdx.x;
    uint32_t mine = 0, before;
    for (int q = t; q < b; q += kBThreads) mine += lost[q];
    block_scan(mine, s_w, &before);
    const uint32_t from = first[b], to = from - before;
    const int cnt = (int)((b + 1 < nb ? first[b + 1] : (uint32_t)n) - from - lost[b]);
    for (int j = t; j < cnt; j += kBThreads) {
        crd_out[to + j] = crd[from + j];
        val_out[to + j] = val[from + j];
        if (seg) seg_out[to + j] = seg[from + j];
    }
    if (!DBL) {
        const int64_t lo = bucket_begin(b, scale, no), hi = b + 1 < nb ? bucket_begin(b + 1, scale, no) : no;
        for (int64_t o = lo + t; o < hi; o += kBThreads) pos1_out[o] = pos1[o] - (P)before;
        if (b == nb - 1 && t == 0) pos1_out[no] = (P)stored;
    }
}

// Joins the buckets' lists of non-empty outer indices and of their first entries: crd[0] and pos[1].  lost: entries
// that buckets hold less than they take up, nullptr = none.
template <typename P, typename I>
__global__ void __launch_bounds__(kBThreads)
k_rows_outer(const Rec* rec, const uint32_t* cursor, const uint32_t* outer_count, const uint32_t* lost, int64_t n, int nb, uint32_t slot,
             uint32_t* stop, unsigned long long* host, P* __restrict__ pos0, I* __restrict__ crd0, P* __restrict__ pos1) {
    sp_wait_for_previous_kernel();
    if (stopped(stop)) return;
    __shared__ uint32_t s_w[kWarps];
    const int t = threadIdx.x, b = blockIdx.x;
    uint32_t before = 0, base, gone = 0;
    if (lost) {
        for (int q = t; q < b; q += kBThreads) before += lost[q];
        block_scan(before, s_w, &gone);
        before = 0;
    }
    for (int q = t; q < b; q += kBThreads) before += outer_count[q];
    block_scan(before, s_w, &base);
    const Rec* list = rec + records_of(b, slot, cursor);
    const uint32_t cnt = outer_count[b];
    for (uint32_t q = t; q < cnt; q += kBThreads) {
        const uint2 x = *reinterpret_cast<const uint2*>(list + q);
        crd0[base + q] = (I)x.x;
        pos1[base + q] = (P)(x.y - gone);
    }
    if (b == nb - 1 && t == 0) {
        pos1[base + cnt] = (P)n;
        pos0[0] = 0;
        pos0[1] = (P)(base + cnt);
        *static_cast<volatile unsigned long long*>(host + kOuterCount) = base + cnt;
    }
}

}  // namespace

// Returns SP_OK with *out set; an error; or SP_ERR_UNSUPPORTED when the caller should take the radix path.
sp_status sp_pack_rows(const int64_t* dims, const int* ord, const int* lt, int64_t n, const void* outer, const void* inner, int coord_bits,
                       const double* vals, int posBits, int crdBits, unsigned flags, cudaStream_t stream, sp_tensor** out) {
    const int64_t no = dims[ord[0]], ni = dims[ord[1]];
    // narrow positions need the radix path's width checks; records hold 32-bit coordinates
    if (posBits < 32 || crdBits < 32 || no >= ((int64_t)1 << 31) || ni >= ((int64_t)1 << 32)) return SP_ERR_UNSUPPORTED;
    // A compressed outer level of many indices that hold nothing: the buckets are as many as its indices ask for and each costs
    // time, while a sort sees the entries alone.  1,000 entries in 2 M, 3 M, 4 M, 8 M rows: 66, 83, 90, 132 us, by radix
    // 62 to 79, 61, 61, 61; 300,000 entries in 3 M, 4 M, 8 M rows: 90, 97, 143 and 97 throughout; 1 M entries in 4 M,
    // 6 M rows: 106, 132 and 118; 3 M entries in 8 M rows: 202 and 206.
    if (lt[0] == SP_COMPRESSED && no > 3000000 + 2 * n) return SP_ERR_UNSUPPORTED;
    // enough buckets for the entries and for the outer indices, no more than there are outer indices
    int64_t buckets = std::max(sp_ceil_div(n, n < kSmall ? kAverageSmall : kAverage), sp_ceil_div(no, kWidth - 48));
    if (buckets > kMaxBuckets) return SP_ERR_UNSUPPORTED;
    if (buckets > no) {
        if (n > no * kCap) return SP_ERR_UNSUPPORTED;
        buckets = no;
    }
    const int nb = (int)buckets;
    int inner_bits = 1, number_bits = 1;                 // what a record holds beside the value has to fit
    while (((int64_t)1 << inner_bits) < ni) ++inner_bits;
    while (((int64_t)1 << number_bits) < n) ++number_bits;
    if (inner_bits + number_bits > kOffShift) return SP_ERR_UNSUPPORTED;
    const uint32_t scale = (uint32_t)std::min<uint64_t>(((uint64_t)nb << 32) / (uint64_t)no, 0xffffffffull);
    for (int64_t b : {(int64_t)0, (int64_t)nb - 1})      // the last range also takes what rounding leaves over
        if ((b + 1 < nb ? bucket_begin(b + 1, scale, no) : no) - bucket_begin(b, scale, no) > kWidth) return SP_ERR_UNSUPPORTED;
    const bool dbl = lt[0] == SP_COMPRESSED;
    const size_t pw = posBits / 8, cw = crdBits / 8;
    sp_workspace ws(stream);
    const bool counted = (int64_t)nb * kCap > 16 * n + 65536;
    const uint32_t slot = counted ? 0u : (uint32_t)kCap;
    const size_t records = counted ? (size_t)n : (size_t)nb * kCap;
    const size_t cursors = sp_workspace::bytes_for<uint32_t>((size_t)nb + 3);
    ws.reserve(3 * cursors + sp_workspace::bytes_for<Rec>(records) + (dbl ? cursors : 0));
    uint32_t* cursor = ws.get<uint32_t>((size_t)nb + 3);
    Rec* rec = ws.get<Rec>(records);
    uint32_t *first = ws.get<uint32_t>((size_t)nb + 3), *lost = ws.get<uint32_t>((size_t)nb + 3);
    uint32_t* outer_count = dbl ? ws.get<uint32_t>((size_t)nb + 3) : nullptr;
    unsigned long long* host = sp_host_words();
    if (ws.failed || !host) return SP_ERR_ALLOC;
    uint32_t *stop = cursor + nb, *ticket = cursor + nb + 1, *total = cursor + nb + 2;

    // counted while the host prepares the rest
    SP_CUDA(cudaMemsetAsync(cursor, 0, (size_t)(nb + 3) * sizeof(uint32_t), stream));
    if (counted) {
        const unsigned blocks = (unsigned)std::min<int64_t>(kCBlocks, sp_ceil_div(n, kCThreads * 16));
        if (coord_bits == 32) k_rows_count<int32_t><<<blocks, kCThreads, 0, stream>>>(static_cast<const int32_t*>(outer), n, no, scale, nb, cursor, stop, ticket, host);
        else k_rows_count<int64_t><<<blocks, kCThreads, 0, stream>>>(static_cast<const int64_t*>(outer), n, no, scale, nb, cursor, stop, ticket, host);
        SP_LAUNCH_CHECK();
        sp_count_launches(1);
    }

    sp_tensor* t = new sp_tensor();
    auto fail = [&](sp_status s) {              // what is under way may still write to the host's words
        cudaStreamSynchronize(stream);
        sp_free(t);
        return s;
    };
    cudaGetDevice(&t->device);
    t->rank = 2;
    t->posBits = posBits;
    t->crdBits = crdBits;
    for (int l = 0; l < 2; ++l) { t->dims[l] = dims[l]; t->lt[l] = lt[l]; t->ord[l] = ord[l]; }
    // the handle's arrays, one allocation, for `entries` stored entries and `outers` outer indices (a compressed outer
    // level's are at first sized for their bound)
    auto arrays = [&](int64_t entries, int64_t outers) {
        const size_t b_pos0 = dbl ? sp_workspace::padded(2 * pw) : 0, b_crd0 = dbl ? sp_workspace::padded((size_t)outers * cw) : 0;
        const size_t b_pos1 = sp_workspace::padded((size_t)(outers + 1) * pw), b_crd1 = sp_workspace::padded((size_t)entries * cw);
        t->block = sp_dev_alloc(b_pos0 + b_crd0 + b_pos1 + b_crd1 + sp_workspace::padded((size_t)entries * sizeof(double)), stream);
        if (!t->block) return false;
        char* p = static_cast<char*>(t->block);
        if (dbl) { t->pos[0] = p; t->crd[0] = p + b_pos0; t->npos[0] = 2; }
        p += b_pos0 + b_crd0;
        t->pos[1] = p;
        t->crd[1] = p + b_pos1;
        t->val = reinterpret_cast<double*>(p + b_pos1 + b_crd1);
        t->ncrd[1] = t->nval = entries;
        if (ord[0] == 1) {                              // column-major: the column of every entry, for SpMM
            sp_partition sg;
            sg.aux = static_cast<int64_t*>(sp_dev_alloc((size_t)entries * sizeof(uint32_t), stream));
            if (!sg.aux) return false;
            t->parts[(uint64_t)SP_PART_SEGIDS << 56] = sg;
        }
        return true;
    };
    auto columns = [&]() { return ord[0] == 1 ? reinterpret_cast<uint32_t*>(t->parts[(uint64_t)SP_PART_SEGIDS << 56].aux) : nullptr; };
    if (!arrays(n, dbl ? std::min(no, n) : no)) return fail(SP_ERR_ALLOC);
    uint32_t* seg_out = columns();

    const bool small = n < kSmall;
    cudaError_t e = cudaSuccess;
#define SP_ROWS_PARTITION(CT)                                                                                             \
    do {                                                                                                                  \
        const CT *oc = static_cast<const CT*>(outer), *ic = static_cast<const CT*>(inner);                                \
        if (small) {                                                                                                      \
            e = sp_launch_dependent(k_rows_partition<CT, 2>, dim3((unsigned)sp_ceil_div(n, kThreads * 2)), dim3(kThreads), \
                                    (size_t)nb * sizeof(uint32_t), stream, oc, ic, vals, n, no, ni, scale, inner_bits, nb, slot, cursor, rec, stop, host); \
        } else {                                                                                                          \
            e = sp_allow_shared<k_rows_partition_tiles<CT>>(t->device, sizeof(TileShared));                               \
            if (e == cudaSuccess)                                                                                         \
                e = sp_launch_dependent(k_rows_partition_tiles<CT>, dim3((unsigned)sp_ceil_div(n, kTTile)), dim3(kThreads), TileShared::bytes(nb), \
                                        stream, oc, ic, vals, n, no, ni, scale, inner_bits, nb, slot, cursor, rec, stop, host);             \
        }                                                                                                                 \
    } while (0)
    if (coord_bits == 32) SP_ROWS_PARTITION(int32_t);
    else SP_ROWS_PARTITION(int64_t);
#undef SP_ROWS_PARTITION
#define SP_ROWS_LAUNCH(kernel, smem, ...) \
    (e = e != cudaSuccess ? e : sp_launch_dependent(kernel, dim3((unsigned)nb), dim3(kBThreads), smem, stream, __VA_ARGS__))
#define SP_ROWS_BUILD(DBL)                                                                                                \
    do {                                                                                                                  \
        if (e == cudaSuccess) e = sp_allow_shared<k_rows_build<P, I, DBL>>(t->device, sizeof(BuildShared));             \
        SP_ROWS_LAUNCH((k_rows_build<P, I, DBL>), sizeof(BuildShared), rec, (const uint32_t*)cursor, n, no, scale, inner_bits, nb, slot, stop, first, lost, total, host, pos1, \
                       crd1, t->val, seg_out, outer_count);                                        \
    } while (0)
    SP_DISPATCH_WIDTHS(t, {
        P* pos0 = static_cast<P*>(t->pos[0]);
        I* crd0 = static_cast<I*>(t->crd[0]);
        P* pos1 = static_cast<P*>(t->pos[1]);
        I* crd1 = static_cast<I*>(t->crd[1]);
        if (dbl) {
            SP_ROWS_BUILD(true);
            SP_ROWS_LAUNCH((k_rows_outer<P, I>), 0, (const Rec*)rec, (const uint32_t*)cursor, (const uint32_t*)outer_count, (const uint32_t*)nullptr, n, nb, slot, stop, host,
                           pos0, crd0, pos1);
        } else {
            SP_ROWS_BUILD(false);
        }
    });
#undef SP_ROWS_BUILD
#undef SP_ROWS_LAUNCH
    sp_count_launches(dbl ? 3 : 2);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return fail(SP_ERR_CUDA);
    if (host[kErrRange]) return fail(SP_ERR_OUT_OF_RANGE);
    if (host[kErrLong]) return fail(SP_ERR_UNSUPPORTED);
    const int64_t outers = dbl ? (int64_t)host[kOuterCount] : no;
    if (host[kErrDup]) {
        if (flags & SP_DUP_ERROR) return fail(SP_ERR_DUPLICATE);
        if (cudaMemcpyAsync(host + kLost, total, sizeof(uint32_t), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
            cudaStreamSynchronize(stream) != cudaSuccess)
            return fail(SP_ERR_CUDA);
        const int64_t stored = n - (int64_t)(uint32_t)host[kLost];
        const void *pos1_was = t->pos[1], *crd_was = t->crd[1], *block_was = t->block;
        const double* val_was = t->val;
        t->block = nullptr;                             // the first arrays go back with the scratch
        ws.ptrs.push_back(const_cast<void*>(block_was));
        if (seg_out) ws.ptrs.push_back(seg_out);
        t->parts.clear();
        for (int l = 0; l < 2; ++l) t->pos[l] = t->crd[l] = nullptr;
        t->val = nullptr;
        if (!arrays(stored, outers)) return fail(SP_ERR_ALLOC);
        SP_DISPATCH_WIDTHS(t, {
            const P* const pos1_in = static_cast<const P*>(pos1_was);
            const I* const crd_in = static_cast<const I*>(crd_was);
            P* const pos1 = static_cast<P*>(t->pos[1]);
            I* const crd1 = static_cast<I*>(t->crd[1]);
            if (dbl) {
                k_rows_close_up<P, I, true><<<(unsigned)nb, kBThreads, 0, stream>>>(first, lost, n, stored, no, scale, nb, pos1_in, crd_in, val_was,
                                                                                   seg_out, pos1, crd1, t->val, columns());
                k_rows_outer<P, I><<<(unsigned)nb, kBThreads, 0, stream>>>(rec, cursor, outer_count, lost, stored, nb, slot, stop, host,
                                                                           static_cast<P*>(t->pos[0]), static_cast<I*>(t->crd[0]), pos1);
            } else {
                k_rows_close_up<P, I, false><<<(unsigned)nb, kBThreads, 0, stream>>>(first, lost, n, stored, no, scale, nb, pos1_in, crd_in, val_was,
                                                                                    seg_out, pos1, crd1, t->val, columns());
            }
        });
        if (cudaGetLastError() != cudaSuccess) return fail(SP_ERR_CUDA);
        sp_count_launches(dbl ? 2 : 1);
    }
    t->npos[1] = outers + 1;
    if (dbl) t->ncrd[0] = outers;
    *out = t;
    return SP_OK;
}
