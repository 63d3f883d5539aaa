// sp_pack for matrices with a compressed inner level and moderate segments (rows of CSR and DCSR, columns of
// CSC and DCSC): no sort by key, the entries pass through memory twice.
//
//   1. k_rows_partition  (k_rows_partition_tiles from 300,000 entries on) range check; entries into buckets, one per range of outer indices, in any order
//   2. k_rows_build      a block per bucket: entries per outer index, order inside every segment, and
//                        everything the bucket contributes to the storage, written in order
//   3. k_rows_outer      (compressed outer level) the buckets' lists of stored outer indices, joined
//
// Buckets hold about kAverage entries and at most kCap.  Random accesses are what a GPU is slow at (about 140 G
// single-lane accesses/s here, hit or miss): this way an entry costs at most one, its 16-byte store in step 1; every
// other scattered access stays in shared memory.  Sizes are known beforehand (a compressed outer level's are
// bounded), so the one read-back comes at the end.  A bucket that overflows (long or very uneven segments)
// and duplicate coordinates, whose values have to be summed, are found on the device; the kernels after that
// return and the caller takes the radix path.
#include "common.cuh"

#include <algorithm>

namespace {

constexpr int kThreads = 512;                   // of k_rows_partition
constexpr int kBThreads = 512;                  // of k_rows_build and k_rows_outer
constexpr int kWarps = kBThreads / 32;
// Entries a bucket can hold.  4096 is faster where no bucket overflows (5 M uniform entries 188 us against 196, 6144 204),
// but power-law rows (mean 16, deviation 54) overflow it and then pay for both paths: 3.2 M of them 279 us against 150,
// a conversion of 2 M 190 against 123.  5120 is five deviations from their mean.
constexpr int kCap = 5120;
constexpr int kIpt = kCap / kBThreads;          // ... per thread of k_rows_build
constexpr int kAverage = 2048;                  // entries per bucket aimed at
constexpr int kAverageSmall = 256;               // ... of a small input, for more blocks (10,486 entries: 37 us; 2048: 39)
constexpr int kWidth = 2048;                    // outer indices of a bucket
constexpr int kMaxBuckets = 4096;
constexpr int kDense = 24;                      // mean compares per entry above which segments are cut into bins

// What the device reports, straight into the caller's pinned words: one word per event, then the number of
// non-empty outer indices.  `stop` is the device's own copy: later blocks and kernels return once it is set.
enum { kErrRange = 0, kErrDup, kErrLong, kOuterCount };
__device__ __forceinline__ void report(int what, uint32_t* stop, unsigned long long* host) {
    *static_cast<volatile unsigned long long*>(host + what) = 1;
    *static_cast<volatile uint32_t*>(stop) = 1;
}

using Rec = uint4;                              // value (low, high word), inner coordinate, outer coordinate

// Outer index o lies in bucket o * scale / 2^32; bucket b begins at the first o that the formula gives b for.
__host__ __device__ __forceinline__ int64_t bucket_begin(int64_t b, uint32_t scale, int64_t no) {
    const int64_t o = (int64_t)((((uint64_t)b << 32) + scale - 1) / scale);
    return o < no ? o : no;
}

// Whether some block has reported an error, the same answer for all threads of a block.
__device__ __forceinline__ bool stopped(const uint32_t* stop) {
    return __syncthreads_or(threadIdx.x == 0 && __ldcg(stop) != 0) != 0;
}

// Exclusive scan over the block of one counter per thread.
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
    for (int i = 0; i < kWarps; ++i) {
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

// A block sends a tile of kThreads * PER entries to their buckets: ranks inside the tile by shared-memory
// atomics, the tile's place in every bucket by one atomic on the bucket's cursor.
template <typename CT, int PER>
__global__ void __launch_bounds__(kThreads, 2)
k_rows_partition(const CT* __restrict__ oc, const CT* __restrict__ ic, const double* __restrict__ vals, int64_t n, int64_t no, int64_t ni,
                 uint32_t scale, int nb, uint32_t* __restrict__ cursor, Rec* __restrict__ rec, uint32_t* stop, unsigned long long* host) {
    extern __shared__ uint32_t s_hist[];
    if (stopped(stop)) return;
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
    if (__syncthreads_or(bad)) {
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
            full |= at[q] + k[q] > (uint32_t)kCap;
            s_hist[t + q * kThreads] = at[q];
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
            rec[(size_t)b * kCap + s_hist[b] + r[i]] =
                make_uint4((uint32_t)__double2loint(v), (uint32_t)__double2hiint(v), (uint32_t)c[i], (uint32_t)o[i]);
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
    uint32_t count[kMaxBuckets];                // entries of the tile, then where they begin in rec
    uint32_t shift[kMaxBuckets];                // place in the bucket minus place in rec
    uint32_t w[kThreads / 32];
};

template <typename CT>
__global__ void __launch_bounds__(kThreads, 2)
k_rows_partition_tiles(const CT* __restrict__ oc, const CT* __restrict__ ic, const double* __restrict__ vals, int64_t n, int64_t no, int64_t ni,
                       uint32_t scale, int nb, uint32_t* __restrict__ cursor, Rec* __restrict__ rec, uint32_t* stop, unsigned long long* host) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    TileShared& s = *reinterpret_cast<TileShared*>(s_raw);
    if (stopped(stop)) return;
    const int t = threadIdx.x;
    for (int b = t; b < nb; b += kThreads) s.count[b] = 0u;
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
        r[i] = i * kThreads + t < cnt ? atomicAdd(&s.count[__umulhi(o[i], scale)], 1u) : 0u;
    }
    if (__syncthreads_or(bad)) {
        if (t == 0) report(kErrRange, stop, host);
        return;
    }
    // all cursors of a thread at once: one wait, not one per bucket
    constexpr int kPerB = (kMaxBuckets + kThreads - 1) / kThreads;
    uint32_t k[kPerB], at[kPerB], mine = 0;
#pragma unroll
    for (int q = 0; q < kPerB; ++q) {
        const int b = t + q * kThreads;
        k[q] = b < nb ? s.count[b] : 0u;
        at[q] = k[q] ? atomicAdd(cursor + b, k[q]) : 0u;
        mine += k[q];
    }
    const int lane = t & 31, w = t >> 5;
    uint32_t incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += u;
    }
    if (lane == 31) s.w[w] = incl;
    __syncthreads();
    uint32_t from = incl - mine;
#pragma unroll
    for (int i = 0; i < kThreads / 32; ++i) from += i < w ? s.w[i] : 0u;
    bool full = false;
#pragma unroll
    for (int q = 0; q < kPerB; ++q)
        if (k[q]) {
            const int b = t + q * kThreads;
            full |= at[q] + k[q] > (uint32_t)kCap;
            s.count[b] = from;
            s.shift[b] = at[q] - from;
            from += k[q];
        }
    if (__syncthreads_or(full)) {
        if (t == 0) report(kErrLong, stop, host);
        return;
    }
#pragma unroll
    for (int i = 0; i < kTIpt; ++i)
        if (i * kThreads + t < cnt)
            s.rec[s.count[__umulhi(o[i], scale)] + r[i]] =
                make_uint4((uint32_t)__double2loint(v[i]), (uint32_t)__double2hiint(v[i]), c[i], o[i]);
    __syncthreads();
#pragma unroll 4
    for (int j = t; j < cnt; j += kThreads) {
        const Rec x = s.rec[j];
        const uint32_t b = __umulhi(x.w, scale);
        rec[(size_t)b * kCap + (s.shift[b] + (uint32_t)j)] = x;
    }
}

struct BuildShared {
    uint32_t count[(kCap / 2 > kWidth ? kCap / 2 : kWidth) + 1];    // entries, then starts, of the bucket's outer indices; later the entries' outer offsets
    uint32_t crd[kCap];
    union {
        double val[kCap];
        struct { uint32_t lo[kWidth], hi[kWidth]; };        // smallest and largest coordinate of a segment
        struct { double unused[kCap / 2]; uint32_t bin[kCap]; };
    };
    uint32_t bin_end;                           // bin[kCap] when the bucket is full
    uint32_t w[kWarps];
};
static_assert(sizeof(uint32_t) * 2 * kWidth <= sizeof(double) * kCap / 2, "lo and hi lie before bin");
static_assert(sizeof(BuildShared::count) >= sizeof(uint16_t) * kCap, "the starts' space holds a 16-bit number per entry");

// The place of an entry is the start of its segment plus the number of smaller coordinates in it, counted over
// shared memory.  Where segments are long (more than kDense compares per entry on average) they are first
// cut into as many bins as they have entries, evenly between their smallest and largest coordinate, and only
// the entries of one bin are compared.
template <typename P, typename I, bool DBL>
__global__ void __launch_bounds__(kBThreads, 2)
k_rows_build(const Rec* rec, const uint32_t* cursor, int64_t n, int64_t no, uint32_t scale, int nb, uint32_t* stop, unsigned long long* host,
             P* __restrict__ pos1, I* __restrict__ crd, double* __restrict__ val, uint32_t* __restrict__ seg_out,
             uint32_t* __restrict__ outer_list, uint32_t* __restrict__ outer_pos, uint32_t* __restrict__ outer_count) {
    sp_wait_for_previous_kernel();
    if (stopped(stop)) return;
    extern __shared__ __align__(16) unsigned char s_raw[];
    BuildShared& s = *reinterpret_cast<BuildShared*>(s_raw);
    const int t = threadIdx.x, b = blockIdx.x;
    const int cnt = (int)cursor[b];
    const int64_t lo = bucket_begin(b, scale, no), hi = b + 1 < nb ? bucket_begin(b + 1, scale, no) : no;
    const int width = (int)(hi - lo);
    // entries of this thread, requested first; the values are fetched again at the end (registers)
    const Rec* mine = rec + (size_t)b * kCap + t;
    uint32_t c[kIpt], qr[kIpt];                 // inner coordinate; outer offset << 16 | rank, later the place
#pragma unroll
    for (int i = 0; i < kIpt; ++i) {
        c[i] = qr[i] = 0u;
        if (i * kBThreads + t < cnt) { const Rec x = mine[i * kBThreads]; c[i] = x.z; qr[i] = x.w - (uint32_t)lo; }
    }
    uint32_t before = 0, base;
    for (int q = t; q < b; q += kBThreads) before += cursor[q];
    for (int q = t; q < width; q += kBThreads) { s.count[q] = 0u; s.lo[q] = ~0u; s.hi[q] = 0u; }
    block_scan(before, s.w, &base);             // (also the barrier after the zeroing)
#pragma unroll
    for (int i = 0; i < kIpt; ++i)
        if (i * kBThreads + t < cnt) qr[i] = qr[i] << 16 | atomicAdd(&s.count[qr[i]], 1u);
    __syncthreads();
    // mean number of compares without bins; outer level
    uint32_t sq = 0, filled = 0, tot_sq, tot_filled;
    constexpr int kPerW = kWidth / kBThreads;
#pragma unroll
    for (int i = 0; i < kPerW; ++i) {
        const int q = t * kPerW + i;
        const uint32_t k = q < width ? s.count[q] : 0u;
        sq += k * k;                            // at most kCap^2 in all
        filled += k != 0;
    }
    const uint32_t at_filled = block_scan(filled, s.w, &tot_filled);
    block_scan(sq, s.w, &tot_sq);
    const bool bins = tot_sq > (uint32_t)kDense * (uint32_t)cnt;
    if (DBL) {
        uint32_t k = 0;                         // the stored indices of this thread's kPerW, in order
#pragma unroll
        for (int i = 0; i < kPerW; ++i) {
            const int q = t * kPerW + i;
            if (q < width && s.count[q]) { outer_list[lo + at_filled + k] = (uint32_t)(lo + q); ++k; }
        }
        if (t == 0) outer_count[b] = tot_filled;
        __syncthreads();
        uint32_t len[kPerW];
#pragma unroll
        for (int i = 0; i < kPerW; ++i) { const int q = t * kPerW + i; len[i] = q < width ? s.count[q] : 0u; }
        scan_shared<kPerW>(s.count, width, s.w);
        k = 0;
#pragma unroll
        for (int i = 0; i < kPerW; ++i)
            if (len[i]) { outer_pos[lo + at_filled + k] = base + s.count[t * kPerW + i]; ++k; }
    } else {
        scan_shared<kPerW>(s.count, width, s.w);
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
    uint32_t tot_sum;
    block_scan(sum, s.w, &tot_sum);             // also the barrier after which coordinates, starts and bins are dead
    if (tot_sum != (uint32_t)(cnt * (cnt - 1) / 2)) {
        if (t == 0) report(kErrDup, stop, host);
        return;
    }
    uint16_t* s_seg = reinterpret_cast<uint16_t*>(s.count);
#pragma unroll
    for (int i = 0; i < kIpt; ++i)
        if (i * kBThreads + t < cnt) {
            const uint2 v = *reinterpret_cast<const uint2*>(mine + i * kBThreads);
            const uint32_t p = to[i] & 0xffffu;
            s.crd[p] = c[i];
            s.val[p] = __hiloint2double((int)v.y, (int)v.x);
            if (seg_out) s_seg[p] = (uint16_t)(to[i] >> 16);
        }
    __syncthreads();
    for (int j = t; j < cnt; j += kBThreads) {
        crd[base + j] = (I)s.crd[j];
        val[base + j] = s.val[j];
        if (seg_out) seg_out[base + j] = (uint32_t)lo + s_seg[j];
    }
}

// Joins the buckets' lists of non-empty outer indices and of their first entries: crd[0] and pos[1].
template <typename P, typename I>
__global__ void __launch_bounds__(kBThreads)
k_rows_outer(const uint32_t* outer_list, const uint32_t* outer_pos, const uint32_t* outer_count, int64_t n, int64_t no, uint32_t scale, int nb,
             uint32_t* stop, unsigned long long* host, P* __restrict__ pos0, I* __restrict__ crd0, P* __restrict__ pos1) {
    sp_wait_for_previous_kernel();
    if (stopped(stop)) return;
    __shared__ uint32_t s_w[kWarps];
    const int t = threadIdx.x, b = blockIdx.x;
    uint32_t before = 0, base;
    for (int q = t; q < b; q += kBThreads) before += outer_count[q];
    block_scan(before, s_w, &base);
    const int64_t lo = bucket_begin(b, scale, no);
    const uint32_t cnt = outer_count[b];
    for (uint32_t q = t; q < cnt; q += kBThreads) {
        crd0[base + q] = (I)outer_list[lo + q];
        pos1[base + q] = (P)outer_pos[lo + q];
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
                       const double* vals, int posBits, int crdBits, cudaStream_t stream, sp_tensor** out) {
    const int64_t no = dims[ord[0]], ni = dims[ord[1]];
    // narrow positions need the radix path's width checks; records hold 32-bit coordinates
    if (posBits < 32 || crdBits < 32 || no >= ((int64_t)1 << 31) || ni >= ((int64_t)1 << 32)) return SP_ERR_UNSUPPORTED;
    // enough buckets for the entries and for the outer indices, no more than there are outer indices
    int64_t buckets = std::max(sp_ceil_div(n, n < 300000 ? kAverageSmall : kAverage), sp_ceil_div(no, kWidth - 48));
    if (buckets > kMaxBuckets) return SP_ERR_UNSUPPORTED;
    if (buckets > no) {
        if (n > no * kCap) return SP_ERR_UNSUPPORTED;
        buckets = no;
    }
    const int nb = (int)buckets;
    const uint32_t scale = (uint32_t)std::min<uint64_t>(((uint64_t)nb << 32) / (uint64_t)no, 0xffffffffull);
    for (int64_t b : {(int64_t)0, (int64_t)nb - 1})      // the last range also takes what rounding leaves over
        if ((b + 1 < nb ? bucket_begin(b + 1, scale, no) : no) - bucket_begin(b, scale, no) > kWidth) return SP_ERR_UNSUPPORTED;
    const bool dbl = lt[0] == SP_COMPRESSED;
    const size_t pw = posBits / 8, cw = crdBits / 8;
    sp_workspace ws(stream);
    const size_t cursors = sp_workspace::bytes_for<uint32_t>((size_t)nb + 1);
    ws.reserve(cursors + sp_workspace::bytes_for<Rec>((size_t)nb * kCap) +
               (dbl ? 2 * sp_workspace::bytes_for<uint32_t>((size_t)no) + cursors : 0));
    uint32_t* cursor = ws.get<uint32_t>((size_t)nb + 1);
    Rec* rec = ws.get<Rec>((size_t)nb * kCap);
    uint32_t* outer_list = dbl ? ws.get<uint32_t>((size_t)no) : nullptr;
    uint32_t* outer_pos = dbl ? ws.get<uint32_t>((size_t)no) : nullptr;
    uint32_t* outer_count = dbl ? ws.get<uint32_t>((size_t)nb + 1) : nullptr;
    unsigned long long* host = sp_host_words();
    if (ws.failed || !host) return SP_ERR_ALLOC;
    uint32_t* stop = cursor + nb;

    sp_tensor* t = new sp_tensor();
    auto fail = [&](sp_status s) { sp_free(t); return s; };
    cudaGetDevice(&t->device);
    t->rank = 2;
    t->posBits = posBits;
    t->crdBits = crdBits;
    for (int l = 0; l < 2; ++l) { t->dims[l] = dims[l]; t->lt[l] = lt[l]; t->ord[l] = ord[l]; }
    // one allocation for the handle's arrays; a compressed outer level's are sized for its bound
    const int64_t nq = dbl ? std::min(no, n) : no;
    const size_t b_pos0 = dbl ? sp_workspace::padded(2 * pw) : 0, b_crd0 = dbl ? sp_workspace::padded((size_t)nq * cw) : 0;
    const size_t b_pos1 = sp_workspace::padded((size_t)(nq + 1) * pw), b_crd1 = sp_workspace::padded((size_t)n * cw);
    t->block = sp_dev_alloc(b_pos0 + b_crd0 + b_pos1 + b_crd1 + sp_workspace::padded((size_t)n * sizeof(double)), stream);
    if (!t->block) return fail(SP_ERR_ALLOC);
    char* p = static_cast<char*>(t->block);
    if (dbl) { t->pos[0] = p; t->crd[0] = p + b_pos0; t->npos[0] = 2; }
    p += b_pos0 + b_crd0;
    t->pos[1] = p;
    t->crd[1] = p + b_pos1;
    t->val = reinterpret_cast<double*>(p + b_pos1 + b_crd1);
    t->ncrd[1] = t->nval = n;
    uint32_t* seg_out = nullptr;
    if (ord[0] == 1) {                                  // column-major: the column of every entry, for SpMM
        sp_partition sg;
        sg.aux = static_cast<int64_t*>(sp_dev_alloc((size_t)n * sizeof(uint32_t), stream));
        if (!sg.aux) return fail(SP_ERR_ALLOC);
        seg_out = reinterpret_cast<uint32_t*>(sg.aux);
        t->parts[(uint64_t)SP_PART_SEGIDS << 56] = sg;
    }

    cudaError_t e = cudaMemsetAsync(cursor, 0, (size_t)(nb + 1) * sizeof(uint32_t), stream);
    if (e == cudaSuccess) {
#define SP_ROWS_PARTITION(CT, PER)                                                                                        \
    k_rows_partition<CT, PER><<<(unsigned)sp_ceil_div(n, kThreads * PER), kThreads, (size_t)nb * sizeof(uint32_t), stream>>>( \
        static_cast<const CT*>(outer), static_cast<const CT*>(inner), vals, n, no, ni, scale, nb, cursor, rec, stop, host)
        // small inputs need the blocks (and have few entries per tile and bucket): 10,486 entries 36.9 us, 38.6 in tiles
        const bool small = n < 300000;
#define SP_ROWS_TILES(CT)                                                                                                 \
    do {                                                                                                                  \
        e = sp_allow_shared<k_rows_partition_tiles<CT>>(t->device, sizeof(TileShared));                                 \
        if (e == cudaSuccess)                                                                                             \
            k_rows_partition_tiles<CT><<<(unsigned)sp_ceil_div(n, kTTile), kThreads, sizeof(TileShared), stream>>>(      \
                static_cast<const CT*>(outer), static_cast<const CT*>(inner), vals, n, no, ni, scale, nb, cursor, rec, stop, host); \
    } while (0)
        if (coord_bits == 32) { if (small) SP_ROWS_PARTITION(int32_t, 2); else SP_ROWS_TILES(int32_t); }
        else { if (small) SP_ROWS_PARTITION(int64_t, 2); else SP_ROWS_TILES(int64_t); }
#undef SP_ROWS_TILES
#undef SP_ROWS_PARTITION
        if (e == cudaSuccess) e = cudaGetLastError();
    }
#define SP_ROWS_LAUNCH(kernel, smem, ...) \
    (e = e != cudaSuccess ? e : sp_launch_dependent(kernel, dim3((unsigned)nb), dim3(kBThreads), smem, stream, __VA_ARGS__))
#define SP_ROWS_BUILD(DBL)                                                                                                \
    do {                                                                                                                  \
        if (e == cudaSuccess) e = sp_allow_shared<k_rows_build<P, I, DBL>>(t->device, sizeof(BuildShared));             \
        SP_ROWS_LAUNCH((k_rows_build<P, I, DBL>), sizeof(BuildShared), (const Rec*)rec, (const uint32_t*)cursor, n, no, scale, nb, stop, host, pos1, \
                       crd1, t->val, seg_out, outer_list, outer_pos, outer_count);                                        \
    } while (0)
    SP_DISPATCH_WIDTHS(t, {
        P* pos0 = static_cast<P*>(t->pos[0]);
        I* crd0 = static_cast<I*>(t->crd[0]);
        P* pos1 = static_cast<P*>(t->pos[1]);
        I* crd1 = static_cast<I*>(t->crd[1]);
        if (dbl) {
            SP_ROWS_BUILD(true);
            SP_ROWS_LAUNCH((k_rows_outer<P, I>), 0, (const uint32_t*)outer_list, (const uint32_t*)outer_pos, (const uint32_t*)outer_count, n, no,
                           scale, nb, stop, host, pos0, crd0, pos1);
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
    if (host[kErrDup] || host[kErrLong]) return fail(SP_ERR_UNSUPPORTED);
    t->npos[1] = (dbl ? (int64_t)host[kOuterCount] : no) + 1;
    if (dbl) t->ncrd[0] = (int64_t)host[kOuterCount];
    *out = t;
    return SP_OK;
}
