// sp_pack for matrices with a compressed inner level and short segments (rows of CSR and DCSR, columns of
// CSC and DCSC): the entries are counted per outer index, scattered to their segment and put in order
// inside it, instead of being sorted by a fused key.
//
//   1. k_rows_count    range check; rank of the entry among those of its outer index seen so far (one atomic)
//   2. k_rows_sums     per tile of outer indices: entries, non-empty indices, sum of squared lengths
//      k_rows_offsets  segment starts; pos[1], and for a compressed outer level crd[0] and the packed pos[1]
//   3. k_rows_scatter  value and both coordinates of every entry as one 16-byte record into its segment
//   4. k_rows_sort     order inside the segments by counting the smaller coordinates; crd[1], values
//
// Every entry is moved twice where the radix sort moves it once per eight key bits, all array sizes are
// known beforehand (the outer level's are bounded), and the one read-back comes at the end.  Step 4 costs the
// sum of the squared segment lengths; a device-side check (k_rows_sums) makes the kernels after it return
// when that or a single segment is too long, and the caller takes the radix path, as it does for
// duplicate coordinates, whose values have to be summed.
//
// Bound: random accesses at L2 (5,000,000 entries by 1,048,576 columns: counting 51 us, scatter 120 us; 100 and
// 42 G accesses/s).  The whole pack of those entries takes 282 us, by radix sort 341 us; of 10,486 entries 63 us
// against 85 us.
#include "common.cuh"

#include <algorithm>

namespace {

constexpr int kThreads = 256;
constexpr int kIpt = 8;                         // entries per thread and tile of k_rows_count / k_rows_scatter
constexpr int kTile = kThreads * kIpt;
constexpr int kRowIpt = 8;                      // outer indices per thread of the two scan kernels
constexpr int kRowTile = kThreads * kRowIpt;
constexpr int kSortTile = 2048;                 // entries whose segments start in a block's share of k_rows_sort
constexpr int kMaxLen = 2048;                   // longest segment taken
constexpr int kSortCap = kSortTile + kMaxLen;
constexpr uint32_t kAbortRank = 4 * kMaxLen;    // a longer segment is not taken, so counting it further is pointless

// What the device reports: word 0 = kErr* bits, 1 = non-empty outer indices, 2 = sum of squared segment lengths.
// kErrIndex: an index derived from the counters fell outside its array (its access was skipped); never for a sound run.
constexpr unsigned long long kErrRange = 1, kErrDup = 2, kErrLong = 4, kErrIndex = 8;

using Rec = uint4;                              // value (low word, high word), inner coordinate, outer coordinate

// Whether the kernels after k_rows_sums go on.
__device__ __forceinline__ bool stopped(const unsigned long long* info, unsigned long long most) {
    return __ldcg(info) != 0 || __ldcg(info + 2) > most;
}

template <typename CT>
__global__ void __launch_bounds__(kThreads)
k_rows_count(const CT* __restrict__ oc, const CT* __restrict__ ic, int64_t n, int64_t no, int64_t ni, uint32_t* __restrict__ count,
             uint32_t* __restrict__ rank, unsigned long long* __restrict__ info) {
    if (__ldcg(info) != 0) return;              // an earlier block met a bad entry or a very long segment
    const int64_t base = (int64_t)blockIdx.x * kTile + threadIdx.x;
    CT o[kIpt], c[kIpt];
    uint32_t r[kIpt];
#pragma unroll
    for (int i = 0; i < kIpt; ++i) {
        const int64_t e = base + i * kThreads;
        o[i] = e < n ? oc[e] : (CT)0;
        c[i] = e < n ? ic[e] : (CT)0;
    }
    bool bad = false, far = false;
#pragma unroll
    for (int i = 0; i < kIpt; ++i) {
        const int64_t e = base + i * kThreads;
        r[i] = 0;
        if (o[i] < 0 || (int64_t)o[i] >= no || c[i] < 0 || (int64_t)c[i] >= ni) bad = true;
        else if (e < n) r[i] = atomicAdd(count + o[i], 1u);
    }
#pragma unroll
    for (int i = 0; i < kIpt; ++i) {
        const int64_t e = base + i * kThreads;
        if (e < n) rank[e] = r[i];
        far |= r[i] >= kAbortRank;
    }
    if (bad) atomicOr(info, kErrRange);
    if (far) atomicOr(info, kErrLong);
}

// Block-wide exclusive scan of two counters at once and their totals.
__device__ __forceinline__ uint2 block_scan2(uint2 v, uint2* s_w, uint2* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint2 incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t ux = __shfl_up_sync(0xffffffffu, incl.x, o), uy = __shfl_up_sync(0xffffffffu, incl.y, o);
        if (lane >= o) { incl.x += ux; incl.y += uy; }
    }
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    uint2 pre = make_uint2(0, 0), tot = make_uint2(0, 0);
#pragma unroll
    for (int i = 0; i < kThreads / 32; ++i) {
        const uint2 s = s_w[i];
        if (i < w) { pre.x += s.x; pre.y += s.y; }
        tot.x += s.x; tot.y += s.y;
    }
    __syncthreads();
    *total = tot;
    return make_uint2(incl.x - v.x + pre.x, incl.y - v.y + pre.y);
}

// A thread's kRowIpt consecutive counters.
__device__ __forceinline__ void load_counts(const uint32_t* count, int64_t no, uint32_t* len) {
    const int64_t q0 = (int64_t)blockIdx.x * kRowTile + (int64_t)threadIdx.x * kRowIpt;
    if (q0 + kRowIpt <= no) {                   // `count` is 256-byte aligned
#pragma unroll
        for (int i = 0; i < kRowIpt; i += 4) {
            const uint4 v = *reinterpret_cast<const uint4*>(count + q0 + i);
            len[i] = v.x; len[i + 1] = v.y; len[i + 2] = v.z; len[i + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < kRowIpt; ++i) len[i] = q0 + i < no ? count[q0 + i] : 0u;
    }
}

__global__ void __launch_bounds__(kThreads)
k_rows_sums(const uint32_t* count, int64_t no, uint2* __restrict__ tile, unsigned long long* __restrict__ info) {
    sp_wait_for_previous_kernel();
    if (__ldcg(info) != 0) return;
    __shared__ uint2 s_w[kThreads / 32];
    __shared__ unsigned long long s_sq[kThreads / 32];
    uint32_t len[kRowIpt];
    load_counts(count, no, len);
    uint2 mine = make_uint2(0, 0), tot;
    unsigned long long sq = 0;
    bool longer = false;
#pragma unroll
    for (int i = 0; i < kRowIpt; ++i) {
        mine.x += len[i];
        mine.y += len[i] != 0;
        sq += (unsigned long long)len[i] * len[i];
        longer |= len[i] > kMaxLen;
    }
    block_scan2(mine, s_w, &tot);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((threadIdx.x & 31) == 0) s_sq[threadIdx.x >> 5] = sq;
    if (__syncthreads_or(longer) && threadIdx.x == 0) atomicOr(info, kErrLong);
    if (threadIdx.x == 0) {
        tile[blockIdx.x] = tot;
        for (int i = 1; i < kThreads / 32; ++i) sq += s_sq[i];
        atomicAdd(info + 2, sq);
    }
}

// start[q] = first entry of outer index q; first[t] = start of the first segment that starts at entry
// t * kSortTile or later (t = 0 .. the number of sort tiles).  DBL: crd0 / pos1 list the non-empty indices.
template <typename P, typename I, bool DBL>
__global__ void __launch_bounds__(kThreads)
k_rows_offsets(const uint32_t* count, int64_t no, const uint2* tile, int64_t n, unsigned long long most,
               uint32_t* __restrict__ start, uint32_t* __restrict__ first, P* __restrict__ pos0, I* __restrict__ crd0,
               P* __restrict__ pos1, int64_t nq, unsigned long long* __restrict__ info) {
    sp_wait_for_previous_kernel();
    if (stopped(info, most)) return;
    const uint32_t stiles = (uint32_t)((n + kSortTile - 1) / kSortTile);
    bool off = false;
    __shared__ uint2 s_w[kThreads / 32];
    uint2 before = make_uint2(0, 0), tot;
    for (int64_t t = threadIdx.x; t < blockIdx.x; t += kThreads) { const uint2 v = tile[t]; before.x += v.x; before.y += v.y; }
    block_scan2(before, s_w, &tot);             // every block adds up the tiles before its own
    before = tot;
    uint32_t len[kRowIpt];
    load_counts(count, no, len);
    uint2 mine = make_uint2(0, 0);
#pragma unroll
    for (int i = 0; i < kRowIpt; ++i) { mine.x += len[i]; mine.y += len[i] != 0; }
    uint2 at = block_scan2(mine, s_w, &tot);
    at.x += before.x;
    at.y += before.y;
    const int64_t q0 = (int64_t)blockIdx.x * kRowTile + (int64_t)threadIdx.x * kRowIpt;
#pragma unroll
    for (int i = 0; i < kRowIpt; ++i) {
        const int64_t q = q0 + i;
        if (q < no) {
            start[q] = at.x;
            if (!DBL) {
                if (sizeof(P) != 4) pos1[q] = (P)at.x;          // 32-bit positions: start is pos1
            } else if (len[i]) {
                if (at.y < nq) {
                    crd0[at.y] = (I)q;
                    pos1[at.y] = (P)at.x;
                } else off = true;
            }
            off |= (int64_t)at.x + len[i] > n;
            for (uint32_t t = at.x / kSortTile + 1; t <= stiles && (int64_t)t * kSortTile <= (int64_t)at.x + len[i]; ++t) first[t] = at.x + len[i];
            at.x += len[i];
            at.y += len[i] != 0;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) first[0] = 0;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kThreads - 1) {
        off |= (int64_t)at.x != n || (DBL && (int64_t)at.y > nq);
        first[stiles] = (uint32_t)n;
        if (!DBL || (int64_t)at.y <= nq) pos1[DBL ? (int64_t)at.y : no] = (P)n;
        if (DBL) { pos0[0] = 0; pos0[1] = (P)at.y; info[1] = at.y; }
    }
    if (off) atomicOr(info, kErrIndex);
}

template <typename CT>
__global__ void __launch_bounds__(kThreads)
k_rows_scatter(const CT* __restrict__ oc, const CT* __restrict__ ic, const double* __restrict__ vals, int64_t n,
               const uint32_t* rank, const uint32_t* start, int64_t no, unsigned long long most,
               unsigned long long* __restrict__ info, Rec* __restrict__ rec) {
    sp_wait_for_previous_kernel();
    if (stopped(info, most)) return;
    const int64_t base = (int64_t)blockIdx.x * kTile + threadIdx.x;
    uint32_t o[kIpt], c[kIpt], r[kIpt];
    double v[kIpt];
#pragma unroll
    for (int i = 0; i < kIpt; ++i) {
        const int64_t e = base + i * kThreads;
        const bool ok = e < n;
        o[i] = ok ? (uint32_t)oc[e] : 0u;
        c[i] = ok ? (uint32_t)ic[e] : 0u;
        r[i] = ok ? rank[e] : 0u;
        v[i] = ok ? vals[e] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < kIpt; ++i) r[i] += o[i] < no ? start[o[i]] : (uint32_t)n;
    bool off = false;
#pragma unroll
    for (int i = 0; i < kIpt; ++i)
        if (base + i * kThreads < n) {
            if (r[i] >= n) { off = true; continue; }
            rec[r[i]] = make_uint4((uint32_t)__double2loint(v[i]), (uint32_t)__double2hiint(v[i]), c[i], o[i]);
        }
    if (off) atomicOr(info, kErrIndex);
}

// A block puts the segments that start among its kSortTile entries in order.  An entry's place is the number
// of smaller coordinates in its segment, counted over shared memory: lanes of one segment read the same word.
template <typename I>
__global__ void __launch_bounds__(kThreads)
k_rows_sort(const Rec* rec, const uint32_t* first, int64_t n, unsigned long long most, unsigned long long* __restrict__ info,
            I* __restrict__ crd, double* __restrict__ val, uint32_t* __restrict__ seg_out) {
    sp_wait_for_previous_kernel();
    if (stopped(info, most)) return;
    __shared__ uint32_t s_c[kSortCap];
    __shared__ uint32_t s_head[kSortCap / 32 + 1];      // one bit per entry: a segment starts here (and one past the end)
    __shared__ int s_prev[kSortCap / 32], s_next[kSortCap / 32 + 1];
    const int64_t e0 = first[blockIdx.x];
    const int64_t span = (int64_t)first[blockIdx.x + 1] - e0;
    const int cnt = (int)(span < kSortCap + 1 ? span : kSortCap + 1);
    if (cnt <= 0) return;
    if (cnt > kSortCap || e0 + cnt > n) {
        if (threadIdx.x == 0) atomicOr(info, kErrIndex);
        return;
    }
    const int t = threadIdx.x, lane = t & 31;
    const int words = (cnt + 31) / 32;
    for (int i = t; i < words * 32; i += kThreads) {
        uint32_t c = 0, o = 0, ob = 0;
        if (i < cnt) {
            const Rec x = rec[e0 + i];
            c = x.z; o = x.w;
            if (lane == 0 && i > 0) ob = rec[e0 + i - 1].w;
        }
        s_c[i] = c;
        const uint32_t up = __shfl_up_sync(0xffffffffu, o, 1);
        const bool head = i < cnt && (i == 0 || o != (lane ? up : ob));
        const uint32_t m = __ballot_sync(0xffffffffu, head);
        if (lane == 0) s_head[i / 32] = m;
    }
    __syncthreads();
    for (int w = t; w < words; w += kThreads) {         // last head before word w, first head from word w on
        int p = w - 1;
        while (p >= 0 && s_head[p] == 0) --p;
        s_prev[w] = p >= 0 ? p * 32 + 31 - __clz(s_head[p]) : 0;
        int q = w;
        while (q < words && s_head[q] == 0) ++q;
        s_next[w] = q < words ? q * 32 + __ffs(s_head[q]) - 1 : cnt;
    }
    if (t == 0) s_next[words] = cnt;
    __syncthreads();
    bool dup = false;
    for (int i = t; i < cnt; i += kThreads) {
        const uint32_t h = s_head[i / 32], below = h & (0xffffffffu >> (31 - lane)), above = lane == 31 ? 0u : h >> (lane + 1);
        const int s = below ? (i & ~31) + 31 - __clz(below) : s_prev[i / 32];
        const int e = above ? i + __ffs(above) : s_next[i / 32 + 1];
        const Rec x = rec[e0 + i];
        const uint32_t c = x.z;
        int less = 0, same = 0;
        for (int j = s; j < e; ++j) {
            const uint32_t cj = s_c[j];
            less += cj < c;
            same += cj == c;
        }
        dup |= same > 1;
        const int64_t p = e0 + s + less;
        crd[p] = (I)c;
        val[p] = __hiloint2double((int)x.y, (int)x.x);
        if (seg_out) seg_out[p] = x.w;
    }
    if (dup) atomicOr(info, kErrDup);
}

}  // namespace

// Returns SP_OK with *out set; an error; or SP_ERR_UNSUPPORTED when the caller should take the radix path.
sp_status sp_pack_rows(const int64_t* dims, const int* ord, const int* lt, int64_t n, const void* outer, const void* inner, int coord_bits,
                       const double* vals, int posBits, int crdBits, cudaStream_t stream, sp_tensor** out) {
    const int64_t no = dims[ord[0]], ni = dims[ord[1]];
    // Counters, starts and one scan over the outer indices are paid whatever they hold, so there may be at
    // most four per entry; records hold 32-bit coordinates; narrow positions need the radix path's width checks.
    if (posBits < 32 || crdBits < 32 || no > 4 * n + 65536 || no >= ((int64_t)1 << 31) || ni >= ((int64_t)1 << 32) || n >= ((int64_t)1 << 31))
        return SP_ERR_UNSUPPORTED;
    // an average this long cannot pass the check below
    const unsigned long long most = 200000000ull + 128ull * (unsigned long long)n;
    if ((double)n * (double)n > (double)most * (double)no) return SP_ERR_UNSUPPORTED;
    const bool dbl = lt[0] == SP_COMPRESSED;
    const int64_t rtiles = sp_ceil_div(no, kRowTile), stiles = sp_ceil_div(n, kSortTile);
    const size_t pw = posBits / 8, cw = crdBits / 8;
    const bool alias = !dbl && posBits == 32;           // pos[1] is the array of segment starts
    sp_workspace ws(stream);
    const size_t counters = sp_workspace::bytes_for<uint32_t>((size_t)no), infob = sp_workspace::bytes_for<unsigned long long>(4);
    ws.reserve(counters + infob + sp_workspace::bytes_for<uint32_t>((size_t)n) + sp_workspace::bytes_for<Rec>((size_t)n) +
               sp_workspace::bytes_for<uint2>((size_t)rtiles) + sp_workspace::bytes_for<uint32_t>((size_t)stiles + 2) +
               (alias ? 0 : sp_workspace::bytes_for<uint32_t>((size_t)no)));
    uint32_t* count = ws.get<uint32_t>((size_t)no);
    unsigned long long* info = ws.get<unsigned long long>(4);
    uint32_t* rank = ws.get<uint32_t>((size_t)n);
    Rec* rec = ws.get<Rec>((size_t)n);
    uint2* tile = ws.get<uint2>((size_t)rtiles);
    uint32_t* first = ws.get<uint32_t>((size_t)stiles + 2);
    uint32_t* start = alias ? nullptr : ws.get<uint32_t>((size_t)no);
    if (ws.failed) return SP_ERR_ALLOC;

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
    if (alias) start = static_cast<uint32_t*>(t->pos[1]);

    cudaError_t e = cudaMemsetAsync(count, 0, counters + infob, stream);
    const dim3 tiles((unsigned)sp_ceil_div(n, kTile)), threads(kThreads);
#define SP_ROWS_LAUNCH(kernel, grid, ...) \
    (e = e != cudaSuccess ? e : sp_launch_dependent(kernel, grid, threads, 0, stream, __VA_ARGS__))
    if (e == cudaSuccess) {                             // the first of the chain: an ordinary launch
        if (coord_bits == 32)
            k_rows_count<int32_t><<<tiles, threads, 0, stream>>>(static_cast<const int32_t*>(outer), static_cast<const int32_t*>(inner), n, no, ni, count, rank, info);
        else
            k_rows_count<int64_t><<<tiles, threads, 0, stream>>>(static_cast<const int64_t*>(outer), static_cast<const int64_t*>(inner), n, no, ni, count, rank, info);
        e = cudaGetLastError();
    }
    SP_ROWS_LAUNCH(k_rows_sums, dim3((unsigned)rtiles), (const uint32_t*)count, no, tile, info);
    SP_DISPATCH_WIDTHS(t, {
        P* pos0 = static_cast<P*>(t->pos[0]);
        I* crd0 = static_cast<I*>(t->crd[0]);
        P* pos1 = static_cast<P*>(t->pos[1]);
        if (dbl) SP_ROWS_LAUNCH((k_rows_offsets<P, I, true>), dim3((unsigned)rtiles), (const uint32_t*)count, no, (const uint2*)tile, n, most, start, first, pos0, crd0, pos1, nq, info);
        else SP_ROWS_LAUNCH((k_rows_offsets<P, I, false>), dim3((unsigned)rtiles), (const uint32_t*)count, no, (const uint2*)tile, n, most, start, first, pos0, crd0, pos1, nq, info);
    });
    if (coord_bits == 32)
        SP_ROWS_LAUNCH(k_rows_scatter<int32_t>, tiles, static_cast<const int32_t*>(outer), static_cast<const int32_t*>(inner), vals, n,
                       (const uint32_t*)rank, (const uint32_t*)start, no, most, info, rec);
    else
        SP_ROWS_LAUNCH(k_rows_scatter<int64_t>, tiles, static_cast<const int64_t*>(outer), static_cast<const int64_t*>(inner), vals, n,
                       (const uint32_t*)rank, (const uint32_t*)start, no, most, info, rec);
    if (crdBits == 32)
        SP_ROWS_LAUNCH(k_rows_sort<uint32_t>, dim3((unsigned)stiles), (const Rec*)rec, (const uint32_t*)first, n, most, info,
                       static_cast<uint32_t*>(t->crd[1]), t->val, seg_out);
    else
        SP_ROWS_LAUNCH(k_rows_sort<uint64_t>, dim3((unsigned)stiles), (const Rec*)rec, (const uint32_t*)first, n, most, info,
                       static_cast<uint64_t*>(t->crd[1]), t->val, seg_out);
#undef SP_ROWS_LAUNCH
    sp_count_launches(5);
    unsigned long long back[3] = {};
    if (e == cudaSuccess) e = cudaMemcpyAsync(back, info, sizeof back, cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return fail(SP_ERR_CUDA);
    if (back[0] & kErrIndex) return fail(SP_ERR_CUDA);
    if (back[0] & kErrRange) return fail(SP_ERR_OUT_OF_RANGE);
    if (back[0] != 0 || back[2] > most) return fail(SP_ERR_UNSUPPORTED);
    t->npos[1] = (dbl ? (int64_t)back[1] : no) + 1;
    if (dbl) t->ncrd[0] = (int64_t)back[1];
    *out = t;
    return SP_OK;
}
