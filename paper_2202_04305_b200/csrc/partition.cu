// Work partitions cached in a handle.
//
// Merge-path partition over the innermost compressed level: the list of segment
// ends pos[1..S] (S segments = rows of a CSR matrix, stored rows of DCSR, columns
// of CSC ...) is merged with the list of entry indices 0..nnz-1; chunk w starts at
// the point of that merge path lying on diagonal w * items.  Every chunk then owns
// the same number of (segment end + entry) items whatever the row-length skew.
#include "common.cuh"

namespace {

template <typename P>
__global__ void k_merge_partition(const P* __restrict__ pos, int64_t nseg, int64_t nnz, int64_t items,
                                  int64_t nchunks, int64_t* __restrict__ row, int64_t* __restrict__ nz) {
    int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (w > nchunks) return;
    const int64_t total = nseg + nnz;
    int64_t d = w * items;
    if (d > total) d = total;
    int64_t lo = d > nnz ? d - nnz : 0;
    int64_t hi = d < nseg ? d : nseg;
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        // segment end `mid` precedes entry (d - mid - 1) when all its entries are consumed
        if ((int64_t)pos[mid + 1] <= d - mid - 1) lo = mid + 1; else hi = mid;
    }
    row[w] = lo;
    nz[w] = d - lo;
}

// MTTKRP: equal ranges of innermost entries; for each range start the fibre
// (level-1 node) and slice (level-0 node or index) that contain it.
template <typename P>
__global__ void k_mttkrp_partition(const P* __restrict__ pos1, int64_t nslice, const P* __restrict__ pos2,
                                   int64_t nfiber, int64_t nnz, int64_t per, int64_t nchunks,
                                   int64_t* __restrict__ fiber, int64_t* __restrict__ nz, int64_t* __restrict__ slice) {
    int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (w > nchunks) return;
    int64_t p = w * per;
    if (p >= nnz) { nz[w] = nnz; fiber[w] = nfiber; slice[w] = nslice; return; }
    int64_t lo = 0, hi = nfiber;            // last f with pos2[f] <= p
    while (hi - lo > 1) { int64_t mid = (lo + hi) >> 1; if ((int64_t)pos2[mid] <= p) lo = mid; else hi = mid; }
    const int64_t f = lo;
    lo = 0; hi = nslice;                    // last s with pos1[s] <= f
    while (hi - lo > 1) { int64_t mid = (lo + hi) >> 1; if ((int64_t)pos1[mid] <= f) lo = mid; else hi = mid; }
    nz[w] = p; fiber[w] = f; slice[w] = lo;
}

// One thread per stored entry: the segment (level-0 node) that holds it, by binary search in pos[1],
// mapped through crd[0] when level 0 is compressed.
template <typename P, typename I>
__global__ void k_segment_ids(const P* __restrict__ pos, int64_t nseg, int64_t nnz, const I* __restrict__ outer,
                              uint32_t* __restrict__ seg) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= nnz) return;
    int64_t lo = 0, hi = nseg;              // last q with pos[q] <= p  (pos[nseg] = nnz > p)
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if ((int64_t)pos[mid] <= p) lo = mid; else hi = mid;
    }
    seg[p] = outer ? (uint32_t)outer[lo] : (uint32_t)lo;
}

// Longest segment: grid-stride maximum of pos[q+1] - pos[q], one atomicMax per block.
template <typename P>
__global__ void k_max_segment(const P* __restrict__ pos, int64_t nseg, unsigned long long* __restrict__ out) {
    unsigned long long m = 0;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nseg; q += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long len = (unsigned long long)pos[q + 1] - (unsigned long long)pos[q];
        m = len > m ? len : m;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long u = __shfl_xor_sync(0xffffffffu, m, o);
        m = u > m ? u : m;
    }
    if ((threadIdx.x & 31) == 0 && m > 0) atomicMax(out, m);
}

// Last i in [0, n) with pos[i] <= v (pos[0] <= v < pos[n]), by a whole warp: 32 probes a round.
template <typename P>
__device__ __forceinline__ int64_t warp_last_le(const P* __restrict__ pos, int64_t n, int64_t v) {
    int64_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const int64_t step = (hi - lo + 31) >> 5, i = lo + ((threadIdx.x & 31) + 1) * step;
        const int le = __popc(__ballot_sync(0xffffffffu, i < hi && (int64_t)pos[i] <= v));
        lo += le * step;
        hi = lo + step < hi ? lo + step : hi;
    }
    return lo;
}

// MTTKRP's word per entry, level-1 coordinate of its fibre << 2 | "the slice ends here" << 1 | "the fibre ends here",
// and the slice that every chunk begins in, with its row.  A block takes a run of tiles of whole chunks: two warps
// look up the fibres and slices at its ends, then each fibre of a tile marks its first entry and an entry's fibre is
// the last mark at or before it, the next tile's fibres being on their way meanwhile.  The look-up is a chain of
// some ten loads: 20 M entries 112 us with a block per tile, 77 with one wave of blocks (for 250 MB read and written).
// The slices of chunks are looked up after the last tile: inside the loop that took 25 us more.
constexpr int kMarkThreads = 256, kMarkTile = 1024, kMarkBlocks = 148 * 6;
template <typename P, typename I>
__global__ void __launch_bounds__(kMarkThreads, 6)
k_mttkrp_marks(const P* __restrict__ pos1, const I* __restrict__ crd0, int64_t nslice, const P* __restrict__ pos2,
               const I* __restrict__ crd1, int64_t nfiber, int64_t nnz, int64_t per, int64_t nchunks, int64_t chunks,
               int64_t* __restrict__ chunk_slice, int64_t* __restrict__ chunk_row, uint32_t* __restrict__ marks, int64_t d0, int64_t d1) {
    // d0, d1: sizes of levels 0 and 1 (used by the bounds-checking debug build only)
    constexpr int kPer = 4;
    static_assert(kMarkTile == kPer * kMarkThreads, "a thread owns four entries");
    __shared__ uint4 s_at4[kMarkTile / 4 + 1];
    __shared__ uint32_t s_crd[kMarkTile];
    __shared__ uint32_t s_w[kMarkThreads / 32];
    __shared__ int64_t s_f[2], s_s[2];
    uint32_t* const s_at = reinterpret_cast<uint32_t*>(s_at4);
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const int64_t c0 = blockIdx.x * chunks, c1 = c0 + chunks < nchunks ? c0 + chunks : nchunks;
    const int64_t e1 = c1 * per < nnz ? c1 * per : nnz;
    const int tile = kMarkTile / (int)per * (int)per;
    int64_t e0 = c0 * per;
    if (w < 2) {
        const int64_t e = w ? e1 : e0;
        const int64_t f = e < nnz ? warp_last_le(pos2, nfiber, e) : nfiber;
        const int64_t q = f < nfiber ? warp_last_le(pos1, nslice, f) : nslice - 1;
        if (lane == 0) { s_f[w] = f; s_s[w] = q; }
    }
    __syncthreads();
    int64_t f0 = s_f[0];
    const int64_t s0 = s_s[0], s1 = s_s[1], fend = s_f[1] + 1 < nfiber ? s_f[1] + 1 : nfiber;
    uint32_t cr[kPer];
    int64_t next[kPer];
    auto load = [&]() {                     // fibres are not empty: kMarkTile of them reach past any tile
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int64_t f = f0 + t + k * kMarkThreads;
            cr[k] = f < fend ? (uint32_t)SP_IDX(crd1[f], d1) : 0u;
            next[k] = f < fend ? (int64_t)pos2[f + 1] : nnz + 1 + kMarkTile;
        }
    };
    load();
    for (; e0 < e1; e0 += tile) {
        const int cnt = (int)(e1 - e0 < tile ? e1 - e0 : tile);
        s_at4[t] = make_uint4(0u, 0u, 0u, 0u);
        if (t == 0) s_at[kMarkTile] = 0u;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            s_crd[t + k * kMarkThreads] = cr[k];
            if (next[k] - e0 <= cnt) s_at[next[k] - e0] = (uint32_t)(t + k * kMarkThreads + 1);
        }
        __syncthreads();
        const uint4 q = s_at4[t];
        const uint32_t here[kPer + 1] = {q.x, q.y, q.z, q.w, s_at[t * kPer + kPer]};
        uint32_t m[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) m[i] = i && here[i] < m[i - 1] ? m[i - 1] : here[i];
        uint32_t run = m[kPer - 1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o && u > run) run = u;
        }
        if (lane == 31) s_w[w] = run;
        uint32_t before = __shfl_up_sync(0xffffffffu, run, 1);
        if (lane == 0) before = 0;
        __syncthreads();
        uint32_t nf = s_at[kMarkTile];      // fibres that end in the tile
#pragma unroll
        for (int i = 0; i < kMarkThreads / 32; ++i) {
            const uint32_t u = s_w[i];
            if (i < w && u > before) before = u;
            if (u > nf) nf = u;
        }
        const int64_t ft = f0;
        f0 += nf;
        if (e0 + tile < e1) load();
        uint32_t word[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const uint32_t fo = m[i] > before ? m[i] : before;
            word[i] = t * kPer + i < cnt ? s_crd[fo] << 2 | (here[i + 1] != 0u ? 1u : 0u) : 0u;
        }
        if (t * kPer + kPer <= cnt)
            reinterpret_cast<uint4*>(marks + e0)[t] = make_uint4(word[0], word[1], word[2], word[3]);
        else
            for (int i = 0; t * kPer + i < cnt; ++i) marks[e0 + t * kPer + i] = word[i];
        if (t * kPer < cnt && t * kPer % (int)per == 0)             // chunks are multiples of four entries
            chunk_slice[e0 / per + t * kPer / (int)per] = ft + (m[0] > before ? m[0] : before);     // the fibre, for now
        __syncthreads();
    }
    for (int64_t c = c0 + t; c < c1; c += kMarkThreads) {
        const int64_t f = chunk_slice[c];
        int64_t lo = s0, hi = s1 + 1;
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) >> 1;
            if ((int64_t)pos1[mid] <= f) lo = mid; else hi = mid;
        }
        chunk_slice[c] = lo;
        chunk_row[c] = SP_IDX(crd0 ? (int64_t)crd0[lo] : lo, d0);
    }
    for (int64_t q = s0 + t; q <= s1; q += kMarkThreads) {          // the last entry of every slice, once the words are written
        const int64_t f = (int64_t)pos1[q + 1];
        if (f > (int64_t)pos1[q] && (int64_t)pos2[f] <= e1) marks[(int64_t)pos2[f] - 1] |= 2u;
    }
}

}  // namespace

// Enqueues the measuring of the longest last-level segment into *host (of sp_host_words), unless it is known or there are none.
static sp_status measure_max_segment(sp_tensor* t, sp_workspace& ws, cudaStream_t stream, unsigned long long** host) {
    *host = nullptr;
    const int last = t->rank - 1;
    const int64_t nseg = t->npos[last] - 1;
    if (t->max_seg >= 0) return SP_OK;
    if (nseg <= 0 || t->ncrd[last] == 0) { t->max_seg = 0; return SP_OK; }
    unsigned long long *d = ws.get<unsigned long long>(1), *h = sp_host_words();
    if (ws.failed || !h) return SP_ERR_ALLOC;
    SP_CUDA(cudaMemsetAsync(d, 0, sizeof *d, stream));
    const unsigned blocks = (unsigned)std::min<int64_t>(sp_ceil_div(nseg, 256), 148 * 8);
    if (t->posBits == 32) k_max_segment<uint32_t><<<blocks, 256, 0, stream>>>(static_cast<const uint32_t*>(t->pos[last]), nseg, d);
    else k_max_segment<uint64_t><<<blocks, 256, 0, stream>>>(static_cast<const uint64_t*>(t->pos[last]), nseg, d);
    SP_LAUNCH_CHECK();
    sp_count_launches(1);
    SP_CUDA(cudaMemcpyAsync(h, d, sizeof *h, cudaMemcpyDeviceToHost, stream));
    *host = h;
    return SP_OK;
}

sp_status sp_get_max_segment(sp_tensor* t, cudaStream_t stream, int64_t* out) {
    std::lock_guard<std::mutex> lock(t->mu);
    sp_workspace ws(stream);
    unsigned long long* h = nullptr;
    const sp_status st = measure_max_segment(t, ws, stream, &h);
    if (st != SP_OK) return st;
    if (h) {
        SP_CUDA(cudaStreamSynchronize(stream));
        t->max_seg = (int64_t)*h;
    }
    *out = t->max_seg;
    return SP_OK;
}

sp_status sp_get_segment_ids(sp_tensor* t, cudaStream_t stream, const uint32_t** out) {
    std::lock_guard<std::mutex> lock(t->mu);
    const uint64_t key = (uint64_t)SP_PART_SEGIDS << 56;
    auto it = t->parts.find(key);
    if (it != t->parts.end()) { *out = reinterpret_cast<const uint32_t*>(it->second.aux); return SP_OK; }
    const int64_t nseg = t->npos[1] - 1, nnz = t->ncrd[1];
    sp_partition p;
    p.aux = static_cast<int64_t*>(sp_dev_alloc((size_t)(nnz ? nnz : 1) * sizeof(uint32_t), stream));
    if (!p.aux) return SP_ERR_ALLOC;
    uint32_t* seg = reinterpret_cast<uint32_t*>(p.aux);
    if (nnz > 0) {
        const unsigned blocks = (unsigned)sp_ceil_div(nnz, 256);
        SP_DISPATCH_WIDTHS(t, {
            k_segment_ids<P, I><<<blocks, 256, 0, stream>>>(static_cast<const P*>(t->pos[1]), nseg, nnz,
                                                           t->lt[0] == SP_COMPRESSED ? static_cast<const I*>(t->crd[0]) : nullptr,
                                                           seg);
        });
        if (cudaGetLastError() != cudaSuccess) { sp_dev_free(p.aux, stream); return SP_ERR_CUDA; }
        sp_count_launches(1);
    }
    if (sp_partition_built(stream) != SP_OK) { sp_dev_free(p.aux, stream); return SP_ERR_CUDA; }
    t->parts[key] = p;
    *out = seg;
    return SP_OK;
}

sp_status sp_get_merge_partition(sp_tensor* t, int64_t items, cudaStream_t stream, sp_partition* out, int64_t* max_seg) {
    std::lock_guard<std::mutex> lock(t->mu);
    const uint64_t key = ((uint64_t)SP_PART_MERGE_LAST << 56) | (uint64_t)items;
    auto it = t->parts.find(key);
    if (it != t->parts.end()) {
        *out = it->second;
        if (!max_seg) return SP_OK;
        *max_seg = t->max_seg;
        if (t->max_seg >= 0) return SP_OK;
        // Not known, and not to be measured in a capture: as if rows were long.
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        SP_CUDA(cudaStreamIsCapturing(stream, &capture));
        if (capture != cudaStreamCaptureStatusNone) { *max_seg = INT64_MAX; return SP_OK; }
    }
    sp_workspace ws(stream);
    unsigned long long* h = nullptr;
    sp_partition p;
    const int last = t->rank - 1;
    const int64_t nseg = t->npos[last] - 1;
    const int64_t nnz = t->ncrd[last];
    const bool missing = it == t->parts.end();
    auto drop = [&](sp_status s) { sp_dev_free(p.row, stream); sp_dev_free(p.nz, stream); return s; };
    if (missing) {
        p.nchunks = sp_ceil_div(nseg + nnz, items);
        if (p.nchunks < 1) p.nchunks = 1;
        p.row = static_cast<int64_t*>(sp_dev_alloc((size_t)(p.nchunks + 1) * sizeof(int64_t), stream));
        p.nz = static_cast<int64_t*>(sp_dev_alloc((size_t)(p.nchunks + 1) * sizeof(int64_t), stream));
        if (!p.row || !p.nz) return drop(SP_ERR_ALLOC);
        const unsigned blocks = (unsigned)sp_ceil_div(p.nchunks + 1, 256);
        if (t->posBits == 32)
            k_merge_partition<uint32_t><<<blocks, 256, 0, stream>>>(static_cast<const uint32_t*>(t->pos[last]), nseg, nnz,
                                                                     items, p.nchunks, p.row, p.nz);
        else
            k_merge_partition<uint64_t><<<blocks, 256, 0, stream>>>(static_cast<const uint64_t*>(t->pos[last]), nseg, nnz,
                                                                     items, p.nchunks, p.row, p.nz);
        if (cudaGetLastError() != cudaSuccess) return drop(SP_ERR_CUDA);
        sp_count_launches(1);
    }
    if (max_seg) {
        const sp_status st = measure_max_segment(t, ws, stream, &h);
        if (st != SP_OK) return drop(st);
    }
    if (sp_partition_built(stream) != SP_OK) return drop(SP_ERR_CUDA);
    if (h) t->max_seg = (int64_t)*h;
    if (max_seg) *max_seg = t->max_seg;
    if (missing) t->parts[key] = *out = p;
    return SP_OK;
}

// ------------------------------------------------------------------ widened shadow ---
namespace {
template <typename S>
__global__ void k_widen(const S* __restrict__ src, uint32_t* __restrict__ dst, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = (uint32_t)src[i];
}

// A 32-bit (or, for bits >= 32, plain) copy of an overhead array.
sp_status widen_array(const void* src, int64_t n, int bits, cudaStream_t stream, void** out) {
    *out = nullptr;
    if (!src) return SP_OK;
    const int obits = bits < 32 ? 32 : bits;
    void* d = sp_dev_alloc((size_t)(n ? n : 1) * (obits / 8), stream);
    if (!d) return SP_ERR_ALLOC;
    *out = d;
    if (n == 0) return SP_OK;
    if (bits >= 32) {
        SP_CUDA(cudaMemcpyAsync(d, src, (size_t)n * (bits / 8), cudaMemcpyDeviceToDevice, stream));
        return SP_OK;
    }
    const unsigned blocks = (unsigned)std::min<int64_t>(sp_ceil_div(n, 256), 148 * 8);
    if (bits == 16) k_widen<uint16_t><<<blocks, 256, 0, stream>>>(static_cast<const uint16_t*>(src), static_cast<uint32_t*>(d), n);
    else k_widen<uint8_t><<<blocks, 256, 0, stream>>>(static_cast<const uint8_t*>(src), static_cast<uint32_t*>(d), n);
    SP_LAUNCH_CHECK();
    sp_count_launches(1);
    return SP_OK;
}
}  // namespace

sp_status sp_widened(sp_tensor* t, cudaStream_t stream, sp_tensor** out) {
    if (t->posBits >= 32 && t->crdBits >= 32) { *out = t; return SP_OK; }
    std::lock_guard<std::mutex> lock(t->mu);
    if (t->wide) {
        *out = t->wide;
        return SP_OK;
    }
    sp_tensor* w = new sp_tensor();
    w->rank = t->rank;
    w->device = t->device;
    w->posBits = t->posBits < 32 ? 32 : t->posBits;
    w->crdBits = t->crdBits < 32 ? 32 : t->crdBits;
    w->val = t->val;
    w->nval = t->nval;
    w->owns_val = false;
    sp_status st = SP_OK;
    for (int l = 0; l < t->rank; ++l) {
        w->dims[l] = t->dims[l]; w->lt[l] = t->lt[l]; w->ord[l] = t->ord[l];
        w->npos[l] = t->npos[l]; w->ncrd[l] = t->ncrd[l];
        if (st == SP_OK) st = widen_array(t->pos[l], t->npos[l], t->posBits, stream, &w->pos[l]);
        if (st == SP_OK) st = widen_array(t->crd[l], t->ncrd[l], t->crdBits, stream, &w->crd[l]);
    }
    if (st != SP_OK) { sp_free(w); return st; }
    if (sp_partition_built(stream) != SP_OK) { sp_free(w); return SP_ERR_CUDA; }
    t->wide = w;
    *out = w;
    return SP_OK;
}

sp_status sp_get_mttkrp_partition(sp_tensor* t, int64_t per, bool with_marks, cudaStream_t stream, sp_partition* out) {
    std::lock_guard<std::mutex> lock(t->mu);
    // the words do not depend on per: a handle has one table of them, and per is the same for all its calls
    const uint64_t key = with_marks ? (uint64_t)SP_PART_MTTKRP_MARKS << 56 : ((uint64_t)SP_PART_MTTKRP << 56) | (uint64_t)per;
    auto it = t->parts.find(key);
    if (it != t->parts.end()) { *out = it->second; return SP_OK; }
    const int64_t nnz = t->ncrd[2];
    const int64_t nfiber = t->ncrd[1];
    const int64_t nslice = t->npos[1] - 1;
    sp_partition p;
    p.nchunks = sp_ceil_div(nnz, per);
    if (p.nchunks < 1) p.nchunks = 1;
    // With marks a chunk's entries are known, per of them from chunk * per on, and row is the row of M it begins in.
    p.row = static_cast<int64_t*>(sp_dev_alloc((size_t)(p.nchunks + 1) * sizeof(int64_t), stream));
    p.aux = static_cast<int64_t*>(sp_dev_alloc((size_t)(p.nchunks + 1) * sizeof(int64_t), stream));
    if (with_marks) p.marks = static_cast<uint32_t*>(sp_dev_alloc((size_t)(nnz ? nnz : 1) * sizeof(uint32_t), stream));
    else p.nz = static_cast<int64_t*>(sp_dev_alloc((size_t)(p.nchunks + 1) * sizeof(int64_t), stream));
    auto drop = [&](sp_status s) { sp_dev_free(p.row, stream); sp_dev_free(p.nz, stream); sp_dev_free(p.aux, stream); sp_dev_free(p.marks, stream); return s; };
    if (!p.row || !p.aux || (with_marks ? !p.marks : !p.nz)) return drop(SP_ERR_ALLOC);
    const unsigned blocks = (unsigned)sp_ceil_div(p.nchunks + 1, 256);
    const int64_t in_tile = kMarkTile / per, run = sp_ceil_div(sp_ceil_div(p.nchunks, in_tile), kMarkBlocks) * in_tile;
    SP_DISPATCH_WIDTHS(t, {
        const P* const pos1 = static_cast<const P*>(t->pos[1]);
        const P* const pos2 = static_cast<const P*>(t->pos[2]);
        if (!with_marks)
            k_mttkrp_partition<P><<<blocks, 256, 0, stream>>>(pos1, nslice, pos2, nfiber, nnz, per, p.nchunks, p.row, p.nz, p.aux);
        else if (nnz > 0)
            k_mttkrp_marks<P, I><<<(unsigned)sp_ceil_div(p.nchunks, run), kMarkThreads, 0, stream>>>(
                pos1, t->lt[0] == SP_COMPRESSED ? static_cast<const I*>(t->crd[0]) : nullptr, nslice, pos2,
                static_cast<const I*>(t->crd[1]), nfiber, nnz, per, p.nchunks, run, p.aux, p.row, p.marks,
                t->dims[t->ord[0]], t->dims[t->ord[1]]);
    });
    if (cudaGetLastError() != cudaSuccess) return drop(SP_ERR_CUDA);
#ifdef SP_DEBUG_BOUNDS
    { const sp_status b = sp_bounds_result(stream); if (b != SP_OK) return drop(b); }
#endif
    sp_count_launches(1);
    if (sp_partition_built(stream) != SP_OK) return drop(SP_ERR_CUDA);
    t->parts[key] = p;
    *out = p;
    return SP_OK;
}
