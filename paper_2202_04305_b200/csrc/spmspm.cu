// sp_spmspm: C[i,j] = sum_k A[i,k] * B[k,j] with A, B and C all stored row-wise as
// (dense, compressed) - the SpMSpM kernel of Section 4.3, measured in Section 6.2 (Table 2).
//
// The paper's loop nest expands each row of C into a dense workspace (values + "filled" flags),
// records which columns were touched, and compresses the row back in index order.  Both paths below
// keep that shape, with the flags as a bitmap whose words, read in order, give the columns sorted.  The
// product runs in two passes: a symbolic one (row lengths -> positions by a scan -> sizes of C's arrays,
// read back once) and a numeric one.  Results of up to 32,768 columns with enough products for their size
// take the bitmap path (k_row_bitmaps, k_symbolic, k_numeric), but for rows of A much longer than the
// others.  Otherwise a block owns a row at a time (k_spmspm): warps walk the entries A[i,k], lanes walk row k of B and add into the block's workspace
// row with atomics, in shared memory when a row of C fits there (dims[1] up to about 25,000), else in
// one workspace row per block in global memory (L2-resident).
#include "common.cuh"

#include <algorithm>

namespace {

constexpr int kPThreads = 256;

__device__ __forceinline__ uint32_t block_excl_scan_u32(uint32_t v, uint32_t* sums, uint32_t* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) sums[w] = incl;
    __syncthreads();
    uint32_t pre = 0, tot = 0;
#pragma unroll
    for (int i = 0; i < kPThreads / 32; ++i) {
        const uint32_t s = sums[i];
        if (i < w) pre += s;
        tot += s;
    }
    __syncthreads();
    *total = tot;
    return incl - v + pre;
}

// NUMERIC = false: rowlen[i] = number of distinct columns of row i.
// NUMERIC = true : crd / val of C filled at cpos[i].. ; the workspace row is left zeroed.
// LONG: only the rows that k_symbolic put in list, *nlong of them.
template <typename P, typename I, bool NUMERIC, bool SMEM, bool LONG>
__global__ void __launch_bounds__(kPThreads)
k_spmspm(const P* __restrict__ apos, const I* __restrict__ acrd, const double* __restrict__ aval,
         const P* __restrict__ bpos, const I* __restrict__ bcrd, const double* __restrict__ bval, int64_t m,
         int64_t n, double* __restrict__ ws_all, uint32_t* __restrict__ bm_all, int64_t* __restrict__ rowlen,
         const void* __restrict__ cpos, int cposBits, void* __restrict__ ccrd, int ccrdBits,
         double* __restrict__ cval, int64_t kdim, const uint32_t* list, const unsigned long long* nlong) {
    sp_wait_for_previous_kernel();
    const int64_t rows = LONG ? (int64_t)*nlong : m;
    if (LONG && blockIdx.x >= rows) return;
    __shared__ uint32_t sums[kPThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t words = (n + 31) >> 5;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    double* ws;          // this block's dense row of C
    uint32_t* bm;        // ... and its "filled" flags, one bit per column
    if (SMEM) {          // [bitmap words, padded to 8 bytes][row of C, numeric pass only]; both start zeroed
        bm = reinterpret_cast<uint32_t*>(s_dyn);
        ws = reinterpret_cast<double*>(s_dyn + ((words * 4 + 7) & ~(int64_t)7));
        for (int64_t x = threadIdx.x; x < words; x += kPThreads) bm[x] = 0u;
        if (NUMERIC)
            for (int64_t x = threadIdx.x; x < n; x += kPThreads) ws[x] = 0.0;
        __syncthreads();
    } else {
        ws = ws_all + (int64_t)blockIdx.x * n;
        bm = bm_all + (int64_t)blockIdx.x * words;
    }

    for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
        const int64_t i = LONG ? (int64_t)list[r] : r;
        // expand: every product of row i lands in the workspace
        const int64_t a0 = (int64_t)apos[i], a1 = (int64_t)apos[i + 1];
        for (int64_t p = a0 + w; p < a1; p += kPThreads / 32) {
            const int64_t k = SP_IDX((int64_t)acrd[p], kdim);
            const double a = aval[p];
            const int64_t b0 = (int64_t)bpos[k], b1 = (int64_t)bpos[k + 1];
            for (int64_t q = b0 + lane; q < b1; q += 32) {
                const int64_t j = SP_IDX((int64_t)bcrd[q], n);
                atomicOr(bm + (j >> 5), 1u << (j & 31));
                if (NUMERIC) atomicAdd(ws + j, a * bval[q]);
            }
        }
        __syncthreads();
        // compress: bitmap words in order give the columns in order
        uint32_t carry = 0;
        const int64_t base = NUMERIC ? (int64_t)sp_load_uint(cpos, i, cposBits) : 0;
        for (int64_t w0 = 0; w0 < words; w0 += kPThreads) {
            const int64_t wi = w0 + threadIdx.x;
            uint32_t bits = wi < words ? bm[wi] : 0u;
            uint32_t tot;
            const uint32_t ex = block_excl_scan_u32((uint32_t)__popc(bits), sums, &tot);
            if (wi < words && bits) bm[wi] = 0u;
            if (NUMERIC && tot >= 8u * kPThreads) {
                // well-filled words: a warp empties its 32 words one after the other, lane = bit, so the
                // workspace row is read (and cleared) 32 adjacent columns at a time and C is written in order
                const uint32_t below = (1u << lane) - 1u;
                for (uint32_t todo = __ballot_sync(0xffffffffu, bits != 0u); todo; todo &= todo - 1u) {
                    const int q = __ffs(todo) - 1;                      // next word of this warp that has columns
                    const uint32_t wbits = __shfl_sync(0xffffffffu, bits, q);
                    const uint32_t woff = __shfl_sync(0xffffffffu, ex, q);
                    if ((wbits >> lane) & 1u) {
                        const int64_t j = ((w0 + (int64_t)(w * 32 + q)) << 5) + lane;
                        const int64_t slot = base + carry + woff + __popc(wbits & below);
                        sp_store_uint(ccrd, slot, (uint64_t)j, ccrdBits);
                        cval[slot] = ws[j];
                        ws[j] = 0.0;
                    }
                }
            } else if (NUMERIC && wi < words && bits) {
                // sparse words: every thread walks the few columns of its own word
                int64_t slot = base + carry + ex;
                while (bits) {
                    const int bpos_ = __ffs(bits) - 1;
                    bits &= bits - 1;
                    const int64_t j = (wi << 5) + bpos_;
                    sp_store_uint(ccrd, slot, (uint64_t)j, ccrdBits);
                    cval[slot] = ws[j];
                    ws[j] = 0.0;
                    ++slot;
                }
            }
            carry += tot;
        }
        if (!NUMERIC && threadIdx.x == 0) rowlen[i] = (int64_t)carry;
        __syncthreads();
    }
}

// Single block: pos[0] = 0, pos[i+1] = rowlen[0] + .. + rowlen[i]; total to *count.
constexpr int kOffThreads = 1024, kOffPer = 8;
__global__ void __launch_bounds__(kOffThreads)
k_row_offsets(const int64_t* rowlen, int64_t m, void* __restrict__ pos, int posBits, int64_t* __restrict__ count) {
    sp_wait_for_previous_kernel();
    __shared__ unsigned long long s_w[kOffThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long run = 0;
    if (threadIdx.x == 0) sp_store_uint(pos, 0, 0, posBits);
    for (int64_t b = 0; b < m; b += kOffThreads * kOffPer) {
        const int64_t i0 = b + (int64_t)threadIdx.x * kOffPer;
        unsigned long long v[kOffPer], mine = 0;
#pragma unroll
        for (int u = 0; u < kOffPer; ++u) {
            v[u] = i0 + u < m ? (unsigned long long)rowlen[i0 + u] : 0ull;
            mine += v[u];
        }
        unsigned long long incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) s_w[w] = incl;
        __syncthreads();
        if (w == 0) {
            unsigned long long x = s_w[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long u = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += u;
            }
            s_w[lane] = x;
        }
        __syncthreads();
        unsigned long long at = run + (w ? s_w[w - 1] : 0ull) + incl - mine;
#pragma unroll
        for (int u = 0; u < kOffPer; ++u) {
            at += v[u];
            if (i0 + u < m) sp_store_uint(pos, i0 + u + 1, at, posBits);
        }
        run += s_w[kOffThreads / 32 - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) *count = (int64_t)run;
}

// ---- results of up to kMaxCols columns whose operand rows are not too sparse --------------------------
// Which columns a row of C holds is the union of the rows of B that it meets: with every row of B as a
// bitmap (k_row_bitmaps) that is an OR of whole words, read 16 bytes a lane (k_symbolic), and the union
// is kept for the numeric pass.  That pass gives a warp a row of C and a block of kColBlk columns, whose
// sums lie in shared memory that no other warp touches: the columns of a row of B are distinct, so the
// lanes of an instruction never meet, and no atomic is needed.
// 8192 x 8192 at density 0.01 (55 M products, 37.5 M results): 463 us for the call, 580 us with one block per row,
// atomics on a shared-memory row and the bitmap built twice (symbolic 112 -> 48 us with the bitmaps, offsets
// 26 -> 10, numeric 434 -> 400).  Bound: the shared-memory pipe, 76 % busy: two accesses of 8 bytes per product.
constexpr int64_t kMaxCols = 32768;
constexpr int kColBlk = 1024;                   // columns of a warp of k_numeric (2048, half the warps: 494 us against 463 below)
constexpr int kBitWarps = 4, kOrWarps = 4, kNumWarps = 4;

// One warp per row of B: its bitmap (stride words, a multiple of four), and split[k * (nblk + 1) + c] =
// the first entry of row k whose column is at least c * kColBlk.
template <typename P, typename I>
__global__ void __launch_bounds__(kBitWarps * 32)
k_row_bitmaps(const P* __restrict__ pos, const I* __restrict__ crd, int64_t rows, int64_t n, int stride, int nblk,
              uint32_t* __restrict__ bits, uint32_t* __restrict__ split, unsigned long long* __restrict__ nlong) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *nlong = 0;        // counted by k_symbolic
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t* mine = reinterpret_cast<uint32_t*>(s_dyn) + (size_t)w * stride;
    const int64_t k = (int64_t)blockIdx.x * kBitWarps + w;
    if (k >= rows) return;
    for (int x = lane; x < stride; x += 32) mine[x] = 0u;
    __syncwarp();
    const int64_t b0 = (int64_t)pos[k], b1 = (int64_t)pos[k + 1];
    uint32_t* sp = split + k * (nblk + 1);
    for (int64_t q = b0 + lane; q < b1; q += 32) {
        const uint32_t j = (uint32_t)SP_IDX(crd[q], n);
        atomicOr(mine + (j >> 5), 1u << (j & 31));
        const int cb = (int)(j / kColBlk);
        for (int c = q > b0 ? (int)((uint32_t)SP_IDX(crd[q - 1], n) / kColBlk) + 1 : 0; c <= cb; ++c) sp[c] = (uint32_t)q;
        if (q == b1 - 1)
            for (int c = cb + 1; c <= nblk; ++c) sp[c] = (uint32_t)b1;
    }
    if (b1 == b0)
        for (int c = lane; c <= nblk; c += 32) sp[c] = (uint32_t)b0;
    __syncwarp();
    for (int x = lane * 4; x < stride; x += 128)
        *reinterpret_cast<uint4*>(bits + k * stride + x) = *reinterpret_cast<const uint4*>(mine + x);
}

// One warp per row of C: the OR of the bitmaps of the rows of B that row i of A names, and its bit count.  Rows of A
// of more than `longest` entries are left to k_spmspm, a block each: one full row of 32,768 entries kept its warp busy
// for 40 ms.
template <typename P, typename I>
__global__ void __launch_bounds__(kOrWarps * 32)
k_symbolic(const P* __restrict__ apos, const I* __restrict__ acrd, const uint32_t* bits, int64_t m, int64_t kdim, int stride,
           int64_t longest, uint32_t* __restrict__ cbits, int64_t* __restrict__ rowlen, uint32_t* __restrict__ list, unsigned long long* nlong) {
    sp_wait_for_previous_kernel();
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * kOrWarps + (threadIdx.x >> 5);
    if (i >= m) return;
    const int64_t a0 = (int64_t)apos[i], a1 = (int64_t)apos[i + 1];
    if (a1 - a0 > longest) {
        if (lane == 0) list[atomicAdd(nlong, 1ull)] = (uint32_t)i;
        return;
    }
    constexpr int kQ = 2, kE = 4;                   // 16-byte runs per lane and entry, entries in flight
    uint32_t total = 0;
    for (int x0 = 0; x0 < stride; x0 += 128 * kQ) {
        uint4 acc[kQ];
#pragma unroll
        for (int t = 0; t < kQ; ++t) acc[t] = make_uint4(0u, 0u, 0u, 0u);
        for (int64_t base = a0; base < a1; base += 32) {
            const int cnt = a1 - base < 32 ? (int)(a1 - base) : 32;
            const uint32_t k_l = lane < cnt ? (uint32_t)SP_IDX(acrd[base + lane], kdim) : 0u;
            for (int e = 0; e < cnt; e += kE) {
                uint4 v[kE][kQ];
#pragma unroll
                for (int u = 0; u < kE; ++u) {
                    const uint32_t k = __shfl_sync(0xffffffffu, k_l, e + u < cnt ? e + u : cnt - 1);   // the tail repeats an entry
                    const uint32_t* row = bits + (int64_t)k * stride + x0 + lane * 4;
#pragma unroll
                    for (int t = 0; t < kQ; ++t)
                        v[u][t] = x0 + t * 128 + lane * 4 < stride ? *reinterpret_cast<const uint4*>(row + t * 128)
                                                                   : make_uint4(0u, 0u, 0u, 0u);
                }
#pragma unroll
                for (int u = 0; u < kE; ++u)
#pragma unroll
                    for (int t = 0; t < kQ; ++t) {
                        acc[t].x |= v[u][t].x; acc[t].y |= v[u][t].y; acc[t].z |= v[u][t].z; acc[t].w |= v[u][t].w;
                    }
            }
        }
#pragma unroll
        for (int t = 0; t < kQ; ++t) {
            if (x0 + t * 128 + lane * 4 < stride)
                *reinterpret_cast<uint4*>(cbits + i * stride + x0 + t * 128 + lane * 4) = acc[t];
            total += (uint32_t)(__popc(acc[t].x) + __popc(acc[t].y) + __popc(acc[t].z) + __popc(acc[t].w));
        }
    }
    total = __reduce_add_sync(0xffffffffu, total);
    if (lane == 0) rowlen[i] = (int64_t)total;
}

// C32: C's coordinates are 32 bits wide (a plain store instead of a width switch).
template <typename P, typename I, bool C32>
__global__ void __launch_bounds__(kNumWarps * 32)
k_numeric(const P* __restrict__ apos, const I* __restrict__ acrd, const double* __restrict__ aval,
          const uint32_t* __restrict__ split, const I* __restrict__ bcrd, const double* __restrict__ bval, int64_t m,
          int nblk, int stride, int64_t longest, const uint32_t* __restrict__ cbits, const void* __restrict__ cpos, int cposBits,
          void* __restrict__ ccrd, int ccrdBits, double* __restrict__ cval, int64_t kdim, int64_t n) {
    // per warp: its columns' sums; the segments of the next 32 entries of A and their factors, read back as
    // broadcasts (a shuffle per word costs the same pipe as a shared-memory access of all of them)
    struct __align__(16) Seg { uint32_t first, len; double a; };
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ Seg s_seg[kNumWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double* acc = reinterpret_cast<double*>(s_dyn) + (size_t)w * kColBlk;
    for (int x = lane; x < kColBlk; x += 32) acc[x] = 0.0;
    __syncwarp();
    const int64_t items = m * nblk;
    const uint32_t below = (1u << lane) - 1u;
    constexpr int kE = 8;                           // segments of B rows fetched together (4: 477 us, 2: 498)
    for (int64_t item = (int64_t)blockIdx.x * kNumWarps + w; item < items; item += (int64_t)gridDim.x * kNumWarps) {
        const int64_t i = item / nblk;
        const int cb = (int)(item - i * nblk);
        const int64_t a0 = (int64_t)apos[i], a1 = (int64_t)apos[i + 1];
        if (a1 - a0 > longest) continue;
        const uint32_t* row = cbits + i * stride;
        const int wb = cb * (kColBlk / 32);
        double* accl = acc - cb * kColBlk;              // indexed by column
        const Seg* seg = s_seg[w];
        for (int64_t base = a0; base < a1; base += 32) {
            const int cnt = a1 - base < 32 ? (int)(a1 - base) : 32;
            Seg mine;
            mine.first = mine.len = 0;                  // past the row's end: empty segments
            mine.a = 0.0;
            if (lane < cnt) {
                const int64_t k = SP_IDX((int64_t)acrd[base + lane], kdim);
                mine.a = aval[base + lane];
                mine.first = split[k * (nblk + 1) + cb];
                mine.len = split[k * (nblk + 1) + cb + 1] - mine.first;
            }
            s_seg[w][lane] = mine;
            const bool any_long = __any_sync(0xffffffffu, mine.len > 32);
            __syncwarp();
            // software pipeline: the next kE segments are requested before these are added
            uint32_t jc[kE], jn[kE];
            double vc[kE], vn[kE];
            auto fetch = [&](int e, uint32_t (&j)[kE], double (&v)[kE]) {
#pragma unroll
                for (int u = 0; u < kE; ++u) {
                    const uint2 sl = *reinterpret_cast<const uint2*>(&seg[e + u]);
                    j[u] = ~0u;
                    if ((uint32_t)lane < sl.y) {
                        j[u] = (uint32_t)SP_IDX(bcrd[sl.x + lane], n);
                        v[u] = bval[sl.x + lane];
                    }
                }
            };
            auto add = [&](int e, const uint32_t (&j)[kE], const double (&v)[kE]) {
#pragma unroll
                for (int u = 0; u < kE; ++u) {
                    if (j[u] != ~0u) accl[j[u]] = fma(seg[e + u].a, v[u], accl[j[u]]);
                    __syncwarp();
                }
                if (any_long)                           // segments of more than 32 entries
                    for (int u = 0; u < kE; ++u) {
                        const Seg g = seg[e + u];
                        for (uint32_t q = 32; q < g.len; q += 32) {
                            if (q + lane < g.len) {
                                const int jj = (int)SP_IDX(bcrd[g.first + q + lane], n);
                                accl[jj] = fma(g.a, bval[g.first + q + lane], accl[jj]);
                            }
                            __syncwarp();
                        }
                    }
            };
            fetch(0, jc, vc);
            for (int e = 0; e < cnt; e += 2 * kE) {
                fetch((e + kE) & 31, jn, vn);           // wraps at 32: a repeated fetch that nobody adds
                add(e, jc, vc);
                if (e + kE >= cnt) break;
                fetch((e + 2 * kE) & 31, jc, vc);
                add(e + kE, jn, vn);
            }
            __syncwarp();                               // s_seg is written again
        }
        // the block's columns in order
        uint32_t before = 0;                            // columns of the row in earlier blocks
        for (int x = lane; x < wb; x += 32) before += (uint32_t)__popc(row[x]);
        before = __reduce_add_sync(0xffffffffu, before);
        int64_t slot = (int64_t)sp_load_uint(cpos, i, cposBits) + before;
#pragma unroll 1
        for (int h = 0; h < kColBlk / 1024; ++h) {
            const int x = wb + h * 32 + lane;
            const uint32_t bits = x < stride ? row[x] : 0u;
            uint32_t at = (uint32_t)__popc(bits), tot = at;     // exclusive prefix over the 32 words
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t u = __shfl_up_sync(0xffffffffu, tot, o);
                if (lane >= o) tot += u;
            }
            at = tot - at;
            tot = __shfl_sync(0xffffffffu, tot, 31);
            double* sums = acc + h * 1024 + lane;
            double* cv = cval + slot;
#pragma unroll 8
            for (int q = 0; q < 32; ++q) {
                const uint32_t wbits = __shfl_sync(0xffffffffu, bits, q), o = __shfl_sync(0xffffffffu, at, q);
                if ((wbits >> lane) & 1u) {
                    const uint32_t to = o + (uint32_t)__popc(wbits & below);
                    const uint32_t col = (uint32_t)(cb * kColBlk + h * 1024 + q * 32 + lane);
                    if (C32) static_cast<uint32_t*>(ccrd)[slot + to] = col;
                    else sp_store_uint(ccrd, slot + to, (uint64_t)col, ccrdBits);
                    cv[to] = sums[q * 32];
                    sums[q * 32] = 0.0;
                }
            }
            slot += tot;
        }
        __syncwarp();
    }
}

}  // namespace

extern "C" sp_status sp_spmspm(const sp_tensor* A, const sp_tensor* B, int posBits, int crdBits, void* stream_,
                               sp_tensor** out) {
    SP_API_RANGE("sp_spmspm");
    if (!out) return SP_ERR_INVALID_ARG;
    *out = nullptr;
    if (!A || !B) return SP_ERR_INVALID_ARG;
    if (posBits == 0) posBits = 64;
    if (crdBits == 0) crdBits = 64;
    if (!sp_valid_width(posBits) || !sp_valid_width(crdBits)) return SP_ERR_INVALID_ARG;
    {   // 8- and 16-bit operands are read through their 32-bit shadows (a cache inside the handle)
        sp_tensor *wa = nullptr, *wb = nullptr;
        sp_status ws_ = sp_widened(const_cast<sp_tensor*>(A), static_cast<cudaStream_t>(stream_), &wa);
        if (ws_ == SP_OK) ws_ = sp_widened(const_cast<sp_tensor*>(B), static_cast<cudaStream_t>(stream_), &wb);
        if (ws_ != SP_OK) return ws_;
        A = wa; B = wb;
    }
    auto is_csr = [](const sp_tensor* t) {
        return t->rank == 2 && t->lt[0] == SP_DENSE && t->lt[1] == SP_COMPRESSED && t->ord[0] == 0 && t->ord[1] == 1;
    };
    if (!is_csr(A) || !is_csr(B)) return SP_ERR_UNSUPPORTED;
    if (A->posBits != B->posBits || A->crdBits != B->crdBits) return SP_ERR_UNSUPPORTED;
    if (A->dims[1] != B->dims[0]) return SP_ERR_INVALID_ARG;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const int64_t m = A->dims[0], n = B->dims[1];
    if (n > 0 && (uint64_t)(n - 1) > sp_width_max(crdBits)) return SP_ERR_WIDTH_OVERFLOW;

    const int64_t words = (n + 31) >> 5;
    // shared-memory workspace if one row of C and its bitmap fit next to a second block's
    int dev = 0, sms = 0, smem_max = 0;
    SP_CUDA(cudaGetDevice(&dev));
    SP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    SP_CUDA(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    const size_t shm_sym = (size_t)((words * 4 + 7) & ~(int64_t)7);
    const size_t shm_num = shm_sym + (size_t)n * sizeof(double);
    // The bitmap path reads a bitmap row per entry of A where the other one walks a row of B, and costs something for
    // every row and block of columns.  It is taken for rows of B of 26 (2048 columns) to 38 entries (8192 and more) on average
    // (uniform operands, 2048 columns, rows of 20, 30: 61.8, 65.3 us, by blocks 62.2, 71.9; 4096, rows of 24, 40: 93.6, 111,
    // by blocks 86.6, 145; 8192, rows of 24, 32, 48: 230, 270, 334, by blocks 154, 223, 395; 16,384, rows of 34, 50: 968, 1209,
    // by blocks 942, 1490) that are also at least a sixteenth of a bitmap row's words, 100 products or more per row and
    // block of columns (8192 columns, 4 x 40 entries a row, 20 products: 149 us, by blocks 100; 30 x 40, 150 products: 324
    // and 317), rows of A that leave work for all warps (100 rows of 2000: 1158 us, by blocks 710) and bitmaps of at
    // most 256 MB.
    const int stride = (int)((words + 3) & ~(int64_t)3);          // words of a bitmap row
    const int64_t kdim = B->dims[0];
    const int nblk = (int)sp_ceil_div(n, kColBlk);
    const double products = (double)A->nval * (double)B->nval / (double)std::max<int64_t>(kdim, 1);
    const bool bitmaps = n <= kMaxCols && m > 0 && m < ((int64_t)1 << 32) && kdim > 0 && B->nval < ((int64_t)1 << 32) &&
                         (m + kdim) * stride * 4 <= ((int64_t)256 << 20) && stride * kdim <= 16 * (B->nval + kdim) &&
                         B->nval >= (22 + std::min(stride, 256) / 16) * kdim && products >= 100.0 * (double)m * nblk && A->nval <= m * std::max<int64_t>(m / 8, 128);
    // rows of A longer than this are not one warp's
    const int64_t longest = bitmaps ? std::max<int64_t>(512, 4 * (A->nval / m)) : 0;
    const bool in_smem = shm_num + 2048 <= (size_t)smem_max;
    auto blocks_for = [&](size_t shm) {
        int64_t per_sm = (int64_t)((size_t)smem_max / (shm + 1024));
        if (per_sm > 8) per_sm = 8;
        if (per_sm < 1) per_sm = 1;
        int64_t b = per_sm * sms;
        if (b > m) b = m;
        return b < 1 ? (int64_t)1 : b;
    };
    int64_t nblocks = m < 148 * 4 ? m : 148 * 4;
    if (nblocks < 1) nblocks = 1;
    sp_workspace ws(stream);
    double* wsrow = nullptr;
    uint32_t* bm = nullptr;
    uint32_t *bbits = nullptr, *cbits = nullptr, *split = nullptr, *list = nullptr;
    if (bitmaps) {
        bbits = ws.get<uint32_t>((size_t)kdim * stride);
        cbits = ws.get<uint32_t>((size_t)m * stride);
        split = ws.get<uint32_t>((size_t)kdim * (nblk + 1));
        list = ws.get<uint32_t>((size_t)(A->nval / (longest + 1)) + 1);
    } else if (!in_smem) {
        wsrow = ws.get<double>((size_t)nblocks * n);
        bm = ws.get<uint32_t>((size_t)nblocks * words);
    }
    int64_t* rowlen = ws.get<int64_t>((size_t)m + 1);
    int64_t* d_count = ws.get<int64_t>(2);                        // entries of C; long rows of A
    unsigned long long* nlong = reinterpret_cast<unsigned long long*>(d_count + 1);
    if (ws.failed) return SP_ERR_ALLOC;
    if (!bitmaps && !in_smem) {
        SP_CUDA(cudaMemsetAsync(wsrow, 0, (size_t)nblocks * n * sizeof(double), stream));
        SP_CUDA(cudaMemsetAsync(bm, 0, (size_t)nblocks * words * sizeof(uint32_t), stream));
    }

    sp_tensor* C = new sp_tensor();
    cudaGetDevice(&C->device);
    C->rank = 2;
    C->dims[0] = m; C->dims[1] = n;
    C->lt[0] = SP_DENSE; C->lt[1] = SP_COMPRESSED;
    C->ord[0] = 0; C->ord[1] = 1;
    C->posBits = posBits; C->crdBits = crdBits;
    C->npos[1] = m + 1;
    C->pos[1] = sp_dev_alloc((size_t)(m + 1) * (posBits / 8), stream);
    if (!C->pos[1]) { sp_free(C); return SP_ERR_ALLOC; }
    auto fail = [&](sp_status s) { sp_free(C); return s; };

#define SP_SPMSPM_ARGS                                                                                            \
    static_cast<const P*>(A->pos[1]), static_cast<const I*>(A->crd[1]), A->val, static_cast<const P*>(B->pos[1]), \
        static_cast<const I*>(B->crd[1]), B->val, m, n, wsrow, bm, rowlen, C->pos[1], posBits, C->crd[1], crdBits, C->val, \
        B->dims[0], list, nlong
#define SP_SPMSPM_LAUNCH(NUM)                                                                                     \
    SP_DISPATCH_WIDTHS(A, {                                                                                       \
        if (in_smem) {                                                                                            \
            const size_t shm = NUM ? shm_num : shm_sym;                                                           \
            if (cudaFuncSetAttribute(k_spmspm<P, I, NUM, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,      \
                                     (int)shm) != cudaSuccess)                                                    \
                return fail(SP_ERR_CUDA);                                                                         \
            k_spmspm<P, I, NUM, true, false><<<(unsigned)blocks_for(shm), kPThreads, shm, stream>>>(SP_SPMSPM_ARGS);     \
        } else {                                                                                                  \
            k_spmspm<P, I, NUM, false, false><<<(unsigned)nblocks, kPThreads, 0, stream>>>(SP_SPMSPM_ARGS);              \
        }                                                                                                         \
    })
    if (bitmaps) {
        SP_DISPATCH_WIDTHS(A, {
            const size_t shm = (size_t)kBitWarps * stride * sizeof(uint32_t);
            k_row_bitmaps<P, I><<<(unsigned)sp_ceil_div(kdim, kBitWarps), kBitWarps * 32, shm, stream>>>(
                static_cast<const P*>(B->pos[1]), static_cast<const I*>(B->crd[1]), kdim, n, stride, nblk, bbits, split, nlong);
            if (sp_launch_dependent(k_symbolic<P, I>, dim3((unsigned)sp_ceil_div(m, kOrWarps)), dim3(kOrWarps * 32), 0, stream,
                                    static_cast<const P*>(A->pos[1]), static_cast<const I*>(A->crd[1]), (const uint32_t*)bbits, m,
                                    kdim, stride, longest, cbits, rowlen, list, nlong) != cudaSuccess)
                return fail(SP_ERR_CUDA);
            if (A->nval > longest &&
                sp_launch_dependent(k_spmspm<P, I, false, true, true>, dim3((unsigned)(2 * sms)), dim3(kPThreads), shm_sym, stream, SP_SPMSPM_ARGS) != cudaSuccess)
                return fail(SP_ERR_CUDA);
        });
        sp_count_launches(A->nval > longest ? 2 : 1);
    } else if (m > 0) {
        SP_SPMSPM_LAUNCH(false);
    }
    if (sp_launch_dependent(k_row_offsets, dim3(1), dim3(kOffThreads), 0, stream, (const int64_t*)rowlen, m, C->pos[1], posBits, d_count) != cudaSuccess)
        return fail(SP_ERR_CUDA);
    if (cudaGetLastError() != cudaSuccess) return fail(SP_ERR_CUDA);
    sp_count_launches(2);
    unsigned long long* h_count = sp_host_words();
    if (!h_count) return fail(SP_ERR_ALLOC);
    if (cudaMemcpyAsync(h_count, d_count, 2 * sizeof *h_count, cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess)
        return fail(SP_ERR_CUDA);
    const int64_t count = (int64_t)h_count[0];
    const int64_t long_rows = bitmaps && A->nval > longest ? (int64_t)h_count[1] : 0;
    if ((uint64_t)count > sp_width_max(posBits)) return fail(SP_ERR_WIDTH_OVERFLOW);
    C->ncrd[1] = count;
    C->nval = count;
    C->crd[1] = sp_dev_alloc((size_t)(count ? count : 1) * (crdBits / 8), stream);
    C->val = static_cast<double*>(sp_dev_alloc((size_t)(count ? count : 1) * sizeof(double), stream));
    if (!C->crd[1] || !C->val) return fail(SP_ERR_ALLOC);
    if (m > 0 && count > 0) {
        if (bitmaps) {
            constexpr size_t shm = (size_t)kNumWarps * kColBlk * sizeof(double);
            const int64_t items = m * nblk;
            const unsigned blocks = (unsigned)std::min<int64_t>(sp_ceil_div(items, kNumWarps), (int64_t)sms * (smem_max / (shm + 1024)));
#define SP_NUMERIC(C32)                                                                                                       \
    do {                                                                                                                      \
        if (sp_allow_shared<k_numeric<P, I, C32>>(dev, shm) != cudaSuccess) return fail(SP_ERR_CUDA);                         \
        k_numeric<P, I, C32><<<blocks, kNumWarps * 32, shm, stream>>>(                                                        \
            static_cast<const P*>(A->pos[1]), static_cast<const I*>(A->crd[1]), A->val, split, static_cast<const I*>(B->crd[1]), B->val, m, \
            nblk, stride, longest, cbits, C->pos[1], posBits, C->crd[1], crdBits, C->val, kdim, n);                                    \
    } while (0)
            SP_DISPATCH_WIDTHS(A, {
                if (crdBits == 32) SP_NUMERIC(true); else SP_NUMERIC(false);
            });
#undef SP_NUMERIC
            if (long_rows > 0) {
                if (cudaGetLastError() != cudaSuccess) return fail(SP_ERR_CUDA);
                const unsigned lblocks = (unsigned)std::min<int64_t>(long_rows, in_smem ? blocks_for(shm_num) : (int64_t)sms);
                if (!in_smem) {
                    wsrow = ws.get<double>((size_t)lblocks * n);
                    bm = ws.get<uint32_t>((size_t)lblocks * words);
                    if (ws.failed) return fail(SP_ERR_ALLOC);
                    if (cudaMemsetAsync(wsrow, 0, (size_t)lblocks * n * sizeof(double), stream) != cudaSuccess ||
                        cudaMemsetAsync(bm, 0, (size_t)lblocks * words * sizeof(uint32_t), stream) != cudaSuccess)
                        return fail(SP_ERR_CUDA);
                }
                SP_DISPATCH_WIDTHS(A, {
                    if (in_smem) {
                        if (cudaFuncSetAttribute(k_spmspm<P, I, true, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm_num) != cudaSuccess)
                            return fail(SP_ERR_CUDA);
                        k_spmspm<P, I, true, true, true><<<lblocks, kPThreads, shm_num, stream>>>(SP_SPMSPM_ARGS);
                    } else {
                        k_spmspm<P, I, true, false, true><<<lblocks, kPThreads, 0, stream>>>(SP_SPMSPM_ARGS);
                    }
                });
                sp_count_launches(1);
            }
        } else {
            SP_SPMSPM_LAUNCH(true);
        }
        if (cudaGetLastError() != cudaSuccess) return fail(SP_ERR_CUDA);
        sp_count_launches(1);
    }
#undef SP_SPMSPM_LAUNCH
#undef SP_SPMSPM_ARGS
#ifdef SP_DEBUG_BOUNDS
    { const sp_status b = sp_bounds_result(stream); if (b != SP_OK) return fail(b); }
#endif
    *out = C;
    return SP_OK;
}
