// sp_mttkrp: M[i,r] = sum_{j,k} T[i,j,k] * B[j,r] * C[k,r]  (Section 6.3).
//
// T is stored (compressed|dense, compressed, compressed) with logical dimension 0
// at level 0.  The derived loop nest walks slices (level 0), fibres (level 1) and
// entries (level 2); the entry loop accumulates val * F2[c2, r] per fibre, the
// fibre's sum is scaled by F1[c1, r] into the slice, and the slice's sum is row i
// of M.  F1 / F2 are B / C, or C / B when the two inner dimensions are stored
// interchanged (the paper's alternative ordering).
//
// The innermost entries are cut into equal ranges, one per group of lanes (per warp, lane = column, in the generic
// kernel).  Slices that start and end inside a range are stored directly; the open slice at
// either end of a range is added into M (zeroed first) with one atomic add per
// column - no atomics in the entry or fibre loops.
#include "common.cuh"

#include <limits.h>

#include <algorithm>

namespace {

constexpr int kTThreads = 256;

// One nnz batch = up to 32 consecutive entries held one per lane (coordinate, value).
// The ends of the fibres that fall inside the batch are turned into a 32-bit mask, so the
// per-entry loop is fully unrolled with static lane indices: all factor-row loads of a group
// of kGroup entries (and the level-1 factor row of every fibre that ends in the group) are
// issued before the first multiply-add that needs them.
constexpr int kGroup = 8;

template <typename P, typename I>
__global__ void __launch_bounds__(kTThreads)
k_mttkrp(const P* __restrict__ pos1, const I* __restrict__ crd0, const P* __restrict__ pos2,
         const I* __restrict__ crd1, const I* __restrict__ crd2, const double* __restrict__ val,
         const double* __restrict__ F1, const double* __restrict__ F2, int64_t R, double* __restrict__ M,
         const int64_t* __restrict__ pfiber, const int64_t* __restrict__ pnz, const int64_t* __restrict__ pslice,
         int64_t nchunks, int64_t nslice, int64_t nfiber, int64_t d0, int64_t d1, int64_t d2) {
    // d0, d1, d2: rows of M, F1, F2 (used by the bounds-checking debug build only)
    // open-slice sums of the block's warps: slot 2*warp = the slice the warp's range starts in,
    // slot 2*warp+1 = the slice it ends in (when different); equal neighbours are added here so
    // that a slice spanning the whole block costs one atomic add per column, not one per warp
    __shared__ double s_car[2 * kTThreads / 32][32];
    __shared__ long long s_id[2 * kTThreads / 32];
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const bool live = w < nchunks;
    const int64_t p0 = live ? pnz[w] : 0, p1 = live ? pnz[w + 1] : 0;
    constexpr int64_t kInf = INT64_MAX;

    for (int64_t rb = 0; rb < R; rb += 32) {
        const bool on = rb + lane < R;
        const int64_t r = on ? rb + lane : rb;      // idle lanes read column rb and never write
        const double* F1r = F1 + r;
        const double* F2r = F2 + r;
        int64_t f = live ? pfiber[w] : 0, s = live ? pslice[w] : 0, p = p0, fb = f;
        int64_t send = (p1 > p0) ? (int64_t)pos1[s + 1] : kInf;
        long long head_id = -1, tail_id = -1;
        double head_v = 0.0, tail_v = 0.0;
        int64_t last_flush = p0;                    // entries before this index are already in M
        double accf = 0.0, accs = 0.0;
        bool first = true;
        int64_t fe_l = (p1 > p0 && fb + lane < nfiber) ? (int64_t)pos2[fb + lane + 1] : kInf;
        I j_l = (p1 > p0 && fb + lane < nfiber) ? crd1[fb + lane] : (I)0;

        while (p < p1) {
            const int64_t fe_last = __shfl_sync(0xffffffffu, fe_l, 31);
            int64_t lim = p1 - p;
            if (fe_last - p < lim) lim = fe_last - p;
            const int cnt = lim < 32 ? (int)lim : 32;
            const I k_l = (lane < cnt) ? crd2[p + lane] : (I)0;
            const double v_l = (lane < cnt) ? val[p + lane] : 0.0;
            const int64_t rel = fe_l - p - 1;
            const unsigned endmask = __reduce_or_sync(0xffffffffu, (rel >= 0 && rel < cnt) ? (1u << (int)rel) : 0u);
            const int fi0 = (int)(f - fb);          // fibre (within the register batch) of the batch's first entry

#pragma unroll
            for (int g = 0; g < 32 / kGroup; ++g) {
                if (g * kGroup < cnt) {
                    double c[kGroup], b[kGroup];
#pragma unroll
                    for (int u = 0; u < kGroup; ++u) {
                        const int t = g * kGroup + u;
                        c[u] = 0.0; b[u] = 0.0;
                        if (t < cnt) {
                            const int64_t k = SP_IDX(__shfl_sync(0xffffffffu, k_l, t), d2);
                            c[u] = F2r[k * R];
                            if ((endmask >> t) & 1u) {
                                const int fi = fi0 + __popc(endmask & ((1u << t) - 1u));
                                const int64_t j = SP_IDX(__shfl_sync(0xffffffffu, j_l, fi), d1);
                                b[u] = F1r[j * R];
                            }
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kGroup; ++u) {
                        const int t = g * kGroup + u;
                        if (t < cnt) {
                            const double v = __shfl_sync(0xffffffffu, v_l, t);
                            accf = fma(v, c[u], accf);
                            if ((endmask >> t) & 1u) {              // the fibre is complete
                                accs = fma(b[u], accf, accs);
                                accf = 0.0;
                                ++f;
                                if (f == send) {                    // and so is the slice
                                    const int64_t i = SP_IDX(crd0 ? (int64_t)crd0[s] : s, d0);
                                    if (first) { head_id = i; head_v = accs; }
                                    else if (on) M[i * R + r] = accs;
                                    first = false;
                                    last_flush = p + t + 1;
                                    accs = 0.0;
                                    ++s;
                                    while (s < nslice && (int64_t)pos1[s + 1] == f) ++s;   // slices with no fibres
                                    send = s < nslice ? (int64_t)pos1[s + 1] : kInf;
                                }
                            }
                        }
                    }
                }
            }
            p += cnt;
            if (f - fb == 32) {
                fb = f;
                fe_l = (fb + lane < nfiber) ? (int64_t)pos2[fb + lane + 1] : kInf;
                j_l = (fb + lane < nfiber) ? crd1[fb + lane] : (I)0;
            }
        }
        if (p1 > last_flush) {                      // the range ends inside slice s
            if (f < nfiber && (int64_t)pos2[f] < p1) {   // ... and inside fibre f
                const double bj = F1r[SP_IDX(crd1[f], d1) * R];
                accs = fma(bj, accf, accs);
            }
            const int64_t i = SP_IDX(crd0 ? (int64_t)crd0[s] : s, d0);
            if (first) { head_id = i; head_v = accs; }
            else { tail_id = i; tail_v = accs; }
        }
        s_car[2 * wi][lane] = head_v;
        s_car[2 * wi + 1][lane] = tail_v;
        if (lane == 0) { s_id[2 * wi] = head_id; s_id[2 * wi + 1] = tail_id; }
        __syncthreads();
        constexpr int kSlots = 2 * kTThreads / 32;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = 2 * wi + h;
            const long long id = s_id[e];
            if (id < 0) continue;
            int q = e - 1;
            while (q >= 0 && s_id[q] < 0) --q;
            if (q >= 0 && s_id[q] == id) continue;          // an earlier slot leads this run
            double sum = s_car[e][lane];
            for (int u = e + 1; u < kSlots; ++u) {
                const long long d = s_id[u];
                if (d < 0) continue;
                if (d != id) break;
                sum += s_car[u][lane];
            }
            if (on) atomicAdd(M + id * R + r, sum);
        }
        __syncthreads();
    }
}


// ---------------------------------------------------------------------------------------------
// Staged warps (R even, factor rows 16-byte aligned, dim * R < 2^29).
//
// The S groups of 32 / S lanes of a warp own a range of entries each and walk it 32 / S entries at a time: a lane
// prepares one entry of its group - the element offsets of its two factor rows, "the fibre ends here", "the slice
// ends here" - and parks that in shared memory; then the group consumes its entries one after the other, a lane
// owning S adjacent output columns.  The groups take the same steps whatever their fibres do: closing a
// fibre is accs += F1[j,:] * accf under a predicate, and only the end of a slice is a branch.
struct __align__(16) Staged {
    uint32_t koff;   // leaf factor row, byte offset (a multiple of 16) | the slice ends here
    uint32_t boff;   // level-1 factor row, byte offset | the fibre ends here
    double v;
};

// A lane's S columns are S/2 pairs; pair n sits at byte offset coff[n] of the 32-column tile,
// laid out so that the lanes of a group read one contiguous run per 16-byte load.
// W256 (S = 4, all 32 columns in use, 32-byte aligned rows): the lane's four columns are adjacent and
// come with one 32-byte load.  Rows are addressed as a uniform base and a 32-bit byte offset: address arithmetic
// in 64 bits per lane was a third of the loop's instructions.
template <int S, bool W256>
__device__ __forceinline__ void ld_cols(const char* base, uint32_t off, const uint32_t* coff, double* a) {
    if (W256) {
        asm volatile("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];"
                     : "=d"(a[0]), "=d"(a[1]), "=d"(a[S > 2 ? 2 : 0]), "=d"(a[S > 3 ? 3 : 0])
                     : "l"(base + (off | coff[0])));     // rows of whole 256-byte runs: the offset has the tile's bits clear
        return;
    }
#pragma unroll
    for (int q = 0; q < S; q += 2) {
        const double2 t = __ldg(reinterpret_cast<const double2*>(base + (off + coff[q / 2])));
        a[q] = t.x;
        a[q + 1] = t.y;
    }
}

// 20 M entries, R = 32: 479 us with ranges of 128 entries and two entries of each group in flight (one: 481, four: 514
// to 525; ranges of 64 and 256: 585, 496); 521 us when a warp walked one range in batches of 32, cut at slice ends and
// closed at every group's last entry.  5 M entries, R = 16, 24, 32: 141, 146, 145 us against 162, 167, 159.  Bound:
// the L1 pipe (64 %), instruction issue (264 M, 52 % of the slots: eight selects and eight masks per step around eight
// multiply-adds) and the latency of the row loads at 19 warps per SM together.
constexpr int kFPer = 128;      // entries per group
constexpr int kFThreads = 64;
template <typename P, typename I, int S, bool W256>
__global__ void __launch_bounds__(kFThreads, 8)
k_mttkrp_staged(const uint32_t* __restrict__ marks, const I* __restrict__ crd2, const double* __restrict__ val,
                const P* __restrict__ pos1, const I* __restrict__ crd0, const double* __restrict__ F1,
                const double* __restrict__ F2, int64_t R, double* __restrict__ M, const int64_t* __restrict__ pslice,
                int64_t nnz, int chunks, int64_t nranges, int64_t nslice,
                int64_t d0, int64_t d1, int64_t d2) {
    // chunks: chunks of the table in a group's range
    // d0, d1, d2: rows of M, F1, F2 (used by the bounds-checking debug build only)
    constexpr int GL = 32 / S;      // lanes per group = entries per group and batch
    constexpr int kStep = 2;       // entries of a group in flight
    constexpr int kWarps = kFThreads / 32, kGroups = kFThreads / GL, kSlots = 2 * kGroups;
    __shared__ Staged s_st[kWarps][32];
    __shared__ double s_sum[kSlots][32];
    __shared__ int64_t s_id[kSlots];
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, gw = lane / GL, hl = lane % GL, g = threadIdx.x / GL;
    const int64_t w = (int64_t)blockIdx.x * kGroups + g;
    const int64_t p0 = w * kFPer;
    const int nz = w < nranges ? (int)(nnz - p0 < kFPer ? nnz - p0 : kFPer) : 0;
    const int nmax = (int)__reduce_max_sync(0xffffffffu, (unsigned)nz);
    const uint32_t rbytes = (uint32_t)R * 8u;
    const int64_t rb = (int64_t)blockIdx.y * 32;
    uint32_t coff[S / 2];                  // bytes
    bool on[S / 2];
#pragma unroll
    for (int n = 0; n < S / 2; ++n) {
        const int c0 = W256 ? 4 * hl + 2 * n : n * 2 * GL + 2 * hl;
        on[n] = rb + c0 < R;
        coff[n] = on[n] ? (uint32_t)c0 * 8u : 0u;      // idle lanes read column rb and never write
    }
    auto column = [&](int q) { return (W256 ? 4 * hl + 2 * (q / 2) : (q / 2) * 2 * GL + 2 * hl) + (q & 1); };
    if (hl == 0) s_id[2 * g] = s_id[2 * g + 1] = -1;
    const char *F1g = reinterpret_cast<const char*>(F1 + rb), *F2g = reinterpret_cast<const char*>(F2 + rb);
    int64_t s = nz > 0 ? pslice[w * chunks] : 0;
    bool first = true;
    double accf[S], accs[S];
#pragma unroll
    for (int q = 0; q < S; ++q) accf[q] = accs[q] = 0.0;
    auto row_of = [&](int64_t q) { return SP_IDX(crd0 ? (int64_t)crd0[q] : q, d0); };
    auto to_slot = [&](int slot) {
#pragma unroll
        for (int q = 0; q < S; ++q) s_sum[slot][column(q)] = accs[q];
        if (hl == 0) s_id[slot] = row_of(s);
    };
    // the slice is complete: to shared memory when it began before this range, else to its row of M
    auto close_slice = [&](int64_t p) {
        if (first) {
            to_slot(2 * g);
        } else {
            double* m = M + row_of(s) * R + rb;
#pragma unroll
            for (int q = 0; q < S; q += 2)
                if (on[q / 2]) *reinterpret_cast<double2*>(m + column(q)) = make_double2(accs[q], accs[q + 1]);
        }
        first = false;
#pragma unroll
        for (int q = 0; q < S; ++q) accs[q] = 0.0;
        ++s;
        if (!crd0) {                       // level 0 dense: slices without fibres begin and end where this one ended
            const P f = pos1[s];
            while (s < nslice && pos1[s + 1] == f) ++s;
        }
    };
    uint32_t k_n = 0, m_n = 0;
    double v_n = 0.0;
    auto fetch = [&](int p) {
        k_n = m_n = 0u;
        v_n = 0.0;
        if (p + hl < nz) {
            const int64_t e = p0 + p + hl;
            const uint32_t mk = marks[e];
            k_n = (uint32_t)SP_IDX(crd2[e], d2) * rbytes | (mk >> 1 & 1u);
            m_n = (uint32_t)SP_IDX(mk >> 2, d1) * rbytes | (mk & 1u) | (p + hl == nz - 1 ? 1u : 0u);
            v_n = val[e];
        }
    };
    fetch(0);
    bool open = nz > 0;
    for (int p = 0; p < nmax; p += GL) {
        Staged st;
        st.koff = k_n;
        st.boff = m_n;
        st.v = v_n;
        s_st[wi][hl * S + gw] = st;        // the S groups read step t's entries from one 16 * S-byte run
        __syncwarp();
        fetch(p + GL);
        const Staged* mine = &s_st[wi][gw];
#pragma unroll
        for (int t0 = 0; t0 < GL; t0 += kStep) {
            // Note: no double is set to a constant zero in this loop.  Zeroing a 64-bit register
            // pair is issued on a narrow pipe that saturates long before the loads do; a closed
            // sum is cleared by masking its bits with integer ops instead, and the level-1 row is
            // read only under the same predicate that consumes it.
            Staged e[kStep];
            double c[kStep][S], b[kStep][S];
#pragma unroll
            for (int u = 0; u < kStep; ++u) {
                e[u] = mine[(t0 + u) * S];
                ld_cols<S, W256>(F2g, e[u].koff & ~1u, coff, c[u]);
                if (e[u].boff & 1u) ld_cols<S, W256>(F1g, e[u].boff & ~1u, coff, b[u]);
            }
#pragma unroll
            for (int u = 0; u < kStep; ++u) {
                const bool cl = e[u].boff & 1u;
                const long long keep = (long long)(int)((e[u].boff & 1u) - 1u);   // all ones, or 0 after a close
#pragma unroll
                for (int q = 0; q < S; ++q) {
                    accf[q] = fma(e[u].v, c[u][q], accf[q]);
                    if (cl) accs[q] = fma(b[u][q], accf[q], accs[q]);
                    accf[q] = __longlong_as_double(__double_as_longlong(accf[q]) & keep);
                }
                if (e[u].koff & 1u) {
                    close_slice(p + t0 + u);
                    open = p + t0 + u + 1 < nz;
                }
            }
        }
        __syncwarp();
    }
    if (open) to_slot(first ? 2 * g : 2 * g + 1);
    __syncthreads();
    for (int e = g; e < kSlots; e += kGroups) {     // the first of a run of equal slices adds them all up
        const int64_t id = s_id[e];
        if (id < 0) continue;
        int q = e - 1;
        while (q >= 0 && s_id[q] < 0) --q;
        if (q >= 0 && s_id[q] == id) continue;
        double sum[S];
#pragma unroll
        for (int j = 0; j < S; ++j) sum[j] = 0.0;
        for (int u = e; u < kSlots; ++u) {
            const int64_t d = s_id[u];
            if (d < 0) continue;
            if (d != id) break;
#pragma unroll
            for (int j = 0; j < S; ++j) sum[j] += s_sum[u][column(j)];
        }
#pragma unroll
        for (int j = 0; j < S; ++j)
            if (on[j / 2]) atomicAdd(M + id * R + rb + column(j), sum[j]);
    }
}

// ---------------------------------------------------------------------------------------------
// Lane groups.  marks[p] (laid out once per handle) says for entry p: level-1 coordinate of its fibre << 2 |
// "the slice ends here" << 1 | "the fibre ends here".
//
// A group of L lanes owns a range of consecutive entries and V columns a lane (L * V columns per blockIdx.y), W of
// them adjacent and fetched by one load.  The leaf rows of kU entries, and the level-1 rows of the fibres that end
// among them, are requested together; closing a fibre is accs += F1[j,:] * accf, closing a slice stores its
// row of M.  The range's last entry closes its fibre in any case: sums are linear, so a fibre may be closed in
// pieces.  Slices that reach beyond the range go through shared memory, where a block adds up what its
// groups hold of the same slice, and from there into M (zeroed first) with one atomic per column.
// Against a warp that walks one staged range: 38,175 entries 27 -> 12 us, 451,180 entries with R = 48 37 -> 28,
// 5 M entries with R = 48 306 -> 238, 3 M with R = 17 (a lane per column) 303 -> 113.  But 20 M entries with
// R = 32 551 against 479: a group that closes a fibre holds up the other groups of its warp, and 120 registers
// leave 16 warps per SM.  (kU = 2, 3, 4, 6 there: 604, 551, 644, 860.)
template <int W>
__device__ __forceinline__ void ld_run(const double* p, double* a) {
    if (W == 2) { const double2 t = *reinterpret_cast<const double2*>(p); a[0] = t.x; a[W - 1] = t.y; }
    else a[0] = *p;
}

constexpr int kGThreads = 64;     // 300,000 to 1 M entries: 128 threads 10 % slower, 256 60 %
// Asked for eight blocks per SM, the compiler spends 116 registers on three single columns a lane, as on the other
// shapes by itself (116 to 150); unasked it stops at 96 there and the loads wait for one another (3 M entries, R = 17:
// 113 us, unasked 133).
template <typename P, typename I, int L, int V, int W, int kU>
__global__ void __launch_bounds__(kGThreads, L == 8 && V == 3 ? 8 : 1)
k_mttkrp_group(const uint32_t* __restrict__ marks, const I* __restrict__ crd2, const double* __restrict__ val,
               const P* __restrict__ pos1, const I* __restrict__ crd0, const double* __restrict__ F1,
               const double* __restrict__ F2, int64_t R, int64_t cols, double* __restrict__ M, const int64_t* __restrict__ pslice,
               const int64_t* __restrict__ prow, int64_t nnz, int per, int chunks, int64_t nranges, int64_t nslice,
               int64_t d0, int64_t d1, int64_t d2) {
    // cols of the R columns, from where F1, F2 and M point on; chunks: of the table, in a group's range of per entries
    // d0, d1, d2: rows of M, F1, F2 (used by the bounds-checking debug build only)
    constexpr int kGroups = kGThreads / L, kSlots = 2 * kGroups;
    __shared__ double s_sum[kSlots][L * V];         // slot 2 g: the slice group g's range begins in, 2 g + 1: the one it ends in
    __shared__ int64_t s_id[kSlots];                // its row of M, -1 = nothing
    const int g = threadIdx.x / L, gl = threadIdx.x % L;
    const int64_t w = (int64_t)blockIdx.x * kGroups + g;
    const int64_t p0 = w * per;
    const int nz = w < nranges ? (int)(nnz - p0 < per ? nnz - p0 : per) : 0;
    const int64_t cb = (int64_t)blockIdx.y * (L * V);
    int coff[V / W];                                // idle lanes read the tile's first run and never write
    bool on[V / W];
#pragma unroll
    for (int j = 0; j < V / W; ++j) {
        const int c = (j * L + gl) * W;
        on[j] = cb + c < cols;
        coff[j] = on[j] ? c : 0;
    }
    auto slot_put = [&](int slot, const double (&a)[V], int64_t id) {
#pragma unroll
        for (int j = 0; j < V; ++j) s_sum[slot][(j / W * L + gl) * W + j % W] = a[j];
        if (gl == 0) s_id[slot] = id;
    };
    if (gl == 0) s_id[2 * g] = s_id[2 * g + 1] = -1;
    if (nz > 0) {
        const double *F1g = F1 + cb, *F2g = F2 + cb;
        const uint32_t* ml = marks + p0;
        const I* cl = crd2 + p0;
        const double* vl = val + p0;
        int64_t s = pslice[w * chunks];
        int64_t i = SP_IDX(prow[w * chunks], d0);
        bool first = true, open = true;
        double accf[V], accs[V];
#pragma unroll
        for (int j = 0; j < V; ++j) accf[j] = accs[j] = 0.0;
        uint32_t mn[kU];
        I kn[kU];
        double vn[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {              // the group's lanes read the same word: one transaction
            const int q = u < nz ? u : nz - 1;
            mn[u] = ml[q] | (q == nz - 1 ? 4u << 29 : 0u);
            kn[u] = cl[q];
            vn[u] = vl[q];
        }
        for (int p = 0; p < nz; p += kU) {
            double c[kU][V], b[kU][V], v[kU];
            uint32_t mk[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                mk[u] = mn[u];
                v[u] = vn[u];
                const double* row = F2g + (int64_t)SP_IDX(kn[u], d2) * R;
#pragma unroll
                for (int j = 0; j < V / W; ++j) ld_run<W>(row + coff[j], c[u] + j * W);
                if (mk[u] & (1u | 1u << 31)) {      // bit 31: the range's last entry
                    const double* brow = F1g + (int64_t)SP_IDX((mk[u] >> 2) & 0x1fffffffu, d1) * R;
#pragma unroll
                    for (int j = 0; j < V / W; ++j) ld_run<W>(brow + coff[j], b[u] + j * W);
                }
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int q = p + kU + u < nz ? p + kU + u : nz - 1;
                mn[u] = ml[q] | (q == nz - 1 ? 4u << 29 : 0u);
                kn[u] = cl[q];
                vn[u] = vl[q];
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                if (p + u < nz) {
#pragma unroll
                    for (int j = 0; j < V; ++j) accf[j] = fma(v[u], c[u][j], accf[j]);
                    if (mk[u] & (1u | 1u << 31)) {
#pragma unroll
                        for (int j = 0; j < V; ++j) { accs[j] = fma(b[u][j], accf[j], accs[j]); accf[j] = 0.0; }
                        if (mk[u] & 2u) {           // the slice is complete
                            if (first) {
                                slot_put(2 * g, accs, i);
                            } else {
#pragma unroll
                                for (int j = 0; j < V / W; ++j)
                                    if (on[j]) {
                                        double* m = M + i * R + cb + coff[j];
                                        if (W == 2) *reinterpret_cast<double2*>(m) = make_double2(accs[j * W], accs[j * W + W - 1]);
                                        else *m = accs[j];
                                    }
                            }
                            first = false;
#pragma unroll
                            for (int j = 0; j < V; ++j) accs[j] = 0.0;
                            ++s;
                            if (!crd0) {            // slices with no fibres
                                const P f = pos1[s];
                                while (s < nslice && pos1[s + 1] == f) ++s;
                            }
                            open = p + u + 1 < nz;
                            if (open) i = SP_IDX(crd0 ? (int64_t)crd0[s] : s, d0);
                        }
                    }
                }
            }
        }
        if (open) slot_put(first ? 2 * g : 2 * g + 1, accs, i);
    }
    __syncthreads();
    for (int e = g; e < kSlots; e += kGroups) {     // the first of a run of equal slices adds them all up
        const int64_t id = s_id[e];
        if (id < 0) continue;
        int q = e - 1;
        while (q >= 0 && s_id[q] < 0) --q;
        if (q >= 0 && s_id[q] == id) continue;
        double sum[V];
#pragma unroll
        for (int j = 0; j < V; ++j) sum[j] = 0.0;
        for (int u = e; u < kSlots; ++u) {
            const int64_t d = s_id[u];
            if (d < 0) continue;
            if (d != id) break;
#pragma unroll
            for (int j = 0; j < V; ++j) sum[j] += s_sum[u][(j / W * L + gl) * W + j % W];
        }
#pragma unroll
        for (int j = 0; j < V; ++j)
            if (on[j / W]) atomicAdd(M + id * R + cb + coff[j / W] + j % W, sum[j]);
    }
}

}  // namespace

// F1 / F2: factor matrices of the dimensions stored at levels 1 / 2; M: rows of the level-0 dimension.
static sp_status mttkrp_levels(sp_tensor* T, const double* F1, const double* F2, int64_t R, double* M, cudaStream_t stream);

extern "C" sp_status sp_mttkrp(sp_tensor* T, const double* B, const double* C, int64_t R, double* M, void* stream_) {
    SP_API_RANGE("sp_mttkrp");
    if (!T || !B || !C || !M || R < 1) return SP_ERR_INVALID_ARG;
    if (T->rank != 3 || T->ord[0] != 0 || T->lt[1] != SP_COMPRESSED || T->lt[2] != SP_COMPRESSED)
        return SP_ERR_UNSUPPORTED;
    return mttkrp_levels(T, T->ord[1] == 1 ? B : C, T->ord[1] == 1 ? C : B, R, M, static_cast<cudaStream_t>(stream_));
}

extern "C" sp_status sp_mttkrp_mode(sp_tensor* T, int mode, const double* const* factors, int64_t R, double* M,
                                    void* stream_) {
    SP_API_RANGE("sp_mttkrp_mode");
    if (!T || !factors || !M || R < 1 || mode < 0 || mode > 2) return SP_ERR_INVALID_ARG;
    if (T->rank != 3 || T->ord[0] != mode || T->lt[1] != SP_COMPRESSED || T->lt[2] != SP_COMPRESSED)
        return SP_ERR_UNSUPPORTED;
    const double* F1 = factors[T->ord[1]];
    const double* F2 = factors[T->ord[2]];
    if (!F1 || !F2) return SP_ERR_INVALID_ARG;
    return mttkrp_levels(T, F1, F2, R, M, static_cast<cudaStream_t>(stream_));
}

static sp_status mttkrp_levels(sp_tensor* T, const double* F1, const double* F2, int64_t R, double* M, cudaStream_t stream) {
    if (sp_check_device(T) != SP_OK) return SP_ERR_INVALID_ARG;
    {   // 8- and 16-bit storage is read through its 32-bit shadow
        sp_tensor* wide_ = nullptr;
        const sp_status ws_ = sp_widened(T, stream, &wide_);
        if (ws_ != SP_OK) return ws_;
        T = wide_;
    }
    const double* B = F1;
    const double* C = F2;
    SP_CUDA(cudaMemsetAsync(M, 0, (size_t)T->dims[T->ord[0]] * R * sizeof(double), stream));
    const int64_t nnz = T->ncrd[2];
    if (nnz == 0) return SP_OK;
    const int64_t d1 = T->dims[T->ord[1]], d2 = T->dims[T->ord[2]];
    const int64_t maxdim = d1 > d2 ? d1 : d2;
    const bool fast = (R % 2 == 0) && maxdim * R < ((int64_t)1 << 29) && reinterpret_cast<uintptr_t>(B) % 16 == 0 &&
                      reinterpret_cast<uintptr_t>(C) % 16 == 0 && reinterpret_cast<uintptr_t>(M) % 16 == 0;
    // Large tensors with 8 < R <= 32 take the staged warps: R = 16, 24, 32 and 5 M entries 141, 146, 145 us against
    // 165, 197, 189; 1 M entries, R = 32: 38 against 44.  R = 8 goes to lane groups, whose four lanes all have columns.
    const bool staged = fast && nnz >= 1000000 && R > 8 && R <= 32;
    // Entries per group, as below per warp.  The table says where chunks begin that both this range and the staged one are
    // whole numbers of, so that every R finds what it needs in the handle's one table.  (Ranges of whole 64s instead, for
    // longer chunks: 1.3 to 4 M entries, R = 17 and 48, 4 to 12 % slower.)
    const int64_t per = std::max<int64_t>(16, std::min<int64_t>(256, sp_ceil_div(sp_ceil_div(nnz, 18944), 16) * 16));
    const int64_t chunk = std::min<int64_t>(per & -per, kFPer);
    if (!staged && d1 < ((int64_t)1 << 29)) {
        sp_partition part;
        sp_status st = sp_get_mttkrp_partition(T, chunk, true, stream, &part);
        if (st != SP_OK) return st;
        const int64_t ranges = sp_ceil_div(nnz, per);
        const bool pairs = R % 2 == 0 && reinterpret_cast<uintptr_t>(B) % 16 == 0 && reinterpret_cast<uintptr_t>(C) % 16 == 0 &&
                           reinterpret_cast<uintptr_t>(M) % 16 == 0;
        // a launch covers at most 65,535 tiles of columns
#define SP_MTTKRP_GROUP(L, V, W, U)                                                                                        \
    for (int64_t c0 = 0; c0 < R; c0 += (int64_t)65535 * (L * V))                                                           \
    k_mttkrp_group<P, I, L, V, W, U><<<dim3((unsigned)sp_ceil_div(ranges * L, kGThreads),                                  \
                                            (unsigned)std::min<int64_t>(65535, sp_ceil_div(R - c0, L * V))), kGThreads, 0, stream>>>( \
        part.marks, static_cast<const I*>(T->crd[2]), T->val, static_cast<const P*>(T->pos[1]),                            \
        T->lt[0] == SP_COMPRESSED ? static_cast<const I*>(T->crd[0]) : nullptr, F1 + c0, F2 + c0, R, R - c0, M + c0,       \
        part.aux, part.row, nnz, (int)per, (int)(per / chunk), ranges, T->npos[1] - 1, T->dims[T->ord[0]], d1, d2)
        SP_DISPATCH_WIDTHS(T, {
            if (pairs) {
                if (R <= 8) SP_MTTKRP_GROUP(4, 2, 2, 6);
                else if (R <= 16) SP_MTTKRP_GROUP(4, 4, 2, 3);
                else if (R <= 24) SP_MTTKRP_GROUP(4, 6, 2, 2);
                else if (R <= 32) SP_MTTKRP_GROUP(8, 4, 2, 3);
                else if (R <= 48) SP_MTTKRP_GROUP(8, 6, 2, 2);
                else SP_MTTKRP_GROUP(16, 4, 2, 3);
            } else {
                if (R <= 8) SP_MTTKRP_GROUP(4, 2, 1, 6);
                else if (R <= 16) SP_MTTKRP_GROUP(8, 2, 1, 6);
                else if (R <= 24) SP_MTTKRP_GROUP(8, 3, 1, 3);
                else if (R <= 32) SP_MTTKRP_GROUP(8, 4, 1, 3);
                else if (R <= 48) SP_MTTKRP_GROUP(16, 3, 1, 3);
                else SP_MTTKRP_GROUP(16, 4, 1, 3);
            }
        });
#undef SP_MTTKRP_GROUP
        SP_LAUNCH_CHECK();
        sp_count_launches(1);
        SP_BOUNDS_RETURN(stream);
        return SP_OK;
    }
    sp_partition part;
    if (staged) {
        sp_status st = sp_get_mttkrp_partition(T, chunk, true, stream, &part);
        if (st != SP_OK) return st;
        const int64_t ranges = sp_ceil_div(nnz, kFPer);
#define SP_MTTKRP_STAGED(S, W)                                                                                             \
    k_mttkrp_staged<P, I, S, W><<<dim3((unsigned)sp_ceil_div(ranges * (32 / S), kFThreads), (unsigned)sp_ceil_div(R, 32)), kFThreads, 0, stream>>>( \
        part.marks, static_cast<const I*>(T->crd[2]), T->val, static_cast<const P*>(T->pos[1]),                            \
        T->lt[0] == SP_COMPRESSED ? static_cast<const I*>(T->crd[0]) : nullptr, F1, F2, R, M, part.aux, nnz, (int)(kFPer / chunk), ranges, \
        T->npos[1] - 1, T->dims[T->ord[0]], d1, d2)
        // one 32-byte load per lane and factor row when every lane has its four columns and rows are 32-byte aligned
        const bool w256 = R % 32 == 0 && reinterpret_cast<uintptr_t>(F1) % 32 == 0 && reinterpret_cast<uintptr_t>(F2) % 32 == 0;
        SP_DISPATCH_WIDTHS(T, {
            if (w256) SP_MTTKRP_STAGED(4, true);
            else if (R % 4 == 0) SP_MTTKRP_STAGED(4, false);
            else SP_MTTKRP_STAGED(2, false);
        });
#undef SP_MTTKRP_STAGED
        SP_LAUNCH_CHECK();
        sp_count_launches(1);
        SP_BOUNDS_RETURN(stream);
        return SP_OK;
    }
    // Level-1 sizes of 2^29 and more: entries per warp as above
    const int64_t wper = std::max<int64_t>(32, std::min<int64_t>(512, sp_ceil_div(sp_ceil_div(nnz, 4736), 32) * 32));
    sp_status st = sp_get_mttkrp_partition(T, wper, false, stream, &part);
    if (st != SP_OK) return st;
    const unsigned blocks = (unsigned)sp_ceil_div(part.nchunks * 32, kTThreads);
    SP_DISPATCH_WIDTHS(T, {
        k_mttkrp<P, I><<<blocks, kTThreads, 0, stream>>>(
            static_cast<const P*>(T->pos[1]), T->lt[0] == SP_COMPRESSED ? static_cast<const I*>(T->crd[0]) : nullptr,
            static_cast<const P*>(T->pos[2]), static_cast<const I*>(T->crd[1]), static_cast<const I*>(T->crd[2]),
            T->val, F1, F2, R, M, part.row, part.nz, part.aux, part.nchunks, T->npos[1] - 1, T->ncrd[1],
            T->dims[T->ord[0]], d1, d2);
    });
    SP_LAUNCH_CHECK();
    sp_count_launches(1);
    SP_BOUNDS_RETURN(stream);
    return SP_OK;
}
