// sp_sddmm: X[i,j] = S[i,j] * sum_k A[i,k] * B[k,j] over the stored (i,j) of S
// (Section 6.2), S in any two-dimensional encoding, row- or column-major.
//
// Compressed inner level (CSR, DCSR, CSC, DCSC):
// Loop shape: for each stored row i, for each p in pos[1][q]..pos[1][q+1]:
// j = crd[1][p]; x[p] = S.val[p] * dot(A[i,:], B[:,j]).  B is given K x n row-major,
// so a column is K elements a whole row apart; it is transposed once per call into
// a workspace so each entry reads one contiguous K-vector.  The (row end, entry)
// merge path is cut into equal pieces, one per lane group (k_sddmm_group).
#include "common.cuh"

namespace {

constexpr int kSThreads = 64;
constexpr int kGThreads = 64;  // of k_sddmm_group (32: the same; 128: 265 us against 262)

__global__ void __launch_bounds__(256)
k_transpose(const double* __restrict__ B, int64_t ldb, int64_t K, int64_t n, double* __restrict__ Bt, int64_t ldt) {
    __shared__ double tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 32 x 8
    const int64_t j0 = (int64_t)blockIdx.x * 32, k0 = (int64_t)blockIdx.y * 32;
#pragma unroll
    for (int r = ty; r < 32; r += 8) {
        int64_t k = k0 + r, j = j0 + tx;
        tile[r][tx] = (k < K && j < n) ? B[k * ldb + j] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int r = ty; r < 32; r += 8) {
        int64_t j = j0 + r, k = k0 + tx;
        if (j < n && k < ldt) Bt[j * ldt + k] = tile[tx][r];      // zeros from K up to ldt
    }
}

template <int V>
__device__ __forceinline__ void ld2(const double* p, double* a) {
    if (V == 2) { const double2 q = *reinterpret_cast<const double2*>(p); a[0] = q.x; a[V - 1] = q.y; }
    else a[0] = *p;
}

// K > 512: a warp per merge-path piece, one dot product at a time; the operand row is re-read (from L1) for
// every entry.
template <typename P, typename I, int V>
__global__ void __launch_bounds__(kSThreads)
k_sddmm(const P* __restrict__ pos, const I* __restrict__ crd, const double* __restrict__ sval,
        const I* __restrict__ outer, const double* A, int64_t lda, const double* Bt,
        int64_t ldt, int64_t K, double* __restrict__ xv, const int64_t* __restrict__ prow,
        const int64_t* __restrict__ pnz, int64_t nchunks, int64_t na, int64_t nb) {
    // na, nb: rows of A and of Bt (used by the bounds-checking debug build only)
    sp_wait_for_previous_kernel();      // the transpose that wrote Bt
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (w >= nchunks) return;
    const int lane = threadIdx.x & 31;
    const int64_t i0 = prow[w], j0 = pnz[w], i1 = prow[w + 1], j1 = pnz[w + 1];
    if (j1 == j0) return;
    int64_t row = i0, p = j0, rbase = i0, nzbase = j0;
    int64_t E = (rbase + lane < i1) ? (int64_t)pos[rbase + lane + 1] : j1;
    I c_l = (nzbase + lane < j1) ? crd[nzbase + lane] : (I)0;
    double v_l = (nzbase + lane < j1) ? sval[nzbase + lane] : 0.0;
    double res = 0.0;

    while (true) {
        const int64_t rend = row < i1 ? __shfl_sync(0xffffffffu, E, (int)(row - rbase)) : j1;
        const double* arow = p < rend ? A + SP_IDX(outer ? (int64_t)outer[row] : row, na) * lda : nullptr;
        while (p < rend) {
            int off = (int)(p - nzbase);
            if (off == 32) {
                if (nzbase + lane < j1) xv[nzbase + lane] = v_l * res;
                nzbase += 32;
                c_l = (nzbase + lane < j1) ? crd[nzbase + lane] : (I)0;
                v_l = (nzbase + lane < j1) ? sval[nzbase + lane] : 0.0;
                off = 0;
            }
            const int cnt = (int)min(rend - p, (int64_t)(32 - off));
            for (int t = 0; t < cnt; ++t) {
                const int64_t j = SP_IDX(__shfl_sync(0xffffffffu, c_l, off + t), nb);
                const double* brow = Bt + j * ldt;
                double part = 0.0;
                for (int64_t kk = (int64_t)lane * V; kk < K; kk += 32 * V) {
                    double b[V], aa[V];
                    ld2<V>(brow + kk, b);
                    ld2<V>(arow + kk, aa);
#pragma unroll
                    for (int q = 0; q < V; ++q) part = fma(aa[q], b[q], part);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
                if (lane == off + t) res = part;
            }
            p += cnt;
        }
        if (row >= i1) break;
        ++row;
        if (row - rbase == 32) {
            rbase += 32;
            E = (rbase + lane < i1) ? (int64_t)pos[rbase + lane + 1] : j1;
        }
    }
    if (nzbase + lane < j1) xv[nzbase + lane] = v_l * res;
}

// K <= 512: a group of L lanes owns a merge-path piece and V factors a lane (K <= L * V), W of them adjacent.  The
// operand row of the piece's current row sits in registers; the gathered rows of the next kDepth entries
// are on their way into shared memory by asynchronous copies, every lane into slots of its own (nobody else
// reads them, so nothing is synchronised and nothing in flight holds a register).  The dot products of
// kDepth entries are folded over the group together, each exchange halving the number of sums a lane
// carries, and the groups of a warp share the loop's instructions.
// 2,000,000 samples, K = 128, operands of 134 MB: 262 us with the transpose, 304 us when a warp took one dot
// product at a time; L = 8, 16, 32: 290, 262, 270 (fewer lanes, fewer copies of the loop in flight; more,
// more instructions).  Bound: HBM, since the gathered operand does not fit L2 (1.22 GB for 0.3 GB of
// operands, 73 % of the pin rate, which is what a copy reaches).  Operand rows kept in registers and loaded ahead cost 190 and more
// registers (342 us); requested through the ring as well, twice the shared memory (273 us).
constexpr int kDepth = 4;

template <int W>
__device__ __forceinline__ void copy_async(double* dst, const double* src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (W == 2) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

template <typename P, typename I, int L, int V, int W, bool FULL>
__global__ void __launch_bounds__(kGThreads)
k_sddmm_group(const P* __restrict__ pos, const I* __restrict__ crd, const double* __restrict__ sval,
              const I* __restrict__ outer, const double* A, int64_t lda, int avec, const double* G, int64_t ldg, int K,
              double* __restrict__ xv, const int64_t* __restrict__ prow, const int64_t* __restrict__ pnz, int64_t nchunks,
              int64_t nseg, int64_t na, int64_t nb) {
    // na, nb: rows of A and of G (used by the bounds-checking debug build only)
    sp_wait_for_previous_kernel();                  // the transpose that wrote one of the operands
    extern __shared__ __align__(16) double s_ring[];            // [kDepth][V / W][threads] runs of W
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / L;
    if (w >= nchunks) return;                       // shuffles below stay inside a group
    const int gl = threadIdx.x % L;
    const unsigned gmask = L == 32 ? 0xffffffffu : ((1u << (L & 31)) - 1u) << (sp_lane() / L * L);
    const int64_t i0 = prow[w], j0 = pnz[w];
    const int nrows = (int)(prow[w + 1] - i0), nz = (int)(pnz[w + 1] - j0);
    if (nz == 0) return;
    const P* ends = pos + i0 + 1;                   // row r of the piece ends at entry ends[r]; the open row at nz
    const I* cl = crd + j0;
    const double* vl = sval + j0;
    double* xl = xv + j0;
    double* slot = s_ring + threadIdx.x * W;
    int koff[V / W];
    bool on[V / W];
#pragma unroll
    for (int j = 0; j < V / W; ++j) {
        const int k = (j * L + gl) * W;
        on[j] = FULL || k < K;
        koff[j] = on[j] ? k : 0;
    }
    auto request = [&](int u, I k) {                // entry's row of G into ring position u
        const double* row = G + (int64_t)SP_IDX(k, nb) * ldg;
#pragma unroll
        for (int j = 0; j < V / W; ++j)
            if (on[j]) copy_async<W>(slot + (u * (V / W) + j) * (kGThreads * W), row + koff[j]);
    };
    double a[V];
    auto load_row = [&](int r) {
        const double* arow = A + SP_IDX(outer ? (int64_t)outer[i0 + r] : i0 + r, na) * lda;
#pragma unroll
        for (int j = 0; j < V / W; ++j) {
            if (W == 2 && avec) {
                const double2 x = *reinterpret_cast<const double2*>(arow + koff[j]);
                a[j * W] = on[j] ? x.x : 0.0;
                a[j * W + W - 1] = on[j] ? x.y : 0.0;
            } else {
#pragma unroll
                for (int q = 0; q < W; ++q) a[j * W + q] = on[j] && koff[j] + q < K ? arow[koff[j] + q] : 0.0;
            }
        }
    };
    auto end_of = [&](int r) { return r < nrows ? (int)((int64_t)ends[r] - j0) : nz; };
    int row = 0, rend = end_of(0);
    while (rend == 0) rend = end_of(++row);         // rows without entries; nz > 0 ends this
    I kn[kDepth];
#pragma unroll
    for (int u = 0; u < kDepth; ++u) {
        if (u < nz) request(u, cl[u]);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    load_row(row);
#pragma unroll
    for (int u = 0; u < kDepth; ++u) kn[u] = cl[kDepth + u < nz ? kDepth + u : nz - 1];
    constexpr int kSpan = L / kDepth < 1 ? 1 : L / kDepth;      // lanes that end up with the same entry's sum
    const int mine = gl / kSpan;
    for (int p = 0; p < nz; p += kDepth) {
        const bool writer = gl % kSpan == 0 && p + mine < nz;
        const double sv = writer ? vl[p + mine] : 0.0;
        double part[kDepth];
#pragma unroll
        for (int u = 0; u < kDepth; ++u) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kDepth - 1) : "memory");
            part[u] = 0.0;
            if (p + u < nz) {
                if (p + u == rend) {                // the next row with entries
                    do rend = end_of(++row); while (rend == p + u);
                    load_row(row);
                }
#pragma unroll
                for (int j = 0; j < V / W; ++j) {
                    const double* x = slot + (u * (V / W) + j) * (kGThreads * W);
                    if (W == 2) {
                        double2 t = *reinterpret_cast<const double2*>(x);
                        if (!FULL && !on[j]) t = make_double2(0.0, 0.0);
                        part[u] = fma(a[j * W], t.x, part[u]);
                        part[u] = fma(a[j * W + W - 1], t.y, part[u]);
                    } else if (FULL || on[j]) {
                        part[u] = fma(a[j], *x, part[u]);
                    }
                }
                if (p + kDepth + u < nz) request(u, kn[u]);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
#pragma unroll
        for (int u = 0; u < kDepth; ++u) kn[u] = cl[p + 2 * kDepth + u < nz ? p + 2 * kDepth + u : nz - 1];
        int o = L / 2;
        {
            const bool h = gl & o;
            const double s0 = __shfl_xor_sync(gmask, h ? part[0] : part[2], o), s1 = __shfl_xor_sync(gmask, h ? part[1] : part[3], o);
            part[0] = (h ? part[2] : part[0]) + s0;
            part[1] = (h ? part[3] : part[1]) + s1;
            o >>= 1;
        }
        {
            const bool h = gl & o;
            const double s0 = __shfl_xor_sync(gmask, h ? part[0] : part[1], o);
            part[0] = (h ? part[1] : part[0]) + s0;
            o >>= 1;
        }
#pragma unroll
        for (; o > 0; o >>= 1) part[0] += __shfl_xor_sync(gmask, part[0], o);
        if (writer) xl[p + mine] = sv * part[0];
    }
}

// S with a dense inner level ((dense|compressed, dense), either ordering): every cell of a stored
// outer index is a stored value, so x[q * ninner + c] = S.val[..] * sum_k Out[o,k] * In[k,c] with
// o the outer coordinate of stored row q.  One thread per inner coordinate c (loads of In[k, c..]
// coalesce, Out[o,k] is a broadcast), kDQ stored outer rows per block share each load of In.
constexpr int kDQ = 4;

template <typename I>
__global__ void __launch_bounds__(256)
k_sddmm_dense_inner(const I* __restrict__ outer, int64_t nouter, int64_t ninner, const double* __restrict__ sval,
                    const double* __restrict__ Out, int64_t out_row_stride, int64_t out_k_stride,
                    const double* __restrict__ In, int64_t ldin, int64_t K, double* __restrict__ xv, int64_t nouter_dim) {
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t q0 = (int64_t)blockIdx.y * kDQ; q0 < nouter; q0 += (int64_t)gridDim.y * kDQ) {
        const double* orow[kDQ];
        double acc[kDQ];
#pragma unroll
        for (int r = 0; r < kDQ; ++r) {
            const int64_t q = q0 + r < nouter ? q0 + r : nouter - 1;
            orow[r] = Out + SP_IDX(outer ? (int64_t)outer[q] : q, nouter_dim) * out_row_stride;
            acc[r] = 0.0;
        }
        if (c < ninner) {
            for (int64_t k = 0; k < K; ++k) {
                const double b = In[k * ldin + c];
#pragma unroll
                for (int r = 0; r < kDQ; ++r) acc[r] = fma(orow[r][k * out_k_stride], b, acc[r]);
            }
#pragma unroll
            for (int r = 0; r < kDQ; ++r) {
                const int64_t p = (q0 + r) * ninner + c;
                if (q0 + r < nouter) xv[p] = sval[p] * acc[r];
            }
        }
    }
}

sp_status sddmm_dense_inner(sp_tensor* S, const double* A, int64_t lda, const double* B, int64_t ldb, int64_t K,
                            double* x_vals, cudaStream_t stream) {
    if (S->nval == 0) return SP_OK;
    if (!x_vals) return SP_ERR_INVALID_ARG;
    const bool colmajor = S->ord[0] == 1;
    const bool dbl = S->lt[0] == SP_COMPRESSED;
    const int64_t ninner = S->dims[S->ord[1]];
    const int64_t nouter = dbl ? S->ncrd[0] : S->dims[S->ord[0]];
    if (nouter == 0 || ninner == 0) return SP_OK;
    sp_workspace ws(stream);
    const double *Out = A, *In = B;
    int64_t out_row = lda, out_k = 1, ldin = ldb;
    if (colmajor) {
        // outer = column j: Out[j,k] = B[k,j]; inner = row i: In[k,i] = A[i,k], transposed once so that
        // neighbouring threads read neighbouring addresses
        const int64_t m = S->dims[0];
        double* At = ws.get<double>((size_t)K * m);
        if (ws.failed) return SP_ERR_ALLOC;
        dim3 tg((unsigned)sp_ceil_div(K, 32), (unsigned)sp_ceil_div(m, 32));
        k_transpose<<<tg, 256, 0, stream>>>(A, lda, m, K, At, m);
        SP_LAUNCH_CHECK();
        sp_count_launches(1);
        Out = B; out_row = 1; out_k = ldb;
        In = At; ldin = m;
    }
    dim3 grid((unsigned)sp_ceil_div(ninner, 256), (unsigned)std::min<int64_t>(sp_ceil_div(nouter, kDQ), 32768));
    if (S->crdBits == 32)
        k_sddmm_dense_inner<uint32_t><<<grid, 256, 0, stream>>>(dbl ? static_cast<const uint32_t*>(S->crd[0]) : nullptr, nouter,
                                                               ninner, S->val, Out, out_row, out_k, In, ldin, K, x_vals, S->dims[S->ord[0]]);
    else
        k_sddmm_dense_inner<uint64_t><<<grid, 256, 0, stream>>>(dbl ? static_cast<const uint64_t*>(S->crd[0]) : nullptr, nouter,
                                                               ninner, S->val, Out, out_row, out_k, In, ldin, K, x_vals, S->dims[S->ord[0]]);
    SP_LAUNCH_CHECK();
    sp_count_launches(1);
    return SP_OK;
}

}  // namespace

extern "C" sp_status sp_sddmm(sp_tensor* S, const double* A, int64_t lda, const double* B, int64_t ldb, int64_t K,
                              double* x_vals, void* stream_) {
    SP_API_RANGE("sp_sddmm");
    if (!S || !A || !B || K < 1 || lda < K) return SP_ERR_INVALID_ARG;
    if (sp_check_device(S) != SP_OK) return SP_ERR_INVALID_ARG;
    {   // 8- and 16-bit storage is read through its 32-bit shadow
        sp_tensor* wide_ = nullptr;
        const sp_status ws_ = sp_widened(S, static_cast<cudaStream_t>(stream_), &wide_);
        if (ws_ != SP_OK) return ws_;
        S = wide_;
    }
    if (S->rank != 2 || S->ord[0] == S->ord[1]) return SP_ERR_UNSUPPORTED;
    if (ldb < S->dims[1]) return SP_ERR_INVALID_ARG;
    if (S->lt[1] == SP_DENSE) return sddmm_dense_inner(S, A, lda, B, ldb, K, x_vals, static_cast<cudaStream_t>(stream_));
    const bool colmajor = S->ord[0] == 1;      // S stored by columns (CSC, DCSC)
    const int64_t n = S->dims[1];
    if (ldb < n) return SP_ERR_INVALID_ARG;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const int64_t nnz = S->ncrd[1];
    if (nnz == 0) return SP_OK;
    if (!x_vals) return SP_ERR_INVALID_ARG;
    const bool dbl = S->lt[0] == SP_COMPRESSED;

    // The pieces of either kernel, so that a handle has one table whatever K is: shorter ones where there are few (30,000 to
    // 115,000 entries, K <= 512: 10 against 14 us; 240,000 and up: no gain).
    const int64_t nseg = S->npos[1] - 1;
    const int64_t items = nseg + nnz < 200000 ? 16 : 32;
    const bool pair_a = K % 2 == 0 && lda % 2 == 0 && reinterpret_cast<uintptr_t>(A) % 16 == 0;
    if (K <= 512) {
        sp_workspace ws(stream);
        const int64_t ldt = (K + 1) & ~(int64_t)1;
        double* Bt = ws.get<double>((size_t)n * ldt + 2);
        if (ws.failed) return SP_ERR_ALLOC;
        Bt = reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(Bt) + 15) & ~(uintptr_t)15);
        k_transpose<<<dim3((unsigned)sp_ceil_div(n, 32), (unsigned)sp_ceil_div(ldt, 32)), 256, 0, stream>>>(B, ldb, K, n, Bt, ldt);
        SP_LAUNCH_CHECK();
        sp_partition part;
        const sp_status st = sp_get_merge_partition(S, items, stream, &part);
        if (st != SP_OK) return st;
        // row in registers / gathered row: A and B^T, or for column-major S the other way round
        const double *reg = colmajor ? Bt : A, *gat = colmajor ? A : Bt;
        const int64_t ldreg = colmajor ? ldt : lda, ldgat = colmajor ? lda : ldt;
        const bool pairs = !colmajor || pair_a;
        const int avec = colmajor || pair_a;
        cudaError_t e = cudaSuccess;
#define SP_SG_LAUNCH(L, V, W, FULL)                                                                                       \
    do {                                                                                                                   \
        constexpr size_t ring = (size_t)kDepth * V * kGThreads * sizeof(double);                                           \
        e = sp_allow_shared<k_sddmm_group<P, I, L, V, W, FULL>>(S->device, ring);                                          \
        if (e == cudaSuccess)                                                                                              \
            e = sp_launch_dependent(k_sddmm_group<P, I, L, V, W, FULL>, dim3((unsigned)sp_ceil_div(part.nchunks * L, kGThreads)), \
                                    dim3(kGThreads), ring, stream, pos, crd, (const double*)S->val, outer, reg, ldreg, avec, gat, ldgat, \
                                    (int)K, x_vals, (const int64_t*)part.row, (const int64_t*)part.nz, part.nchunks, nseg, \
                                    S->dims[S->ord[0]], S->dims[S->ord[1]]);                                               \
    } while (0)
        SP_DISPATCH_WIDTHS(S, {
            const P* pos = static_cast<const P*>(S->pos[1]);
            const I* crd = static_cast<const I*>(S->crd[1]);
            const I* outer = dbl ? static_cast<const I*>(S->crd[0]) : nullptr;
            // K that fills a shape's lanes needs no masks: K = 16, 256, 512 with them 66.0, 414, 546 us, without 59.2, 388,
            // 532 (2 M, 1 M, 0.5 M samples of a 131,072-square matrix)
            if (pairs) {
                if (K == 512) SP_SG_LAUNCH(32, 16, 2, true);
                else if (K == 256) SP_SG_LAUNCH(16, 16, 2, true);
                else if (K == 128) SP_SG_LAUNCH(16, 8, 2, true);
                else if (K == 96) SP_SG_LAUNCH(16, 6, 2, true);
                else if (K == 64) SP_SG_LAUNCH(16, 4, 2, true);
                else if (K == 32) SP_SG_LAUNCH(8, 4, 2, true);
                else if (K == 16) SP_SG_LAUNCH(4, 4, 2, true);
                else if (K <= 16) SP_SG_LAUNCH(4, 4, 2, false);
                else if (K < 32) SP_SG_LAUNCH(8, 4, 2, false);
                else if (K < 64) SP_SG_LAUNCH(16, 4, 2, false);
                else if (K < 96) SP_SG_LAUNCH(16, 6, 2, false);
                else if (K < 128) SP_SG_LAUNCH(16, 8, 2, false);
                else if (K <= 256) SP_SG_LAUNCH(16, 16, 2, false);
                else SP_SG_LAUNCH(32, 16, 2, false);
            } else {
                if (K <= 16) SP_SG_LAUNCH(4, 4, 1, false);
                else if (K <= 32) SP_SG_LAUNCH(8, 4, 1, false);
                else if (K <= 64) SP_SG_LAUNCH(8, 8, 1, false);
                else if (K <= 128) SP_SG_LAUNCH(16, 8, 1, false);
                else if (K <= 256) SP_SG_LAUNCH(32, 8, 1, false);
                else SP_SG_LAUNCH(32, 16, 1, false);
            }
        });
#undef SP_SG_LAUNCH
        SP_CUDA(e);
        SP_LAUNCH_CHECK();
        sp_count_launches(2);
        SP_BOUNDS_RETURN(stream);
        return SP_OK;
    }
    sp_workspace ws(stream);
    const int64_t ldt = (K + 1) & ~(int64_t)1;   // even, so rows stay 16-byte aligned
    int64_t ldt_k = ldt;                         // leading dimension of the gathered operand in the kernel
    double* Bt = ws.get<double>((size_t)n * ldt);
    if (ws.failed) return SP_ERR_ALLOC;
    dim3 tg((unsigned)sp_ceil_div(n, 32), (unsigned)sp_ceil_div(K, 32));
    k_transpose<<<tg, 256, 0, stream>>>(B, ldb, K, n, Bt, ldt);
    SP_LAUNCH_CHECK();

    sp_partition part;
    sp_status st = sp_get_merge_partition(S, items, stream, &part);
    if (st != SP_OK) return st;
    const bool vec2 = (K % 2 == 0) && (lda % 2 == 0) && (reinterpret_cast<uintptr_t>(A) % 16 == 0) &&
                      (reinterpret_cast<uintptr_t>(Bt) % 16 == 0);
    const unsigned blocks = (unsigned)sp_ceil_div(part.nchunks * 32, kSThreads);
    // The kernel keeps the operand row of the outer (segment) index in registers and gathers the
    // row of the inner index: for column-major S the two operands simply trade places
    // (segment = column j -> row j of B^T; inner coordinate = row i -> row i of A).
    if (colmajor) {
        const double* ta = A; A = Bt; Bt = const_cast<double*>(ta);
        const int64_t tl = lda; lda = ldt; ldt_k = tl;
    }
#define SP_SDDMM_LAUNCH(V)                                                                                     \
    sddmm_launch_st = sp_launch_dependent(k_sddmm<P, I, V>, dim3(blocks), dim3(kSThreads), 0, stream, pos, crd,  \
                                          (const double*)S->val, outer, (const double*)A, lda, (const double*)Bt, ldt_k, K, \
                                          x_vals, (const int64_t*)part.row, (const int64_t*)part.nz, part.nchunks,        \
                                          S->dims[S->ord[0]], S->dims[S->ord[1]])
    cudaError_t sddmm_launch_st = cudaSuccess;
    SP_DISPATCH_WIDTHS(S, {
        const P* pos = static_cast<const P*>(S->pos[1]);
        const I* crd = static_cast<const I*>(S->crd[1]);
        const I* outer = dbl ? static_cast<const I*>(S->crd[0]) : nullptr;
        if (vec2) SP_SDDMM_LAUNCH(2); else SP_SDDMM_LAUNCH(1);
    });
#undef SP_SDDMM_LAUNCH
    SP_CUDA(sddmm_launch_st);
    SP_LAUNCH_CHECK();
    sp_count_launches(2);
    SP_BOUNDS_RETURN(stream);
    return SP_OK;
}
