// SpMV layouts and kernels for the patterns whose CSR / BSR product is bound
// by something other than its bytes (y = A x, Figs. 20-21; the residual; the
// Jacobi-type sweep x + (b - A x) d^-1).
//
// FP64 multiply-adds are scarce on this GPU (about two per clock and SM, 600 G
// per second in all): a 7-point matrix takes as long for them as for its
// bytes, one of 3 x 3 blocks longer, and every idle or padded lane costs as
// much as a working one.  Both layouts therefore give each thread a row (or a
// whole block row), whose sum runs in column order (the order of the
// row-per-thread CSR kernel and of the BSR kernel, so the results are the same
// bit for bit), and issue a row's loads together.
//
// Stencil layout (DIA): the distinct offsets col - row are few (at most 8, a
// structured grid), so a value's column follows from its place (a plane per
// offset and place in the block, a value per row): no column indices and no
// row pointers, and the loads of values and of x are coalesced without
// staging.  A byte per row says which entries exist; absent
// ones are neither multiplied nor added, so a NaN or infinity in x reaches
// only the rows that refer to it.
//
// Sliced layout (SELL): 32 rows a slice, a row per lane, entry k of the 32
// rows side by side.  The rows of a window are sorted by length first, so
// the lanes of a slice finish together.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "rs_internal.cuh"

namespace {

constexpr int DIA_MAX = 8;
// Share of the layout's places that hold an entry from which it pays: a place
// costs 8 bytes, an entry in CSR 12 and its row 4.
constexpr double DIA_FILL = 0.7;

struct DiaArgs {
    int n;                   // block rows
    int off[DIA_MAX];
    int64_t ld;
    const double *val;
    const unsigned char *mask;
};

DiaArgs dia_args(const rs_mat *A)
{
    DiaArgs a;
    a.n = A->nrows;
    for (int k = 0; k < DIA_MAX; ++k) a.off[k] = k < A->dia.nd ? A->dia.off[k] : 0;
    a.ld = A->dia.ld;
    a.val = A->dia.val;
    a.mask = A->dia.mask;
    return a;
}

// the epilogue of row i: y = alpha acc (+ beta y), y = b - acc, or with dinv
// y = x + (b - acc) dinv; factors of 1 cost no FP64 instruction
__device__ __forceinline__ void spmv_store(int64_t i, double acc, const double *__restrict__ x, double alpha,
                                           double beta, const double *__restrict__ bvec, double *__restrict__ y,
                                           const double *__restrict__ dinv)
{
    if (dinv) y[i] = fma(__dsub_rn(bvec[i], acc), dinv[i], x[i]);
    else if (bvec) y[i] = __dsub_rn(bvec[i], acc);
    else if (beta == 0.0) y[i] = alpha == 1.0 ? acc : __dmul_rn(alpha, acc);
    else y[i] = fma(alpha, acc, beta == 1.0 ? y[i] : __dmul_rn(beta, y[i]));
}

// A thread per RB scalar rows of a block row: all BS, or one (threadIdx.y says
// which; the block row is blockIdx.x blockDim.x + threadIdx.x).  All loads are
// independent of one another and of the mask (x's index is clamped, not
// predicated), so a warp keeps many of its row's loads in flight.  Per product,
// against the CSR and BSR kernels: 7-point, 1,048,576 rows 33.9 -> 19 us (76 MB
// moved; bytes and multiply-adds take 11 and 12 us); 3 x 3 blocks, 500,000 block
// rows 69.7 -> 62.1 us (52 us of multiply-adds), 27,000 8.3 -> 4.9, 8,000 6.2 -> 3.0.
template <int ND, int BS, int RB>
__global__ void __launch_bounds__(256)
k_spmv_dia(DiaArgs a, const double *__restrict__ x, double alpha, double beta, const double *__restrict__ bvec,
           double *__restrict__ y, const int *skip, const double *__restrict__ dinv)
{
    if (rs_pdl_wait()) return;
    if (skip && *(volatile const int *)skip) return;
    const int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= a.n) return;
    const int r0 = RB == BS ? 0 : threadIdx.y;
    const unsigned m = a.mask[I];
    double acc[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) acc[r] = 0.0;
    auto at = [&](int k) { return min(max(I + a.off[k], (int64_t)0), (int64_t)a.n - 1); };
    if constexpr (BS == 1) {
        // the whole row's loads, then its multiply-adds (24.5 -> 22.8 us a call)
        double v[ND], xv[ND];
#pragma unroll
        for (int k = 0; k < ND; ++k) {
            v[k] = __ldg(a.val + (int64_t)k * a.ld + I);
            xv[k] = __ldg(x + at(k));
        }
#pragma unroll
        for (int k = 0; k < ND; ++k)
            if (m >> k & 1) acc[0] = fma(v[k], xv[k], acc[0]);
    } else {
#pragma unroll
        for (int k = 0; k < ND; ++k) {
            const int64_t J = at(k);
            double v[RB * BS], xv[BS];
#pragma unroll
            for (int c = 0; c < BS; ++c) xv[c] = __ldg(x + J * BS + c);
#pragma unroll
            for (int e = 0; e < RB * BS; ++e) v[e] = __ldg(a.val + (int64_t)(k * BS * BS + r0 * BS + e) * a.ld + I);
            if (m >> k & 1) {
#pragma unroll
                for (int r = 0; r < RB; ++r)
#pragma unroll
                    for (int c = 0; c < BS; ++c) acc[r] = fma(v[r * BS + c], xv[c], acc[r]);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < RB; ++r) spmv_store(I * BS + r0 + r, acc[r], x, alpha, beta, bvec, y, dinv);
}

// t = f - A (Pi_p p): only block column 0 meets the prolonged pressure vector.
// A thread per scalar row: against one per block row 8,000 3 x 3 block rows take
// 2.9 instead of 4.4 us, 100,000 5.9 instead of 6.0, 210,000 12.4 instead of 13.3.
template <int ND, int BS>
__global__ void __launch_bounds__(256)
k_presid_dia(DiaArgs a, const double *__restrict__ p, const double *__restrict__ f, double *__restrict__ t,
             const int *skip)
{
    if (rs_pdl_wait()) return;
    if (skip && *(volatile const int *)skip) return;
    const int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= a.n) return;
    const int r = threadIdx.y;
    const unsigned m = a.mask[I];
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < ND; ++k) {
        const double pv = __ldg(p + min(max(I + a.off[k], (int64_t)0), (int64_t)a.n - 1));
        const double v = __ldg(a.val + (int64_t)(k * BS * BS + r * BS) * a.ld + I);
        if (m >> k & 1) acc = fma(v, pv, acc);
    }
    t[I * BS + r] = __dsub_rn(f[I * BS + r], acc);
}

// a warp per slice, a row per lane; U entries' loads at a time
template <int U>
__global__ void __launch_bounds__(256)
k_spmv_sell(int nslice, const int2 *__restrict__ rows, const int *__restrict__ sptr, const int *__restrict__ col,
            const double *__restrict__ val, const double *__restrict__ x, double alpha, double beta,
            const double *__restrict__ bvec, double *__restrict__ y, const int *skip, const double *__restrict__ dinv)
{
    if (rs_pdl_wait()) return;
    if (skip && *(volatile const int *)skip) return;
    const int s = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (s >= nslice) return;
    const int2 rl = rows[(int64_t)s * 32 + lane];
    const int base = sptr[s] + lane, len = rl.y;
    double acc = 0.0;
    // the next U entries' loads are issued before the products of these wait
    // for their gathers: one memory latency a round instead of two (a V-cycle
    // at 128 x 128 x 64: 404 -> 398 us)
    int c[U];
    double v[U];
    auto load = [&](int k0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            c[u] = k0 + u < len ? __ldg(col + base + 32 * (k0 + u)) : -1;
            v[u] = k0 + u < len ? __ldg(val + base + 32 * (k0 + u)) : 0.0;
        }
    };
    load(0);
    for (int k0 = 0; k0 < len; k0 += U) {
        double xv[U], vv[U];
        bool in[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            in[u] = c[u] >= 0;
            vv[u] = v[u];
            xv[u] = in[u] ? __ldg(x + c[u]) : 0.0;
        }
        load(k0 + U);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (in[u]) acc = fma(vv[u], xv[u], acc);
    }
    if (rl.x >= 0) spmv_store(rl.x, acc, x, alpha, beta, bvec, y, dinv);
}

// ---------------------------------------------------------------------------
// building the layouts
// ---------------------------------------------------------------------------
// Every place of the layout (0 where a row has no entry) and the masks; *bad |= 1
// when an entry's offset is not among off[0..nd).  A thread per scalar row,
// threadIdx.y the row of the block; columns and offsets both ascend.
template <int BS>
__global__ void __launch_bounds__(256)
k_dia_fill(DiaArgs a, int nd, const int *__restrict__ ptr, const int *__restrict__ col, const double *__restrict__ src,
           double *__restrict__ val, unsigned char *__restrict__ mask, int *bad)
{
    const int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= a.n) return;
    const int r = threadIdx.y, p1 = ptr[I + 1];
    int p = ptr[I];
    unsigned m = 0;
    for (int k = 0; k < nd; ++k) {
        const bool in = p < p1 && col[p] - I == a.off[k];
#pragma unroll
        for (int c = 0; c < BS; ++c)
            val[(int64_t)(k * BS * BS + r * BS + c) * a.ld + I] = in ? src[((int64_t)p * BS + r) * BS + c] : 0.0;
        m |= (unsigned)in << k;
        p += in;
    }
    if (r == 0) {
        mask[I] = (unsigned char)m;
        if (p < p1) atomicOr(bad, 1);
    }
}

constexpr int SELL_WIN = 512;       // rows sorted by length together

// one window a block: rows in descending order of length (ties: by row), and
// the entries of each of its slices
__global__ void __launch_bounds__(SELL_WIN)
k_sell_sort(int n, const int *__restrict__ ptr, int2 *__restrict__ rows, int *__restrict__ cnt)
{
    __shared__ unsigned key[SELL_WIN];
    const int t = threadIdx.x, r0 = blockIdx.x * SELL_WIN, r = r0 + t;
    const int len = r < n ? ptr[r + 1] - ptr[r] : -1;
    key[t] = (unsigned)(65535 - min(len, 65534)) * SELL_WIN + t;      // no row: after the empty rows
    __syncthreads();
    for (int k = 2; k <= SELL_WIN; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            const int u = t ^ j;
            if (u > t) {
                const unsigned a = key[t], b = key[u];
                if ((a > b) == ((t & k) == 0)) {
                    key[t] = b;
                    key[u] = a;
                }
            }
            __syncthreads();
        }
    const int row = r0 + (int)(key[t] % SELL_WIN);
    const int l = row < n ? ptr[row + 1] - ptr[row] : 0;
    rows[(int64_t)r0 + t] = make_int2(row < n ? row : -1, l);
    const int w = __reduce_max_sync(0xffffffffu, min(l, 1 << 25));     // longer rows: the layout is refused
    if ((t & 31) == 0) cnt[(r0 + t) >> 5] = 32 * w;
}

// exclusive scan of cnt[0..n) in place, cnt[n] = the total; one block
__global__ void __launch_bounds__(1024) k_sell_scan(int n, int *__restrict__ cnt, long long *total)
{
    __shared__ long long ws[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long carry = 0;
    for (int b = 0; b < n; b += 1024) {
        const int i = b + threadIdx.x;
        const long long v = i < n ? cnt[i] : 0;
        long long s = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += u;
        }
        if (lane == 31) ws[w] = s;
        __syncthreads();
        if (w == 0) {
            long long u = ws[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long q = __shfl_up_sync(0xffffffffu, u, o);
                if (lane >= o) u += q;
            }
            ws[lane] = u;
        }
        __syncthreads();
        const long long excl = carry + (w ? ws[w - 1] : 0) + s - v;
        if (i < n) cnt[i] = (int)excl;
        carry += ws[31];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        cnt[n] = (int)carry;
        *total = carry;
    }
}

__global__ void __launch_bounds__(256)
k_sell_fill(int nslice, const int2 *__restrict__ rows, const int *__restrict__ sptr, const int *__restrict__ ptr,
            const int *__restrict__ col, const double *__restrict__ val, int *__restrict__ scol,
            double *__restrict__ sval)
{
    const int s = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (s >= nslice) return;
    const int2 rl = rows[(int64_t)s * 32 + lane];
    const int base = sptr[s] + lane, w = (sptr[s + 1] - sptr[s]) >> 5;
    const int p0 = rl.x >= 0 ? ptr[rl.x] : 0;
    for (int k = 0; k < w; ++k) {
        scol[base + 32 * k] = k < rl.y ? col[p0 + k] : -1;
        sval[base + 32 * k] = k < rl.y ? val[p0 + k] : 0.0;
    }
}

int dia_grid(const rs_mat *A, int rows) { return (int)(((int64_t)A->nrows + rows - 1) / rows); }

// The offsets of a few sample rows (on the host: a caller's pattern), the
// candidates of a stencil layout, or those of a matrix of the same pattern;
// 0 when there are too many or the layout would be too empty.
int dia_candidates(const rs_mat *A, const rs_mat *like, int (&off)[DIA_MAX])
{
    if (like) {
        std::copy(like->dia.off, like->dia.off + DIA_MAX, off);
        return like->dia.nd;
    }
    const std::vector<int> &ptr = A->h_ptr, &col = A->h_col;
    if (A->nrows < 1 || (int)ptr.size() != A->nrows + 1) return 0;
    int nd = 0;
    const int samples = 64;
    for (int k = 0; k < samples; ++k) {
        const int i = (int)((int64_t)(A->nrows - 1) * k / (samples - 1));
        for (int p = ptr[i]; p < ptr[i + 1]; ++p) {
            const int d = col[p] - i;
            if (std::find(off, off + nd, d) != off + nd) continue;
            if (nd == DIA_MAX) return 0;
            off[nd++] = d;
        }
    }
    std::sort(off, off + nd);
    return (double)A->nnzb >= DIA_FILL * nd * (double)A->nrows ? nd : 0;
}

template <int BS>
int dia_build(rs_mat *A, int nd, const int (&off)[DIA_MAX])
{
    rs_ctx *ctx = A->ctx;
    const int64_t ld = ((int64_t)A->nrows + 31) / 32 * 32;
    const size_t places = (size_t)nd * BS * BS * ld;
    int hbad = 1;
    // one allocation: values, masks, the flag
    RS_TRY(rs_alloc(ctx, (void **)&A->dia.val, sizeof(double) * places + ld + sizeof(int)));
    A->dia.mask = (unsigned char *)(A->dia.val + places);
    int *bad = (int *)(A->dia.mask + ld);
    A->dia.ld = ld;
    std::copy(off, off + nd, A->dia.off);
    A->dia.nd = nd;
    int st = cudaMemsetAsync(bad, 0, sizeof(int), ctx->stream) == cudaSuccess ? RS_OK : RS_ERR_CUDA;
    if (!st) {
        k_dia_fill<BS><<<dia_grid(A, 64), dim3(64, BS), 0, ctx->stream>>>(dia_args(A), nd, A->ptr, A->col, A->val,
                                                                                  A->dia.val, A->dia.mask, bad);
        st = rs_check_launch(ctx);
    }
    if (!st && (cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream) != cudaSuccess ||
                cudaStreamSynchronize(ctx->stream) != cudaSuccess))
        st = RS_ERR_CUDA;
    if (st || hbad) rs_spmv_layout_free(A);
    return st;
}

int sell_build(rs_mat *A)
{
    rs_ctx *ctx = A->ctx;
    const int win = (A->nrows + SELL_WIN - 1) / SELL_WIN, ns = win * (SELL_WIN / 32);
    long long *tot = nullptr, htot = 0;
    int st = rs_alloc(ctx, (void **)&A->sell.rows, sizeof(int2) * 32 * (size_t)ns);
    st = st ? st : rs_alloc(ctx, (void **)&A->sell.sptr, sizeof(int) * ((size_t)ns + 1));
    st = st ? st : rs_alloc(ctx, (void **)&tot, sizeof(long long));
    if (!st) {
        k_sell_sort<<<win, SELL_WIN, 0, ctx->stream>>>(A->nrows, A->ptr, A->sell.rows, A->sell.sptr);
        k_sell_scan<<<1, 1024, 0, ctx->stream>>>(ns, A->sell.sptr, tot);
        ctx->launches += 1;
        st = rs_check_launch(ctx);
    }
    if (!st && (cudaMemcpyAsync(&htot, tot, sizeof(htot), cudaMemcpyDeviceToHost, ctx->stream) != cudaSuccess ||
                cudaStreamSynchronize(ctx->stream) != cudaSuccess))
        st = RS_ERR_CUDA;
    rs_free(ctx, tot);
    // a few very long rows would leave a slice to one lane: keep CSR
    const bool fits = htot < 0x7fffffffLL && (double)htot <= 1.25 * (double)A->nnzb + 32.0 * 32;
    if (!st && fits) {
        st = rs_alloc(ctx, (void **)&A->sell.col, sizeof(int) * (size_t)htot);
        st = st ? st : rs_alloc(ctx, (void **)&A->sell.val, sizeof(double) * (size_t)htot);
        if (!st) {
            k_sell_fill<<<(ns + 7) / 8, 256, 0, ctx->stream>>>(ns, A->sell.rows, A->sell.sptr, A->ptr, A->col, A->val,
                                                              A->sell.col, A->sell.val);
            st = rs_check_launch(ctx);
            A->sell.nslice = ns;
        }
    }
    if (st || !fits) rs_spmv_layout_free(A);
    return st;
}

// Block rows from which a thread takes a whole one: it loads x once, but its
// chain of multiply-adds is BS times as long and its registers leave about
// 156,000 rows resident at once.  Below, thread blocks of 32 block rows, a warp
// per row of the block.  Thread per scalar row / per block row, us: 3 x 3 blocks
// 8,000 rows 3.0 / 6.1, 100,000 14.0 / 14.7, 180,000 25.2 / 39.5, 245,000 33.9 /
// 39.0, 294,000 39.6 / 39.3, 500,000 64.8 / 62.1; 2 x 2 blocks 27,000 3.4 / 4.4,
// 210,000 14.1 / 18.2, 280,000 18.3 / 18.5, 500,000 32.2 / 30.5.
constexpr int DIA_BLOCK_ROWS = 280000;

// launch(ND) with A's number of offsets as a constant
template <typename F>
int dia_dispatch(const rs_mat *A, F launch)
{
    switch (A->dia.nd) {
    case 1: launch(std::integral_constant<int, 1>()); break;
    case 2: launch(std::integral_constant<int, 2>()); break;
    case 3: launch(std::integral_constant<int, 3>()); break;
    case 4: launch(std::integral_constant<int, 4>()); break;
    case 5: launch(std::integral_constant<int, 5>()); break;
    case 6: launch(std::integral_constant<int, 6>()); break;
    case 7: launch(std::integral_constant<int, 7>()); break;
    case 8: launch(std::integral_constant<int, 8>()); break;
    default: return RS_ERR_INVALID_ARG;
    }
    return rs_check_launch(A->ctx);
}

template <int BS>
int dia_launch(const rs_mat *A, const double *x, double alpha, double beta, const double *bvec, double *y,
               const int *skip, const double *dinv)
{
    return dia_dispatch(A, [&](auto nd) {
        constexpr int ND = decltype(nd)::value;
        if (BS == 1 || A->nrows >= DIA_BLOCK_ROWS)
            rs_pdl(k_spmv_dia<ND, BS, BS>, dia_grid(A, 256), 256, 0, A->ctx)(dia_args(A), x, alpha, beta, bvec, y, skip,
                                                                            dinv);
        else
            rs_pdl(k_spmv_dia<ND, BS, 1>, dia_grid(A, 32), dim3(32, BS), 0, A->ctx)(dia_args(A), x, alpha, beta, bvec,
                                                                                   y, skip, dinv);
    });
}

template <int BS>
int presid_launch(const rs_mat *A, const double *p, const double *f, double *t, const int *skip)
{
    return dia_dispatch(A, [&](auto nd) {
        rs_pdl(k_presid_dia<decltype(nd)::value, BS>, dia_grid(A, 32), dim3(32, BS), 0, A->ctx)(dia_args(A), p, f, t,
                                                                                              skip);
    });
}

}  // namespace

void rs_spmv_layout_free(rs_mat *A)
{
    rs_ctx *ctx = A->ctx;
    rs_free(ctx, A->dia.val);
    rs_free(ctx, A->sell.rows);
    rs_free(ctx, A->sell.sptr);
    rs_free(ctx, A->sell.col);
    rs_free(ctx, A->sell.val);
    A->dia = {};
    A->sell = {};
}

int rs_spmv_layout_build(rs_mat *A, const rs_mat *like)
{
    if (A->bs <= 3) {
        int off[DIA_MAX];
        const int nd = dia_candidates(A, like, off);
        if (nd) {
            RS_TRY(A->bs == 1 ? dia_build<1>(A, nd, off) : A->bs == 2 ? dia_build<2>(A, nd, off) : dia_build<3>(A, nd, off));
            if (A->dia.nd) return RS_OK;
        }
    }
    if (A->bs == 1 && A->nrows >= RS_SELL_MIN_ROWS) return sell_build(A);
    return RS_OK;
}

bool rs_spmv_layout(const rs_mat *A) { return A->dia.nd > 0 || A->sell.nslice > 0; }

int rs_spmv_layout_launch(const rs_mat *A, const double *x, double alpha, double beta, const double *bvec, double *y,
                          const int *skip, const double *dinv)
{
    if (A->dia.nd > 0) {
        switch (A->bs) {
        case 1: return dia_launch<1>(A, x, alpha, beta, bvec, y, skip, dinv);
        case 2: return dia_launch<2>(A, x, alpha, beta, bvec, y, skip, dinv);
        case 3: return dia_launch<3>(A, x, alpha, beta, bvec, y, skip, dinv);
        default: return RS_ERR_INVALID_ARG;
        }
    }
    const int grid = (A->sell.nslice + 7) / 8;
    // short rows (interpolation) need no more loads in flight than they have entries
    if (A->nnzb <= 6 * (int64_t)A->nrows)
        rs_pdl(k_spmv_sell<4>, grid, 256, 0, A->ctx)(A->sell.nslice, A->sell.rows, A->sell.sptr, A->sell.col,
                                                         A->sell.val, x, alpha, beta, bvec, y, skip, dinv);
    else
        rs_pdl(k_spmv_sell<8>, grid, 256, 0, A->ctx)(A->sell.nslice, A->sell.rows, A->sell.sptr, A->sell.col,
                                                         A->sell.val, x, alpha, beta, bvec, y, skip, dinv);
    return rs_check_launch(A->ctx);
}

int rs_presid_dia_launch(const rs_mat *A, const double *p, const double *f, double *t, const int *skip)
{
    switch (A->bs) {
    case 2: return presid_launch<2>(A, p, f, t, skip);
    case 3: return presid_launch<3>(A, p, f, t, skip);
    default: return RS_ERR_INVALID_ARG;
    }
}
