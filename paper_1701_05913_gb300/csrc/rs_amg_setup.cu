// The AMG setup (Alg. 3) on the GPU, level by level:
//   1. strength: j strongly influences i when j != i and
//      -a_ij >= theta max_{k != i} (-a_ik), and its transpose;
//   2. C/F splitting by PMIS (De Sterck, Yang and Heys 2006, one of the
//      coarsenings Sec. 4.2 names): lambda_i = |S_i^T| + w_i with w_i from a
//      counter-based SplitMix64 keyed by (level, i); points that influence no
//      point are F; then in rounds every undecided point whose measure exceeds
//      that of every undecided point of S_i and S_i^T becomes C and every
//      undecided point that strongly depends on a C point becomes F;
//   3. direct interpolation (as in Sec. 4.2's classical AMG);
//   4. R = P^T;  5. A_{l+1} = R (A_l P) (Eq. 4);
// then the smoother's diagonal and the coarsest level's dense inverse.
//
// Arithmetic follows the definitions term by term in the same order as a
// sequential reading, each product and sum rounded once (no contraction):
// the strength, splitting and patterns are exact, and a Galerkin entry is the
// sum of its products in the order (row entry of the left factor, row entry
// of the right factor), so the coarse matrices come out bit for bit the same
// as a sequential row-by-row product.  Host work is sizes and allocation.
#include <algorithm>
#include <vector>

#include "rs_internal.cuh"

namespace {

constexpr int SG_CAP = 2048;     // candidate terms of one row of a product

// ---------------------------------------------------------------------------
// exclusive prefix sums of int counts (out[n] = total)
// ---------------------------------------------------------------------------
constexpr int SCAN_T = 1024;

__device__ __forceinline__ int block_excl_scan(int v, int *sh, int *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int s = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        sh[lane] = s;
    }
    __syncthreads();
    const int before = wid ? sh[wid - 1] : 0;
    *total = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    return before + x - v;
}

__global__ void __launch_bounds__(SCAN_T) k_scan_blocks(int n, const int *__restrict__ in, int *__restrict__ out,
                                                        int *__restrict__ bsum)
{
    __shared__ int sh[32];
    const int i = blockIdx.x * SCAN_T + threadIdx.x;
    int tot;
    const int e = block_excl_scan(i < n ? in[i] : 0, sh, &tot);
    if (i < n) out[i] = e;
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

// one block: exclusive scan of n values (out may be in); the sum in *total and,
// where end is given, *end
__global__ void __launch_bounds__(SCAN_T) k_scan_top(int n, const int *in, int *out, int *__restrict__ total,
                                                     int *__restrict__ end)
{
    __shared__ int sh[32];
    int carry = 0;
    for (int b0 = 0; b0 < n; b0 += SCAN_T) {
        const int i = b0 + threadIdx.x;
        int tot;
        const int v = i < n ? in[i] : 0;
        const int e = block_excl_scan(v, sh, &tot);
        if (i < n) out[i] = carry + e;
        carry += tot;
    }
    if (threadIdx.x == 0) {
        *total = carry;
        if (end) *end = carry;
    }
}

__global__ void __launch_bounds__(SCAN_T) k_scan_add(int n, int *__restrict__ out, const int *__restrict__ bsum,
                                                     const int *__restrict__ total)
{
    const int i = blockIdx.x * SCAN_T + threadIdx.x;
    if (i < n) out[i] += bsum[blockIdx.x];
    if (i == 0) out[n] = *total;
}

// ---------------------------------------------------------------------------
// 1. strength and its transpose
// ---------------------------------------------------------------------------
// The kernels below go over a row's entries.  What bounds them is the latency
// of a row's loads (a coarse level has a few rows of 30 to 60 entries and
// cannot fill the chip), so the loads of ROW_U entries are issued before the
// first is used, with clamped indices instead of predicates, and nothing is
// looked up twice: the strength threshold is kept per row instead of found by
// searching S.  128 x 128 x 64 hierarchy: strength 713 -> 380 us, interpolation
// 1486 -> 565 us, sorting the rows of the transposes 327 -> 73 us.
constexpr int ROW_U = 8;

// body(p, col, val) for the entries p of [s, e) in order
template <typename F>
__device__ __forceinline__ void each_entry(int s, int e, const int *__restrict__ col, const double *__restrict__ val,
                                           F body)
{
    for (int p0 = s; p0 < e; p0 += ROW_U) {
        int c[ROW_U];
        double v[ROW_U];
#pragma unroll
        for (int u = 0; u < ROW_U; ++u) {
            const int p = min(p0 + u, e - 1);
            c[u] = col[p];
            v[u] = val[p];
        }
#pragma unroll
        for (int u = 0; u < ROW_U; ++u)
            if (p0 + u < e) body(c[u], v[u]);
    }
}

// th[i]: entries with -a_ij >= th[i], j != i, are strong (none when infinite:
// the row has no negative off-diagonal entry); cnt[i] = |S_i|
__global__ void k_strength_count(int n, const int *__restrict__ ptr, const int *__restrict__ col,
                                 const double *__restrict__ val, double theta, double *__restrict__ th,
                                 int *__restrict__ cnt)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int s = ptr[i], e = ptr[i + 1];
        double mx = 0.0;
        each_entry(s, e, col, val, [&](int c, double v) { mx = c != i && -v > mx ? -v : mx; });
        const double t = mx > 0.0 ? __dmul_rn(theta, mx) : (double)INFINITY;
        int k = 0;
        if (mx > 0.0) each_entry(s, e, col, val, [&](int c, double v) { k += c != i && -v >= t; });
        th[i] = t;
        cnt[i] = k;
    }
}

__global__ void k_strength_fill(int n, const int *__restrict__ ptr, const int *__restrict__ col,
                                const double *__restrict__ val, const double *__restrict__ th,
                                const int *__restrict__ sptr, int *__restrict__ scol)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double t = th[i];
        int k = sptr[i];
        each_entry(ptr[i], ptr[i + 1], col, val, [&](int c, double v) {
            if (c != i && -v >= t) scol[k++] = c;
        });
    }
}

__global__ void k_count_cols(int64_t nnz, const int *__restrict__ col, int *__restrict__ cnt)
{
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&cnt[col[p]], 1);
}

// transpose fill: entries land at an atomic slot of their column; values
// optional; rows of the transpose are sorted afterwards where it has values
__global__ void k_transpose_fill(int n, const int *__restrict__ ptr, const int *__restrict__ col,
                                 const double *__restrict__ val, int *__restrict__ fill, int *__restrict__ tcol,
                                 double *__restrict__ tval)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        for (int p = ptr[i]; p < ptr[i + 1]; ++p) {
            const int q = atomicAdd(&fill[col[p]], 1);
            tcol[q] = i;
            if (tval) tval[q] = val[p];
        }
}

// rows by column into (col, val): SORT_L lanes a row, an entry's place is the
// number of the row's columns below its own (no column occurs twice)
constexpr int SORT_L = 8;
__global__ void k_sort_rows(int n, const int *__restrict__ ptr, const int *__restrict__ ucol,
                            const double *__restrict__ uval, int *__restrict__ col, double *__restrict__ val)
{
    const int lane = threadIdx.x % SORT_L;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) / SORT_L; i < n; i += gridDim.x * blockDim.x / SORT_L) {
        const int s = ptr[i], e = ptr[i + 1];
        for (int a = s + lane; a < e; a += SORT_L) {
            const int c = ucol[a];
            int k = 0;
#pragma unroll 8
            for (int b = s; b < e; ++b) k += ucol[b] < c;
            col[s + k] = c;
            val[s + k] = uval[a];
        }
    }
}

// ---------------------------------------------------------------------------
// 2. PMIS
// ---------------------------------------------------------------------------
// SplitMix64 (Steele, Lea and Flood 2014), counter-based: the k-th output of
// the generator started from state 0
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long k)
{
    unsigned long long z = (k + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void k_pmis_init(int n, const int *__restrict__ tptr, int level, double *__restrict__ lam,
                            char *__restrict__ st, int *__restrict__ und)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int t = tptr[i + 1] - tptr[i];
        const unsigned long long k = ((unsigned long long)(unsigned)level << 32) | (unsigned)i;
        const double w = (double)(splitmix64(k) >> 11) * 0x1.0p-53;
        lam[i] = __dadd_rn((double)t, w);
        st[i] = t == 0 ? 2 : 0;
        if (t != 0) atomicAdd(und, 1);
    }
}

// undecided points that are the strict maximum of their undecided
// neighbourhood (states of the round's start: old) become C
__global__ void k_pmis_select(int n, const int *__restrict__ sptr, const int *__restrict__ scol,
                              const int *__restrict__ tptr, const int *__restrict__ tcol,
                              const double *__restrict__ lam, const char *__restrict__ old, char *__restrict__ st)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (old[i] != 0) continue;
        const double li = lam[i];
        bool top = true;
        auto look = [&](int s, int e, const int *__restrict__ nb) {
            for (int q0 = s; q0 < e && top; q0 += ROW_U) {
                int c[ROW_U];
#pragma unroll
                for (int u = 0; u < ROW_U; ++u) c[u] = nb[min(q0 + u, e - 1)];
#pragma unroll
                for (int u = 0; u < ROW_U; ++u) top = top & !((old[c[u]] == 0) & !(li > lam[c[u]]));
            }
        };
        look(sptr[i], sptr[i + 1], scol);
        look(tptr[i], tptr[i + 1], tcol);
        if (top) st[i] = 1;
    }
}

// undecided points that depend strongly on a C point become F; count the rest
__global__ void k_pmis_f(int n, const int *__restrict__ sptr, const int *__restrict__ scol, char *__restrict__ st,
                         int *__restrict__ und)
{
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        if (st[j] != 0) continue;
        bool f = false;
        const int s = sptr[j], e = sptr[j + 1];
        for (int q0 = s; q0 < e && !f; q0 += ROW_U) {
            int c[ROW_U];
#pragma unroll
            for (int u = 0; u < ROW_U; ++u) c[u] = scol[min(q0 + u, e - 1)];
#pragma unroll
            for (int u = 0; u < ROW_U; ++u) f = f | (st[c[u]] == 1);
        }
        if (f) st[j] = 2;
        else atomicAdd(und, 1);
    }
}

__global__ void k_cflag(int n, const char *__restrict__ st, int *__restrict__ flag)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) flag[i] = st[i] == 1;
}

__global__ void k_cidx(int n, const char *__restrict__ st, const int *__restrict__ scan, int *__restrict__ cidx)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        cidx[i] = st[i] == 1 ? scan[i] : -1;
}

// ---------------------------------------------------------------------------
// 3. direct interpolation: C points inject; an F point interpolates from
// its strong C neighbours k with w_ik = -alpha a_ik / d (a_ik < 0) or
// -beta a_ik / d (a_ik > 0), alpha (beta) = the row's sum of negative
// (positive) off-diagonal entries over that of its strong C neighbours,
// d = a_ii, plus the positive couplings when no strong C coupling is positive
// ---------------------------------------------------------------------------
__global__ void k_interp_count(int n, const int *__restrict__ sptr, const int *__restrict__ scol,
                               const int *__restrict__ cidx, int *__restrict__ cnt)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int k = 1;
        if (cidx[i] < 0) {
            k = 0;
#pragma unroll 4
            for (int r = sptr[i]; r < sptr[i + 1]; ++r) k += cidx[scol[r]] >= 0;
        }
        cnt[i] = k;
    }
}

// the strong C couplings go to pval as they are met and become weights once
// the row's sums are known
__global__ void k_interp_fill(int n, const int *__restrict__ ptr, const int *__restrict__ col,
                              const double *__restrict__ val, const double *__restrict__ th,
                              const int *__restrict__ cidx, const int *__restrict__ pptr, int *__restrict__ pcol,
                              double *__restrict__ pval)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int k0 = pptr[i], ci = cidx[i];
        if (ci >= 0) {
            pcol[k0] = ci;
            pval[k0] = 1.0;
            continue;
        }
        const double t = th[i];
        const int s = ptr[i], e = ptr[i + 1];
        double aii = 0.0, neg = 0.0, pos = 0.0, negc = 0.0, posc = 0.0;
        int k = k0;
        for (int p0 = s; p0 < e; p0 += ROW_U) {
            int c[ROW_U], cc[ROW_U];
            double v[ROW_U];
#pragma unroll
            for (int u = 0; u < ROW_U; ++u) {
                const int p = min(p0 + u, e - 1);
                c[u] = col[p];
                v[u] = val[p];
            }
#pragma unroll
            for (int u = 0; u < ROW_U; ++u) cc[u] = cidx[c[u]];
#pragma unroll
            for (int u = 0; u < ROW_U; ++u) {
                if (p0 + u >= e) continue;
                if (c[u] == i) {
                    aii = v[u];
                    continue;
                }
                const bool strong_c = cc[u] >= 0 && -v[u] >= t;
                if (v[u] < 0.0) {
                    neg = __dadd_rn(neg, v[u]);
                    if (strong_c) negc = __dadd_rn(negc, v[u]);
                } else {
                    pos = __dadd_rn(pos, v[u]);
                    if (strong_c) posc = __dadd_rn(posc, v[u]);
                }
                if (strong_c) {
                    pcol[k] = cc[u];
                    pval[k++] = v[u];
                }
            }
        }
        double diag = aii, beta = 0.0;
        if (posc == 0.0) diag = __dadd_rn(diag, pos);
        else beta = __ddiv_rn(pos, posc);
        const double alpha = negc != 0.0 ? __ddiv_rn(neg, negc) : 0.0;
        for (int q = k0; q < k; ++q) {
            const double v = pval[q];
            pval[q] = __ddiv_rn(__dmul_rn(-(v < 0.0 ? alpha : beta), v), diag);
        }
    }
}

// ---------------------------------------------------------------------------
// 5. sparse products C = A B, a warp per row.  The row's candidate terms
// (entry p of A's row, entry q of B's row p) are numbered in that order; a
// column of the result is the sum of its terms in number order.  Rows are
// taken by class of their number of terms, one launch per class that occurs,
// so that a row's scratch is a few KB and not the largest row's: up to 32
// terms stay in registers, one per lane; longer rows go through a hash table
// of their columns in shared memory, 32 terms at a time.
//
// What bounds it: the chain of dependent loads of a row (A's entries, B's row
// pointers, B's entries), so the rate is rows in flight.  With one sort of
// 2048 slots (32 KB) per warp for every row, four rows in flight per SM, the
// 14 products of a 128 x 128 x 64 hierarchy took 48 ms of the setup's 77.2;
// the products now take 2.7 ms.
// ---------------------------------------------------------------------------
constexpr int SG_CLASSES = 4;
__host__ __device__ constexpr int sg_hi(int c) { return c == 0 ? 32 : c == 1 ? 128 : c == 2 ? 512 : SG_CAP; }
// shared memory of one warp: table of 2 hi columns and sums, the distinct
// columns and their slots
constexpr size_t sg_warp_smem(int c)
{
    return c == 0 ? 0 : (size_t)sg_hi(c) * (2 * (sizeof(double) + sizeof(int)) + 2 * sizeof(int));
}
// 16 to 64 KB a block: up to 48 warps per SM for rows of up to 128 terms, 12
// for up to 512, 3 beyond
constexpr int sg_warps(int c) { return c < 2 ? 4 : c == 2 ? 2 : 1; }

// terms of every row, the rows in each class (cls[0..3]) and those with more
// than SG_CAP terms (cls[4])
__global__ void k_sg_len(int n, const int *__restrict__ aptr, const int *__restrict__ acol,
                         const int *__restrict__ bptr, int *__restrict__ len, int *__restrict__ cls)
{
    __shared__ int sc[SG_CLASSES + 1];
    if (threadIdx.x <= SG_CLASSES) sc[threadIdx.x] = 0;
    __syncthreads();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int64_t m = 0;
        for (int p = aptr[i]; p < aptr[i + 1]; ++p) m += bptr[acol[p] + 1] - bptr[acol[p]];
        const int c = m <= sg_hi(0) ? 0 : m <= sg_hi(1) ? 1 : m <= sg_hi(2) ? 2 : m <= sg_hi(3) ? 3 : 4;
        len[i] = c < SG_CLASSES ? (int)m : SG_CAP + 1;
        atomicAdd(&sc[c], 1);
    }
    __syncthreads();
    if (threadIdx.x <= SG_CLASSES && sc[threadIdx.x]) atomicAdd(&cls[threadIdx.x], sc[threadIdx.x]);
}

// the number of lanes whose (non-decreasing) value is <= t, at most 31
__device__ __forceinline__ int sg_find(int inc, int t)
{
    int pos = 0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1)
        if (__shfl_sync(0xffffffffu, inc, pos + s - 1) <= t) pos += s;
    return pos;
}

// 32 consecutive entries of A's row, one per lane: value, first entry of B's
// row, and the inclusive scan of those rows' lengths
struct SgChunk {
    double a;
    int q0, m, inc, total;
};
template <bool FILL>
__device__ __forceinline__ SgChunk sg_chunk(int p, int pe, int lane, const int *__restrict__ acol,
                                            const double *__restrict__ aval, const int *__restrict__ bptr)
{
    SgChunk k;
    k.a = 0.0;
    k.q0 = k.m = 0;
    if (p + lane < pe) {
        const int j = acol[p + lane];
        if (FILL) k.a = aval[p + lane];
        k.q0 = bptr[j];
        k.m = bptr[j + 1] - k.q0;
    }
    k.inc = k.m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, k.inc, o);
        if (lane >= o) k.inc += y;
    }
    k.total = __shfl_sync(0xffffffffu, k.inc, 31);
    return k;
}

// term t of a chunk (a lane's own t; every lane calls): its column and product
template <bool FILL>
__device__ __forceinline__ void sg_term(const SgChunk &k, int t, bool in, const int *__restrict__ bcol,
                                        const double *__restrict__ bval, int &c, double &v)
{
    const int pos = sg_find(k.inc, t);
    const int q = __shfl_sync(0xffffffffu, k.q0 + k.m - k.inc, pos) + t;
    const double a = FILL ? __shfl_sync(0xffffffffu, k.a, pos) : 0.0;
    if (in) {
        c = bcol[q];
        if (FILL) v = __dmul_rn(a, bval[q]);
    }
}

// s plus the values v of the lanes in mask, in lane order (every lane calls;
// mask 0: s as it is)
__device__ __forceinline__ double sg_sum(double s, double v, unsigned mask, int lane)
{
    while (__any_sync(0xffffffffu, mask != 0)) {
        const double x = __shfl_sync(0xffffffffu, v, mask ? __ffs(mask) - 1 : lane);
        if (mask) {
            s = __dadd_rn(s, x);
            mask &= mask - 1;
        }
    }
    return s;
}

// Count pass (FILL false): out[i] = the distinct columns of row i; fill pass:
// columns (ascending) and sums from cptr[i].  A warp takes `chunk` (<= 32)
// consecutive rows at a time and of these the rows of class cls.
template <bool FILL>
__global__ void __launch_bounds__(128)
k_spgemm(int n, int cls, int chunk, const int *__restrict__ len, const int *__restrict__ aptr,
         const int *__restrict__ acol, const double *__restrict__ aval, const int *__restrict__ bptr,
         const int *__restrict__ bcol, const double *__restrict__ bval, const int *__restrict__ cptr,
         int *__restrict__ out, double *__restrict__ cval)
{
    extern __shared__ __align__(16) unsigned char sg_smem[];
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int hi = sg_hi(cls), lo = cls ? sg_hi(cls - 1) : -1;
    // all warps' sums, then all tables, distinct columns and slots
    double *tsum = (double *)sg_smem + (size_t)wid * 2 * hi;
    int *ibase = (int *)(sg_smem + (size_t)nw * 2 * hi * sizeof(double));
    int *tcol = ibase + (size_t)wid * 2 * hi;
    int *dc = ibase + (size_t)nw * 2 * hi + (size_t)wid * hi;
    int *dl = ibase + (size_t)nw * 3 * hi + (size_t)wid * hi;
    const unsigned lt = (1u << lane) - 1;
    for (int64_t b0 = ((int64_t)blockIdx.x * nw + wid) * chunk; b0 < n; b0 += (int64_t)gridDim.x * nw * chunk) {
        const int myl = lane < chunk && b0 + lane < n ? len[b0 + lane] : SG_CAP + 2;
        for (unsigned todo = __ballot_sync(FULL, myl > lo && myl <= hi); todo; todo &= todo - 1) {
            const int r = __ffs(todo) - 1, i = (int)b0 + r;
            const int rowlen = __shfl_sync(FULL, myl, r);
            const int p0 = aptr[i], pe = aptr[i + 1];
            const int o0 = FILL ? cptr[i] : 0;
            if (cls == 0) {
                // one term per lane
                int c = -1, base = 0;
                double v = 0.0;
                for (int p = p0; p < pe; p += 32) {
                    const SgChunk k = sg_chunk<FILL>(p, pe, lane, acol, aval, bptr);
                    const int t = lane - base;
                    sg_term<FILL>(k, t, t >= 0 && t < k.total, bcol, bval, c, v);
                    base += k.total;
                }
                const bool in = lane < rowlen;
                unsigned same = __match_any_sync(FULL, c);
                const bool first = in && __ffs(same) - 1 == lane;
                const unsigned firsts = __ballot_sync(FULL, first);
                if (!FILL) {
                    if (lane == 0) out[i] = __popc(firsts);
                    continue;
                }
                const double s = sg_sum(0.0, v, first ? same : 0u, lane);
                int rank = 0;
                for (unsigned f = firsts; f; f &= f - 1) rank += __shfl_sync(FULL, c, __ffs(f) - 1) < c;
                if (first) {
                    out[o0 + rank] = c;
                    cval[o0 + rank] = s;
                }
                continue;
            }
            // 32 terms at a time through the row's hash table of columns
            const int lg = 32 - __clz(2 * rowlen - 1);      // table: the power of two >= 2 rowlen (<= 2 hi)
            const int tsz = 1 << lg;
            for (int k = lane; k < tsz; k += 32) tcol[k] = -1;
            __syncwarp();
            int nd = 0;
            for (int p = p0; p < pe; p += 32) {
                const SgChunk k = sg_chunk<FILL>(p, pe, lane, acol, aval, bptr);
                for (int t0 = 0; t0 < k.total; t0 += 32) {
                    const bool in = t0 + lane < k.total;
                    int c = -1;
                    double v = 0.0;
                    sg_term<FILL>(k, t0 + lane, in, bcol, bval, c, v);
                    // the first lane of each column finds or claims its slot;
                    // the claiming lanes have different columns
                    const unsigned same = __match_any_sync(FULL, c);
                    const bool first = in && __ffs(same) - 1 == lane;
                    bool fresh = false;
                    int h = 0;
                    if (first) {
                        h = (int)(((unsigned)c * 2654435761u) >> (32 - lg));
                        for (;;) {
                            const int cur = atomicCAS(&tcol[h], -1, c);
                            fresh = cur == -1;
                            if (fresh || cur == c) break;
                            h = (h + 1) & (tsz - 1);
                        }
                    }
                    if (FILL) {
                        const double s = sg_sum(first && !fresh ? tsum[h] : 0.0, v, first ? same : 0u, lane);
                        if (first) tsum[h] = s;
                    }
                    const unsigned nm = __ballot_sync(FULL, fresh);
                    if (FILL && fresh) {
                        const int k2 = nd + __popc(nm & lt);
                        dc[k2] = c;
                        dl[k2] = h;
                    }
                    nd += __popc(nm);
                    __syncwarp();
                }
            }
            if (!FILL) {
                if (lane == 0) out[i] = nd;
                __syncwarp();
                continue;
            }
            if (nd <= 128) {
                // a column's place: the number of smaller ones
                int ck[4], rk[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    ck[u] = lane + 32 * u < nd ? dc[lane + 32 * u] : 0x7fffffff;
                    rk[u] = 0;
                }
                for (int j = 0; j < nd; ++j) {
                    const int cj = dc[j];
#pragma unroll
                    for (int u = 0; u < 4; ++u) rk[u] += cj < ck[u];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (lane + 32 * u < nd) {
                        out[o0 + rk[u]] = ck[u];
                        cval[o0 + rk[u]] = tsum[dl[lane + 32 * u]];
                    }
            } else {
                // bitonic sort of (column, slot); a power of two >= nd fits (nd <= hi)
                int sz = 256;
                while (sz < nd) sz <<= 1;
                for (int k = nd + lane; k < sz; k += 32) dc[k] = 0x7fffffff;
                __syncwarp();
                for (int k = 2; k <= sz; k <<= 1)
                    for (int j = k >> 1; j > 0; j >>= 1) {
                        for (int t = lane; t < sz; t += 32) {
                            const int u = t ^ j;
                            if (u > t) {
                                const int ct = dc[t], cu = dc[u];
                                if ((ct > cu) == ((t & k) == 0) && ct != cu) {
                                    dc[t] = cu;
                                    dc[u] = ct;
                                    const int x = dl[t];
                                    dl[t] = dl[u];
                                    dl[u] = x;
                                }
                            }
                        }
                        __syncwarp();
                    }
                for (int k = lane; k < nd; k += 32) {
                    out[o0 + k] = dc[k];
                    cval[o0 + k] = tsum[dl[k]];
                }
            }
            __syncwarp();
        }
    }
}

// ---------------------------------------------------------------------------
// smoother diagonal, zero-diagonal check, coarsest dense inverse
// ---------------------------------------------------------------------------
// dinv_i = 1 / sum_j |a_ij|; *bad |= 1 when a diagonal entry is 0 (needed by
// hybrid Gauss-Seidel)
__global__ void k_amg_l1(int n, const int *__restrict__ ptr, const int *__restrict__ col,
                         const double *__restrict__ val, double *__restrict__ dinv, int *__restrict__ bad)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double s = 0.0, dg = 0.0;
        each_entry(ptr[i], ptr[i + 1], col, val, [&](int c, double v) {
            s = __dadd_rn(s, fabs(v));
            dg = c == i ? v : dg;
        });
        dinv[i] = __ddiv_rn(1.0, s);
        if (dg == 0.0) atomicOr(bad, 1);
    }
}

// the coarsest matrix into [A | I] (n x 2n, row-major)
__global__ void k_dense_aug(int n, const int *__restrict__ ptr, const int *__restrict__ col,
                            const double *__restrict__ val, double *__restrict__ m)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)n * 2 * n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / (2 * n)), c = (int)(e - (int64_t)r * 2 * n);
        m[e] = c >= n ? (c - n == r ? 1.0 : 0.0) : 0.0;
    }
}
__global__ void k_dense_scatter(int n, const int *__restrict__ ptr, const int *__restrict__ col,
                                const double *__restrict__ val, double *__restrict__ m)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        for (int p = ptr[i]; p < ptr[i + 1]; ++p) m[(size_t)i * 2 * n + col[p]] = val[p];
}

// Gauss-Jordan with partial pivoting, column c: one block finds the pivot
// (largest |m_rc|, r >= c, lowest row on ties), swaps it into row c and
// divides row c by it; *bad |= 1 on a zero or non-finite pivot
__global__ void __launch_bounds__(256) k_gj_pivot(int n, int c, double *__restrict__ m, int *__restrict__ bad)
{
    __shared__ double bv[256];
    __shared__ int br[256];
    const int w = 2 * n;
    double best = -1.0;
    int row = c;
    for (int r = c + threadIdx.x; r < n; r += blockDim.x) {
        const double a = fabs(m[(size_t)r * w + c]);
        if (a > best) {
            best = a;
            row = r;
        }
    }
    bv[threadIdx.x] = best;
    br[threadIdx.x] = row;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            const double o = bv[threadIdx.x + s];
            const int orow = br[threadIdx.x + s];
            if (o > bv[threadIdx.x] || (o == bv[threadIdx.x] && orow < br[threadIdx.x])) {
                bv[threadIdx.x] = o;
                br[threadIdx.x] = orow;
            }
        }
        __syncthreads();
    }
    const int p = br[0];
    const double piv = m[(size_t)p * w + c];
    __syncthreads();         // every thread has the pivot before row p changes
    if (!(piv != 0.0) || !isfinite(piv)) {
        if (threadIdx.x == 0) atomicOr(bad, 1);
        return;
    }
    for (int j = threadIdx.x; j < w; j += blockDim.x) {
        const double a = m[(size_t)p * w + j], b = m[(size_t)c * w + j];
        m[(size_t)c * w + j] = __ddiv_rn(a, piv);
        if (p != c) m[(size_t)p * w + j] = b;
    }
}

// rows r != c: m_r -= m_rc m_c (m_rc read before the row changes)
__global__ void k_gj_elim(int n, int c, double *__restrict__ m, const int *__restrict__ bad)
{
    if (*bad) return;
    const int w = 2 * n;
    for (int r = blockIdx.x; r < n; r += gridDim.x) {
        if (r == c) continue;
        const double f = m[(size_t)r * w + c];
        __syncthreads();
        if (f != 0.0)
            for (int j = threadIdx.x; j < w; j += blockDim.x)
                m[(size_t)r * w + j] = __dsub_rn(m[(size_t)r * w + j], __dmul_rn(f, m[(size_t)c * w + j]));
        __syncthreads();
    }
}

// the right half of [I | inv] into inv (n x n)
__global__ void k_dense_take(int n, const double *__restrict__ m, double *__restrict__ inv)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)n * n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / n), c = (int)(e - (int64_t)r * n);
        inv[e] = m[(size_t)r * 2 * n + n + c];
    }
}

// The same elimination of a small coarsest matrix in one launch: a cluster of
// GJ_CTAS blocks holds the matrix in shared memory, row s in block s % GJ_CTAS.
// Of [A | I] only n columns are ever live: at step c column c of the left half
// is done, and of the right half only the columns of rows that have been
// pivots differ from the identity, so the column of pivot row sp takes the
// place of column c.
// Rows stay where they are; slot_of and pos_of say which row stands where
// after the swaps, and every block keeps them alike.  Per column: each block's
// pivot candidate goes to all blocks, one cluster barrier, then every block
// reads the pivot row from its owner, divides it by the pivot and eliminates
// its own rows.  The owner puts the divided row in place after the next barrier, when
// all blocks have read the old one.  Same pivots, operations and order per
// element as the two kernels above.
//
// What bounds it: n steps of a cluster barrier, n divisions per block (about
// 4 us a step together) and n / 8 rows of FP64 on one SM (4 us more at n =
// 256), against two launches a step and all SMs.  Setup of one dense level,
// us, at n = 24, 97, 160, 256, 300: 316, 1090, 1764, 3200, 3818 -> 137, 527,
// 899, 2182, 3364; the lines meet a little above GJ_MAX_N.
constexpr int GJ_CTAS = 8, GJ_THREADS = 256;
constexpr int GJ_MAX_N = 304;
constexpr size_t gj_smem(int n) { return sizeof(double) * ((size_t)(n + GJ_CTAS - 1) / GJ_CTAS + 2) * n; }
static_assert(gj_smem(GJ_MAX_N) <= 200 * 1024, "the coarsest matrix fits in a cluster's shared memory");

__device__ __forceinline__ unsigned cluster_addr(const void *p, int rank)
{
    unsigned a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ double ld_cluster(unsigned a)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

__global__ void __cluster_dims__(GJ_CTAS, 1, 1) __launch_bounds__(GJ_THREADS)
k_gj_cluster(int n, const int *__restrict__ ptr, const int *__restrict__ col, const double *__restrict__ val,
             double *__restrict__ inv, int *__restrict__ bad)
{
    extern __shared__ __align__(16) double gj[];
    __shared__ double cv[2][GJ_CTAS];                   // candidates of the blocks, by the step's parity
    __shared__ int cp[2][GJ_CTAS];
    __shared__ int slot_of[GJ_MAX_N], pos_of[GJ_MAX_N];
    const int R = (n + GJ_CTAS - 1) / GJ_CTAS;
    double *tile = gj, *row = gj + (size_t)R * n;       // row: the divided pivot rows of two steps
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = blockIdx.x;   // one cluster: the grid
    for (int t = tid; t < R * n; t += GJ_THREADS) tile[t] = 0.0;
    for (int t = tid; t < n; t += GJ_THREADS) slot_of[t] = pos_of[t] = t;
    __syncthreads();
    for (int i = warp; rank + GJ_CTAS * i < n; i += GJ_THREADS / 32) {
        const int s = rank + GJ_CTAS * i;
        for (int p = ptr[s] + lane; p < ptr[s + 1]; p += 32) tile[(size_t)i * n + col[p]] = val[p];
    }
    cluster_sync();                                     // every block has started
    int last = -1;                                      // the row divided in the step before
    bool singular = false;
    for (int c = 0; c < n; ++c) {
        const int b = c & 1;
        double *rb = row + (size_t)b * n, *ro = row + (size_t)(b ^ 1) * n;
        __syncthreads();
        if (warp == 0) {                                // largest |a|, lowest position on ties
            double best = -1.0;
            int bp = n;
            for (int i = lane; rank + GJ_CTAS * i < n; i += 32) {
                const int ps = pos_of[rank + GJ_CTAS * i];
                const double a = fabs(tile[(size_t)i * n + c]);
                if (ps >= c && (a > best || (a == best && ps < bp))) {
                    best = a;
                    bp = ps;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double a = __shfl_xor_sync(0xffffffffu, best, o);
                const int ps = __shfl_xor_sync(0xffffffffu, bp, o);
                if (a > best || (a == best && ps < bp)) {
                    best = a;
                    bp = ps;
                }
            }
            if (lane < GJ_CTAS) {
                asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cluster_addr(&cv[b][rank], lane)), "d"(best)
                             : "memory");
                asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cluster_addr(&cp[b][rank], lane)), "r"(bp)
                             : "memory");
            }
        }
        cluster_sync();
        if (last >= 0 && last % GJ_CTAS == rank)
            for (int j = tid; j < n; j += GJ_THREADS) tile[(size_t)(last / GJ_CTAS) * n + j] = ro[j];
        double best = -1.0;
        int p = n;
#pragma unroll
        for (int q = 0; q < GJ_CTAS; ++q)
            if (cv[b][q] > best || (cv[b][q] == best && cp[b][q] < p)) {
                best = cv[b][q];
                p = cp[b][q];
            }
        if (p >= n) p = c;                              // a column of NaN: refused below
        const int sp = slot_of[p], sc = slot_of[c];
        const unsigned src = cluster_addr(tile + (size_t)(sp / GJ_CTAS) * n, sp % GJ_CTAS);
        const double piv = ld_cluster(src + 8 * c);
        if (!(piv != 0.0) || !isfinite(piv)) {          // the same value in every block
            singular = true;
            break;
        }
        for (int j = tid; j < n; j += GJ_THREADS) rb[j] = __ddiv_rn(j == c ? 1.0 : ld_cluster(src + 8 * j), piv);
        __syncthreads();
        if (tid == 0) {
            slot_of[p] = sc;
            slot_of[c] = sp;
            pos_of[sc] = p;
            pos_of[sp] = c;
        }
        for (int i = warp; rank + GJ_CTAS * i < n; i += GJ_THREADS / 32) {
            if (rank + GJ_CTAS * i == sp) continue;
            double *t = tile + (size_t)i * n;
            const double f = t[c];
            __syncwarp();                               // every lane has f
            if (f != 0.0) {
#pragma unroll 4
                for (int j = lane; j < n; j += 32) t[j] = __dsub_rn(j == c ? 0.0 : t[j], __dmul_rn(f, rb[j]));
            } else if (lane == 0) {
                t[c] = 0.0;
            }
        }
        last = sp;
    }
    __syncthreads();
    if (singular) {
        if (rank == 0 && tid == 0) atomicOr(bad, 1);
    } else {
        for (int i = warp; rank + GJ_CTAS * i < n; i += GJ_THREADS / 32) {
            const int s = rank + GJ_CTAS * i;
            const double *t = s == last ? row + (size_t)((n - 1) & 1) * n : tile + (size_t)i * n;
            for (int j = lane; j < n; j += 32) inv[(size_t)pos_of[s] * n + slot_of[j]] = t[j];
        }
    }
    cluster_sync();                                     // no block leaves while another reads its rows
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct Dev {
    rs_ctx *ctx;
    std::vector<void *> tmp;
    explicit Dev(rs_ctx *c) : ctx(c) {}
    ~Dev()
    {
        for (void *p : tmp) rs_free(ctx, p);
    }
    template <typename T>
    int alloc(T **p, size_t count)
    {
        *p = nullptr;
        int st = rs_alloc(ctx, (void **)p, sizeof(T) * std::max<size_t>(count, 1));
        if (!st) tmp.push_back(*p);
        return st;
    }
};

int grid_for(rs_ctx *ctx, int64_t n, int threads)
{
    return (int)std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads, (int64_t)ctx->num_sms * 8));
}

// exclusive scan of n counts into out[0..n]; *total on the host
int scan(rs_ctx *ctx, Dev &D, const int *in, int *out, int n, int *total)
{
    const int nb = std::max(1, (n + SCAN_T - 1) / SCAN_T);
    int *bsum, *dt;
    RS_TRY(D.alloc(&bsum, nb));
    RS_TRY(D.alloc(&dt, 1));
    if (nb <= 4) {        // a coarse level: a block's few rounds are shorter than two more launches
        k_scan_top<<<1, SCAN_T, 0, ctx->stream>>>(n, in, out, dt, out + n);
    } else {
        k_scan_blocks<<<nb, SCAN_T, 0, ctx->stream>>>(n, in, out, bsum);
        k_scan_top<<<1, SCAN_T, 0, ctx->stream>>>(nb, bsum, bsum, dt, nullptr);
        k_scan_add<<<nb, SCAN_T, 0, ctx->stream>>>(n, out, bsum, dt);
        ctx->launches += 2;
    }
    RS_TRY(rs_check_launch(ctx));
    RS_CUDA_TRY(cudaMemcpyAsync(total, dt, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    RS_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    return RS_OK;
}

int read_flag(rs_ctx *ctx, const int *d, int *h)
{
    RS_CUDA_TRY(cudaMemcpyAsync(h, d, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    RS_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    return RS_OK;
}

// transpose; with values its rows are sorted (without, their order is open)
int transpose(rs_ctx *ctx, Dev &D, int n, int m, int64_t nnz, const int *ptr, const int *col, const double *val,
              int **tptr, int **tcol, double **tval)
{
    int *cnt, *fill, *ucol = nullptr, tot = 0;
    double *uval = nullptr;
    RS_TRY(D.alloc(&cnt, m));
    RS_TRY(D.alloc(tptr, m + 1));
    RS_TRY(D.alloc(tcol, nnz));
    if (tval) {
        RS_TRY(D.alloc(tval, nnz));
        RS_TRY(D.alloc(&ucol, nnz));
        RS_TRY(D.alloc(&uval, nnz));
    }
    RS_TRY(D.alloc(&fill, m));
    RS_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(int) * std::max(m, 1), ctx->stream));
    k_count_cols<<<grid_for(ctx, nnz, 256), 256, 0, ctx->stream>>>(nnz, col, cnt);
    RS_TRY(rs_check_launch(ctx));
    RS_TRY(scan(ctx, D, cnt, *tptr, m, &tot));
    RS_CUDA_TRY(cudaMemcpyAsync(fill, *tptr, sizeof(int) * std::max(m, 1), cudaMemcpyDeviceToDevice, ctx->stream));
    k_transpose_fill<<<grid_for(ctx, n, 256), 256, 0, ctx->stream>>>(n, ptr, col, val, fill, tval ? ucol : *tcol,
                                                                     uval);
    RS_TRY(rs_check_launch(ctx));
    if (!tval) return RS_OK;
    k_sort_rows<<<grid_for(ctx, (int64_t)m * SORT_L, 128), 128, 0, ctx->stream>>>(m, *tptr, ucol, uval, *tcol, *tval);
    return rs_check_launch(ctx);
}

// one pass of the product: a launch per class of rows that occurs
template <bool FILL>
int spgemm_pass(rs_ctx *ctx, const int (&ncls)[SG_CLASSES + 1], int n, const int *len, const int *aptr,
                const int *acol, const double *aval, const int *bptr, const int *bcol, const double *bval,
                const int *cptr, int *out, double *cval)
{
    static unsigned long long raised = 0;      // one bit per device
    const unsigned long long bit = 1ull << (ctx->device & 63);
    if (!(raised & bit)) {
        RS_CUDA_TRY(cudaFuncSetAttribute(k_spgemm<FILL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(sg_warps(3) * sg_warp_smem(3))));
        raised |= bit;
    }
    for (int c = 0; c < SG_CLASSES; ++c) {
        if (!ncls[c]) continue;
        const int w = sg_warps(c);
        const int per_sm = c == 0 ? 12 : (int)std::min<size_t>(12, 220 * 1024 / (w * sg_warp_smem(c) + 1024));
        // consecutive rows a warp looks through: few enough that every warp has some
        const int64_t resident = (int64_t)ctx->num_sms * per_sm * w;
        const int chunk = (int)std::max<int64_t>(1, std::min<int64_t>(32, n / resident));
        const int64_t need = ((int64_t)n + (int64_t)chunk * w - 1) / ((int64_t)chunk * w);
        const int gb = (int)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)ctx->num_sms * per_sm));
        k_spgemm<FILL><<<gb, 32 * w, w * sg_warp_smem(c), ctx->stream>>>(n, c, chunk, len, aptr, acol, aval, bptr,
                                                                         bcol, bval, cptr, out, cval);
        RS_TRY(rs_check_launch(ctx));
    }
    return RS_OK;
}

// C = A B (n x k by k x m) into freshly allocated device arrays
int spgemm(rs_ctx *ctx, Dev &D, int n, const int *aptr, const int *acol, const double *aval, const int *bptr,
           const int *bcol, const double *bval, int **cptr, int **ccol, double **cval, int64_t *cnnz)
{
    int *cnt, *len, *cls, tot = 0, ncls[SG_CLASSES + 1];
    RS_TRY(D.alloc(&cnt, n));
    RS_TRY(D.alloc(&len, n));
    RS_TRY(D.alloc(cptr, n + 1));
    RS_TRY(D.alloc(&cls, SG_CLASSES + 1));
    RS_CUDA_TRY(cudaMemsetAsync(cls, 0, sizeof(ncls), ctx->stream));
    k_sg_len<<<grid_for(ctx, n, 128), 128, 0, ctx->stream>>>(n, aptr, acol, bptr, len, cls);
    RS_TRY(rs_check_launch(ctx));
    RS_CUDA_TRY(cudaMemcpyAsync(ncls, cls, sizeof(ncls), cudaMemcpyDeviceToHost, ctx->stream));
    RS_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    if (ncls[SG_CLASSES]) return RS_ERR_INVALID_ARG;     // a row of the product has more than SG_CAP terms
    RS_TRY(spgemm_pass<false>(ctx, ncls, n, len, aptr, acol, aval, bptr, bcol, bval, nullptr, cnt, nullptr));
    RS_TRY(scan(ctx, D, cnt, *cptr, n, &tot));
    *cnnz = tot;
    RS_TRY(D.alloc(ccol, tot));
    RS_TRY(D.alloc(cval, tot));
    return spgemm_pass<true>(ctx, ncls, n, len, aptr, acol, aval, bptr, bcol, bval, *cptr, *ccol, *cval);
}

}  // namespace

// The hierarchy of Alg. 3 on the device: M->A[0] is given; builds M->P, M->R,
// M->A[1..], M->cidx, M->d and the coarsest inverse M->cinv; sets M->nlev.
int rs_amg_setup_device(AmgData *M, double theta, int max_levels, int max_coarse)
{
    rs_ctx *ctx = M->ctx;
    int l = 0;
    for (;; ++l) {
        const rs_mat *A = M->A[l];
        const int n = A->n;
        if (n <= max_coarse || l + 1 >= max_levels) break;
        Dev D(ctx);
        const int g = grid_for(ctx, n, 128);
        // 1. strength S and its transpose
        int *scnt, *sptr, *scol, *tptr, *tcol, ns = 0;
        double *th;
        RS_TRY(D.alloc(&th, n));
        RS_TRY(D.alloc(&scnt, n));
        RS_TRY(D.alloc(&sptr, n + 1));
        k_strength_count<<<g, 128, 0, ctx->stream>>>(n, A->ptr, A->col, A->val, theta, th, scnt);
        RS_TRY(rs_check_launch(ctx));
        RS_TRY(scan(ctx, D, scnt, sptr, n, &ns));
        RS_TRY(D.alloc(&scol, ns));
        k_strength_fill<<<g, 128, 0, ctx->stream>>>(n, A->ptr, A->col, A->val, th, sptr, scol);
        RS_TRY(rs_check_launch(ctx));
        RS_TRY(transpose(ctx, D, n, n, ns, sptr, scol, nullptr, &tptr, &tcol, nullptr));
        // 2. PMIS
        double *lam;
        char *st, *old;
        int *und, *flag, *cscan, *cidx, hund = 0, nc = 0;
        RS_TRY(D.alloc(&lam, n));
        RS_TRY(D.alloc(&st, n));
        RS_TRY(D.alloc(&old, n));
        RS_TRY(D.alloc(&und, 1));
        RS_CUDA_TRY(cudaMemsetAsync(und, 0, sizeof(int), ctx->stream));
        k_pmis_init<<<g, 128, 0, ctx->stream>>>(n, tptr, l, lam, st, und);
        RS_TRY(rs_check_launch(ctx));
        RS_TRY(read_flag(ctx, und, &hund));
        for (int round = 0; hund > 0; ++round) {
            if (round > n) return RS_ERR_INVALID_ARG;          // cannot happen: every round decides a point
            RS_CUDA_TRY(cudaMemcpyAsync(old, st, n, cudaMemcpyDeviceToDevice, ctx->stream));
            RS_CUDA_TRY(cudaMemsetAsync(und, 0, sizeof(int), ctx->stream));
            k_pmis_select<<<g, 128, 0, ctx->stream>>>(n, sptr, scol, tptr, tcol, lam, old, st);
            k_pmis_f<<<g, 128, 0, ctx->stream>>>(n, sptr, scol, st, und);
            ctx->launches += 1;
            RS_TRY(rs_check_launch(ctx));
            RS_TRY(read_flag(ctx, und, &hund));
        }
        RS_TRY(D.alloc(&flag, n));
        RS_TRY(D.alloc(&cscan, n + 1));
        k_cflag<<<g, 128, 0, ctx->stream>>>(n, st, flag);
        RS_TRY(rs_check_launch(ctx));
        RS_TRY(scan(ctx, D, flag, cscan, n, &nc));
        if (nc == 0 || nc >= n) break;
        RS_TRY(rs_alloc(ctx, (void **)&cidx, sizeof(int) * n));
        M->cidx[l] = cidx;
        k_cidx<<<g, 128, 0, ctx->stream>>>(n, st, cscan, cidx);
        RS_TRY(rs_check_launch(ctx));
        // 3. direct interpolation P (n x nc)
        int *pcnt, *pptr, *pcol, np = 0;
        double *pval;
        RS_TRY(D.alloc(&pcnt, n));
        RS_TRY(D.alloc(&pptr, n + 1));
        k_interp_count<<<g, 128, 0, ctx->stream>>>(n, sptr, scol, cidx, pcnt);
        RS_TRY(rs_check_launch(ctx));
        RS_TRY(scan(ctx, D, pcnt, pptr, n, &np));
        RS_TRY(D.alloc(&pcol, np));
        RS_TRY(D.alloc(&pval, np));
        k_interp_fill<<<g, 128, 0, ctx->stream>>>(n, A->ptr, A->col, A->val, th, cidx, pptr, pcol, pval);
        RS_TRY(rs_check_launch(ctx));
        // 4. R = P^T (nc x n)
        int *rptr, *rcol;
        double *rval;
        RS_TRY(transpose(ctx, D, n, nc, np, pptr, pcol, pval, &rptr, &rcol, &rval));
        // 5. A_{l+1} = R (A P)
        int *xptr, *xcol, *cptr, *ccol;
        double *xval, *cval;
        int64_t nx = 0, ncn = 0;
        RS_TRY(spgemm(ctx, D, n, A->ptr, A->col, A->val, pptr, pcol, pval, &xptr, &xcol, &xval, &nx));
        RS_TRY(spgemm(ctx, D, nc, rptr, rcol, rval, xptr, xcol, xval, &cptr, &ccol, &cval, &ncn));
        RS_TRY(rs_mat_create_dev(ctx, n, np, pptr, pcol, pval, nullptr, &M->P[l]));
        RS_TRY(rs_mat_create_dev(ctx, nc, np, rptr, rcol, rval, nullptr, &M->R[l]));
        RS_TRY(rs_mat_create_dev(ctx, nc, ncn, cptr, ccol, cval, nullptr, &M->A[l + 1]));
    }
    M->nlev = l + 1;
    const int ncoarse = M->A[l]->n;
    if (ncoarse > RS_AMG_MAX_DENSE) return RS_ERR_INVALID_ARG;   // coarsening stalled: no small coarsest level
    // smoother diagonals, the zero-diagonal check of hybrid Gauss-Seidel
    Dev D(ctx);
    int *bad, hbad = 0;
    RS_TRY(D.alloc(&bad, 1));
    for (int k = 0; k < M->nlev; ++k) {
        const rs_mat *A = M->A[k];
        RS_TRY(rs_alloc(ctx, (void **)&M->d[k], sizeof(double) * A->n));
        RS_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(int), ctx->stream));
        k_amg_l1<<<grid_for(ctx, A->n, 128), 128, 0, ctx->stream>>>(A->n, A->ptr, A->col, A->val, M->d[k], bad);
        RS_TRY(rs_check_launch(ctx));
        RS_TRY(read_flag(ctx, bad, &hbad));
        if (hbad && M->smoother == 1 && k + 1 < M->nlev) return RS_ERR_ZERO_PIVOT;
    }
    // the coarsest matrix's dense inverse
    double *aug;
    RS_TRY(rs_alloc(ctx, (void **)&M->cinv, sizeof(double) * (size_t)ncoarse * ncoarse));
    const rs_mat *Cm = M->A[l];
    RS_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(int), ctx->stream));
    if (ncoarse <= GJ_MAX_N) {
        static unsigned long long raised = 0;  // one bit per device
        const unsigned long long bit = 1ull << (ctx->device & 63);
        if (!(raised & bit)) {
            RS_CUDA_TRY(cudaFuncSetAttribute(k_gj_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)gj_smem(GJ_MAX_N)));
            raised |= bit;
        }
        k_gj_cluster<<<GJ_CTAS, GJ_THREADS, gj_smem(ncoarse), ctx->stream>>>(ncoarse, Cm->ptr, Cm->col, Cm->val,
                                                                             M->cinv, bad);
        RS_TRY(rs_check_launch(ctx));
        RS_TRY(read_flag(ctx, bad, &hbad));
        return hbad ? RS_ERR_ZERO_PIVOT : RS_OK;
    }
    RS_TRY(D.alloc(&aug, (size_t)ncoarse * 2 * ncoarse));
    k_dense_aug<<<grid_for(ctx, (int64_t)ncoarse * 2 * ncoarse, 256), 256, 0, ctx->stream>>>(ncoarse, Cm->ptr,
                                                                                          Cm->col, Cm->val, aug);
    k_dense_scatter<<<grid_for(ctx, ncoarse, 128), 128, 0, ctx->stream>>>(ncoarse, Cm->ptr, Cm->col, Cm->val, aug);
    ctx->launches += 1;
    RS_TRY(rs_check_launch(ctx));
    const int ge = std::max(1, std::min(ncoarse, ctx->num_sms * 4));
    for (int c = 0; c < ncoarse; ++c) {
        k_gj_pivot<<<1, 256, 0, ctx->stream>>>(ncoarse, c, aug, bad);
        k_gj_elim<<<ge, 256, 0, ctx->stream>>>(ncoarse, c, aug, bad);
        ctx->launches += 1;
    }
    RS_TRY(rs_check_launch(ctx));
    RS_TRY(read_flag(ctx, bad, &hbad));
    if (hbad) return RS_ERR_ZERO_PIVOT;
    k_dense_take<<<grid_for(ctx, (int64_t)ncoarse * ncoarse, 256), 256, 0, ctx->stream>>>(ncoarse, aug, M->cinv);
    RS_TRY(rs_check_launch(ctx));
    RS_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    return RS_OK;
}
