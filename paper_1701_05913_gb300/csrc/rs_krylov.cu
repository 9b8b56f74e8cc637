// Krylov solvers: restarted GMRES(m) (Sec. 3, Alg. 1), flexible GMRES and
// BiCGSTAB (named in Sec. 3), right-preconditioned, FP64.
//
// Device-resident design: the Hessenberg matrix, the Givens rotations, the
// rotated residual and every BiCGSTAB scalar live in device memory and are
// updated by the last block of the reduction that produces them, so a whole
// GMRES cycle (or a batch of BiCGSTAB iterations) is enqueued without waiting
// for the host.  Once a cycle has converged, a device flag makes every later
// kernel of the cycle return at once.  The host reads the state back twice
// per GMRES cycle and once per batch of BiCGSTAB iterations.
//
// Orthogonalisation is classical Gram-Schmidt with one full
// reorthogonalisation pass (CGS2) instead of the modified Gram-Schmidt loop
// printed in Alg. 1: the 2(i+1) dot products of step i become three fused
// passes over the basis V (dots; update + dots; update + norm), each a
// tall-skinny product computed row-wise with per-block partial sums.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <chrono>

#include "rs_internal.cuh"

#define RS_PSTRIDE (RS_MAX_RESTART + 8)   // partials per block in ctx->red_partials

struct GmresDev {
    double H[(RS_MAX_RESTART + 1) * RS_MAX_RESTART];   // column-major, ld = m+1
    double cs[RS_MAX_RESTART], sn[RS_MAX_RESTART];
    double g[RS_MAX_RESTART + 1], y[RS_MAX_RESTART + 1];
    double h1[RS_MAX_RESTART + 2], h2[RS_MAX_RESTART + 2];
    double bnorm, tol, beta, hdiv, w0sq, implicit, r2;
    int iters, k, cycle_done, converged, maxit, m, noupd, status;
    double augn2;           // ||Z y||^2 of the last cycle (LGMRES)
    double *hist;           // residual history (device), hist_len entries
    int *host_done;         // pinned host copy of cycle_done
    int hist_len, pad_;
};

// The solver's relative residual estimate after iteration it (from 1) into
// the history, when one is recorded.
__device__ __forceinline__ void record_hist(double *hist, int hist_len, int it, double res, double bnorm)
{
    if (hist && it >= 1 && it - 1 < hist_len) hist[it - 1] = res / bnorm;
}

// A device array for the residual history of one solve, when the context
// records one (rs_set_history); null otherwise.
static int hist_begin(rs_ctx *ctx, double **dh, int *len)
{
    *dh = nullptr;
    *len = ctx->hist_host ? ctx->hist_len : 0;
    if (*len == 0) return RS_OK;
    return rs_alloc(ctx, (void **)dh, sizeof(double) * (size_t)*len);
}

// Copies the first min(len, iters) entries back to the caller's array and
// frees the device array.
static int hist_end(rs_ctx *ctx, double *dh, int len, int iters)
{
    int st = RS_OK;
    const int k = std::min(len, iters);
    if (dh && k > 0) {
        if (cudaMemcpyAsync(ctx->hist_host, dh, sizeof(double) * (size_t)k, cudaMemcpyDeviceToHost, ctx->stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(ctx->stream) != cudaSuccess)
            st = RS_ERR_CUDA;
    }
    rs_free(ctx, dh);
    return st;
}

// ---------------------------------------------------------------------------
// block reduction of up to NC+1 per-thread sums with a last-block finish
// ---------------------------------------------------------------------------
template <int NV, int NW = RS_RED_THREADS / 32>
__device__ __forceinline__ bool reduce_partials(double (&acc)[NV], int nv, double *partials,
                                                unsigned *ticket, double *out)
{
    __shared__ double sm[NW][NV];
    __shared__ bool last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        if (k < nv) {
            const double v = warp_sum(acc[k]);
            if (lane == 0) sm[warp][k] = v;
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nv; k += blockDim.x) {
        double s = 0.0;
        for (int w = 0; w < NW; ++w) s += sm[w][k];
        partials[(size_t)blockIdx.x * RS_PSTRIDE + k] = s;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return false;
    __threadfence();
    for (int k = warp; k < nv; k += NW) {
        double s = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) s += __ldcg(partials + (size_t)b * RS_PSTRIDE + k);
        s = warp_sum(s);
        if (lane == 0) out[k] = s;
    }
    if (threadIdx.x == 0) *ticket = 0;
    __syncthreads();
    return true;
}

// Warp reduce-scatter of NC per-lane values (NC a power of two): after
// log2(NC) exchange-and-add steps lane l holds complete sums of columns
// [l*NC/32, (l+1)*NC/32) (NC >= 32) or of column l/(32/NC) (NC < 32), for
// about NC FP64 additions per lane instead of 5 per column.  Each step is a
// template instance, so every index is a compile-time constant and the
// values stay in registers.
template <int NC, int W, int M>
struct ReduceScatter {
    static __device__ __forceinline__ void run(double (&v)[NC], int lane)
    {
        if constexpr (M >= 1) {
            if constexpr (W > 1) {
                // split: keep one half of the live values, send the other to lane ^ M
                const bool up = lane & M;
#pragma unroll
                for (int j = 0; j < W / 2; ++j) {
                    const double send = up ? v[j] : v[j + W / 2];
                    const double keep = up ? v[j + W / 2] : v[j];
                    v[j] = keep + __shfl_xor_sync(0xffffffffu, send, M);
                }
                ReduceScatter<NC, W / 2, M / 2>::run(v, lane);
            } else {
                v[0] += __shfl_xor_sync(0xffffffffu, v[0], M);
                ReduceScatter<NC, 1, M / 2>::run(v, lane);
            }
        }
    }
};

template <int NC>
__device__ __forceinline__ void warp_reduce_scatter(double (&v)[NC], int lane)
{
    ReduceScatter<NC, NC, 16>::run(v, lane);
}

// Block reduction of NC per-thread column sums (and one extra scalar) with a
// last-block finish: out[k] for k < nc, out[nc] = the extra scalar's sum.
template <int NC, int NW = RS_RED_THREADS / 32>
__device__ __forceinline__ bool reduce_columns(double (&acc)[NC], double extra, bool has_extra, int nc,
                                               double *partials, unsigned *ticket, double *out)
{
    __shared__ double sm[NW][NC + 1];
    __shared__ bool last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    warp_reduce_scatter<NC>(acc, lane);
    if (NC >= 32) {
#pragma unroll
        for (int j = 0; j < NC / 32; ++j) sm[warp][lane * (NC / 32) + j] = acc[j];
    } else {
        constexpr int G = NC < 32 ? 32 / NC : 1;   // lanes sharing one column
        if (lane % G == 0) sm[warp][lane / G] = acc[0];
    }
    if (has_extra) {
        const double e = warp_sum(extra);
        if (lane == 0) sm[warp][NC] = e;
    }
    __syncthreads();
    const int nv = nc + (has_extra ? 1 : 0);
    for (int k = threadIdx.x; k < nv; k += blockDim.x) {
        const int src = k < nc ? k : NC;
        double t = 0.0;
        for (int w = 0; w < NW; ++w) t += sm[w][src];
        partials[(size_t)blockIdx.x * RS_PSTRIDE + k] = t;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return false;
    __threadfence();
    for (int k = warp; k < nv; k += NW) {
        double t = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) t += __ldcg(partials + (size_t)b * RS_PSTRIDE + k);
        t = warp_sum(t);
        if (lane == 0) out[k] = t;
    }
    if (threadIdx.x == 0) *ticket = 0;
    __syncthreads();
    return true;
}

// ---------------------------------------------------------------------------
// CGS2 passes for Arnoldi step i (nc = i+1 basis vectors, w in V[:, i+1])
// ---------------------------------------------------------------------------
// The passes are FP64-bound (one to two multiply-adds per 8 bytes read, on a
// GPU with about two FP64 lanes per clock per SM), so the loads are taken off
// the FP64 warps: one producer thread streams tiles of TILE rows of the nc
// basis vectors and of w into a shared-memory ring of 3 to 8 stages with bulk copies
// (completion counted by an mbarrier per stage), and the consumer warps,
// one row per thread, run only shared-memory loads and multiply-adds.
//   pass 1 (CGS_DOTS):        h1 = V^T w, and ||w||^2 for the breakdown test
//   pass 2 (CGS_UPDATE_DOTS): w -= V h1; h2 = V^T w; H[:, i] = h1 + h2
//   pass 3 (CGS_UPDATE_NORM): w -= V h2; h_{i+1,i} = ||w||; Givens update
// A block's consumer thread adds its rows in tile order and the block sums go
// through the fixed last-block reduction, so the results are deterministic.
enum { CGS_DOTS = 0, CGS_UPDATE_DOTS = 1, CGS_UPDATE_NORM = 2 };

template <int NC>
struct CgsCfg {
    static constexpr int CW = NC <= 32 ? 4 : 2;        // consumer warps
    static constexpr int NW = CW + 1;                   // + the producer warp
    static constexpr int THREADS = 32 * NW;
    static constexpr int TILE = 32 * CW;                // rows per tile, one per consumer thread
    static constexpr int STAGE = (NC + 1) * TILE;       // doubles per stage: NC columns, then w
    // stages: about 100 KB of ring per block (two blocks per SM), so that a
    // narrow basis still keeps enough bytes in flight to feed the FP64 pipe
    static constexpr int S = 100 * 1024 / (STAGE * 8) < 3 ? 3 : (100 * 1024 / (STAGE * 8) > 8 ? 8 : 100 * 1024 / (STAGE * 8));
    static constexpr size_t SMEM = (size_t)S * STAGE * sizeof(double) + 2 * S * sizeof(unsigned long long);
};

// The Givens rotations on the new Hessenberg column h[0..nc) with
// h_{nc,nc-1} = hnext (h[nc] is set to 0), the rotated residual, the
// convergence and happy-breakdown tests and the next vector's scale.  cs, sn:
// the earlier rotations (nc - 1 of them are read).
// A warp calls it.  An FP64 instruction takes a warp 64 cycles whether one lane
// works or all, so only what depends on the rotation before stays in the chain
// (two of the six operations a rotation); the products beside it, the new
// column and the three quotients are taken lane by lane.  Same operations.
__device__ __forceinline__ void givens_update(GmresDev *d, int nc, double *h, const double *cs, const double *sn,
                                              double hnext, double w0sq, int lane)
{
    __shared__ double av[RS_MAX_RESTART], cb[RS_MAX_RESTART];
    const int i = nc - 1;
    double sb[(RS_MAX_RESTART + 31) / 32];
#pragma unroll
    for (int q = 0; q < (RS_MAX_RESTART + 31) / 32; ++q) {
        const int k = lane + 32 * q;
        if (k >= i) continue;
        cb[k] = __dmul_rn(cs[k], h[k + 1]);
        sb[q] = __dmul_rn(sn[k], h[k + 1]);
    }
    __syncwarp();
    double a = h[0];
#pragma unroll 4
    for (int k = 0; k < i; ++k) {
        if (lane == 0) av[k] = a;
        a = __dadd_rn(__dmul_rn(-sn[k], a), cb[k]);
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < (RS_MAX_RESTART + 31) / 32; ++q) {
        const int k = lane + 32 * q;
        if (k < i) h[k] = __dadd_rn(__dmul_rn(cs[k], av[k]), sb[q]);
    }
    const double rho = hypot(a, hnext);
    const double quot = __ddiv_rn(lane == 0 ? a : lane == 1 ? hnext : 1.0, lane < 2 ? rho : hnext);
    const double c = __shfl_sync(0xffffffffu, quot, 0), s = __shfl_sync(0xffffffffu, quot, 1);
    const double hinv = __shfl_sync(0xffffffffu, quot, 2);
    __syncwarp();
    if (lane != 0) return;
    const double g = d->g[i];
    d->cs[i] = c;
    d->sn[i] = s;
    h[i] = rho;
    h[nc] = 0.0;
    const double g1 = __dmul_rn(-s, g);
    d->g[i + 1] = g1;
    d->g[i] = __dmul_rn(c, g);
    const int iters = d->iters + 1;
    d->iters = iters;
    d->k = i + 1;
    const double implicit = fabs(g1);
    d->implicit = implicit;
    record_hist(d->hist, d->hist_len, iters, implicit, d->bnorm);
    const bool happy = hnext <= 1e-14 * sqrt(w0sq);
    if (implicit <= d->tol || iters >= d->maxit || happy || i == d->m - 1) {
        d->cycle_done = 1;
        *(volatile int *)d->host_done = 1;
    }
    d->hdiv = hinv;            // v_{i+1} = w / h_{i+1,i}
}

// NC: columns of the ring and of the reduction (a power of two); NCC: the
// unrolled bound of the multiply-add loops (nc rounded down to 4); the last
// nc - NCC (0 to 3) columns take a warp-uniform branch, so that no FP64
// multiply-add is issued for a column that does not exist (predicated-off
// FP64 instructions still occupy the FP64 pipe on this GPU).
template <int NC, int NCC, int MODE>
__global__ void __launch_bounds__(CgsCfg<NC>::THREADS)
k_cgs_pass(int n, int ld, int nc, const double *__restrict__ V, double *w, double *partials, unsigned *ticket,
           GmresDev *d, int *err, long long limit)
{
    typedef CgsCfg<NC> C;
    extern __shared__ __align__(128) unsigned char cgs_smem[];
    double *ring = (double *)cgs_smem;
    unsigned long long *full = (unsigned long long *)(ring + C::S * C::STAGE);
    unsigned long long *empty = full + C::S;
    __shared__ double hs[NC];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], C::CW);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (rs_pdl_wait()) return;
    if (*(volatile int *)&d->cycle_done) return;
    if (MODE != CGS_DOTS)
        for (int k = threadIdx.x; k < nc; k += blockDim.x) hs[k] = MODE == CGS_UPDATE_DOTS ? d->h1[k] : d->h2[k];
    __syncthreads();
    const int ntiles = (n + C::TILE - 1) / C::TILE;
    double acc[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) acc[k] = 0.0;
    double extra = 0.0;
    if (warp == C::CW) {
        if (lane == 0) {
            // producer: whole tiles, the last one rounded up to an even row
            // count (inside the column padding: ld is a multiple of 32)
            int it = 0;
            for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
                const int s = it % C::S;
                if (it >= C::S) mbar_wait(&empty[s], (unsigned)((it / C::S - 1) & 1), limit, err);
                const int r0 = tile * C::TILE;
                const int rows = min(C::TILE, n - r0);
                const unsigned bytes = (unsigned)((rows + 1) & ~1) * 8u;
                double *st = ring + s * C::STAGE;
                mbar_arrive_expect_tx(&full[s], bytes * (unsigned)(nc + 1));
                for (int k = 0; k < nc; ++k) bulk_g2s(st + k * C::TILE, V + (size_t)k * ld + r0, bytes, &full[s]);
                bulk_g2s(st + NC * C::TILE, w + r0, bytes, &full[s]);
            }
        }
    } else {
        int it = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
            const int s = it % C::S;
            mbar_wait(&full[s], (unsigned)((it / C::S) & 1), limit, err);
            const double *st = ring + s * C::STAGE + threadIdx.x;
            const int r = tile * C::TILE + threadIdx.x;
            if (r < n) {
                const double wr = st[NC * C::TILE];
                const int rem = nc - NCC;   // 0..3, the same for the whole grid
                if (MODE == CGS_DOTS) {
#pragma unroll
                    for (int k = 0; k < NCC; ++k) acc[k] = fma(st[k * C::TILE], wr, acc[k]);
#pragma unroll
                    for (int k = NCC; k < NCC + 3 && k < NC; ++k)
                        if (k - NCC < rem) acc[k] = fma(st[k * C::TILE], wr, acc[k]);
                    extra = fma(wr, wr, extra);
                } else {
                    double s0 = 0.0, s1 = 0.0;
#pragma unroll
                    for (int k = 0; k < NCC; ++k) {
                        if (k & 1) s1 = fma(st[k * C::TILE], hs[k], s1);
                        else s0 = fma(st[k * C::TILE], hs[k], s0);
                    }
#pragma unroll
                    for (int k = NCC; k < NCC + 3 && k < NC; ++k) {
                        if (k - NCC < rem) {
                            if (k & 1) s1 = fma(st[k * C::TILE], hs[k], s1);
                            else s0 = fma(st[k * C::TILE], hs[k], s0);
                        }
                    }
                    const double w1 = wr - (s0 + s1);
                    w[r] = w1;
                    if (MODE == CGS_UPDATE_DOTS) {
#pragma unroll
                        for (int k = 0; k < NCC; ++k) acc[k] = fma(st[k * C::TILE], w1, acc[k]);
#pragma unroll
                        for (int k = NCC; k < NCC + 3 && k < NC; ++k)
                            if (k - NCC < rem) acc[k] = fma(st[k * C::TILE], w1, acc[k]);
                    } else {
                        extra = fma(w1, w1, extra);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[s]);
        }
    }
    if (MODE == CGS_DOTS) {
        if (reduce_columns<NC, C::NW>(acc, extra, true, nc, partials, ticket, d->h1)) {
            if (threadIdx.x == 0) d->w0sq = d->h1[nc];
        }
    } else if (MODE == CGS_UPDATE_DOTS) {
        if (reduce_columns<NC, C::NW>(acc, 0.0, false, nc, partials, ticket, d->h2)) {
            const int i = nc - 1, m1 = d->m + 1;
            for (int k = threadIdx.x; k < nc; k += blockDim.x) d->H[(size_t)i * m1 + k] = hs[k] + d->h2[k];
        }
    } else {
        double a1[1] = {extra};
        if (reduce_partials<1, C::NW>(a1, 1, partials, ticket, &d->r2)) {
            // the new Hessenberg column and the rotations through shared
            // memory: one thread's chain of rotations then waits for no load
            // (the ring is free: every tile has been consumed)
            double *h = ring, *cs = ring + NC + 1, *sn = ring + 2 * NC + 2;
            double *hcol = d->H + (size_t)(nc - 1) * (d->m + 1);
            for (int k = threadIdx.x; k < nc; k += blockDim.x) {
                h[k] = hcol[k];
                cs[k] = d->cs[k];
                sn[k] = d->sn[k];
            }
            __syncthreads();
            if (warp == 0) givens_update(d, nc, h, cs, sn, sqrt(d->r2), d->w0sq, lane);
            __syncthreads();
            for (int k = threadIdx.x; k <= nc; k += blockDim.x) hcol[k] = h[k];
        }
    }
}

// ---------------------------------------------------------------------------
// The same step of a small system in one launch: a cluster of CS_CTAS blocks,
// each with its rows of the nc basis vectors and of w in shared memory from
// the first product to the last.  Column sums go block to block through
// distributed shared memory and are added in block order, and the new basis
// vector is written already scaled by 1 / h_{i+1,i}.  What bounds it: three
// cluster barriers and the FP64 multiply-adds of CS_CTAS SMs (4 n nc in all:
// about 4 of 21 us at 1920 rows and 15 columns).  The basis is loaded while the
// product before still runs.  Against three passes and the scaling, GMRES(30)
// with ILU(0) at 16x12x10: 3521 -> 2830 us, 57 -> 46 us an iteration (3136 with the
// loads after the wait; a cluster of 16 blocks took 5 % longer than 8, with
// more to exchange).
// ---------------------------------------------------------------------------
#define CS_CTAS 8
#define CS_THREADS 256
// Beyond, the passes' more SMs win.  A GMRES(30) cycle with ILU(0), us, in one
// launch a step / in passes: 960 rows 1242 / 1611, 1920 1521 / 1813, 3072 1866 /
// 2159, 4096 2118 / 2334, 6144 2314 / 2420; 7168 rows (24 columns fit) 2428 / 2452,
// 9216 (19 columns) 2923 / 2853.
#define CS_MAX_ROWS 6144
#define CS_SMEM (190 * 1024)

// rows of a block: even, so that a column's rows are whole 16-byte copies
__host__ __device__ __forceinline__ int cgs_small_rows(int n) { return ((n + CS_CTAS - 1) / CS_CTAS + 1) & ~1; }

static size_t cgs_small_smem(int n, int nc) { return sizeof(double) * (size_t)cgs_small_rows(n) * (nc + 1); }

__global__ void __cluster_dims__(CS_CTAS, 1, 1) __launch_bounds__(CS_THREADS)
k_cgs_small(int n, int ld, int nc, double *__restrict__ V, GmresDev *d)
{
    extern __shared__ __align__(16) double cs_tile[];           // [nc + 1][R]: basis vectors, then w
    __shared__ double ex[3][CS_CTAS][RS_MAX_RESTART + 2];       // the blocks' sums, one buffer an exchange
    __shared__ double part[RS_MAX_RESTART + 2], h[RS_MAX_RESTART + 2], h2[RS_MAX_RESTART + 2];
    __shared__ double cs[RS_MAX_RESTART], sn[RS_MAX_RESTART];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = blockIdx.x;                                // one cluster: the grid
    const int R = cgs_small_rows(n), r0 = rank * R, rows = max(0, min(R, n - r0));
    double *w = cs_tile + (size_t)nc * R;
    // columns [k0, k1) through L2; ld has room for an odd last row's neighbour
    auto load = [&](int k0, int k1) {
        const int pairs = (rows + 1) / 2;
        for (int t = tid; t < (k1 - k0) * pairs; t += CS_THREADS) {
            const int k = t / pairs, q = 2 * (t - k * pairs);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(cs_tile + (size_t)(k0 + k) * R + q)),
                         "l"(V + (size_t)(k0 + k) * ld + r0 + q)
                         : "memory");
        }
    };
    // the kernel before is the product that writes w: the basis is older
    load(0, nc);
    const bool never = rs_pdl_wait(), done = never || *(volatile int *)&d->cycle_done;  // set by this step at the
                                                                                        // earliest after its barriers
    if (!done) load(nc, nc + 1);
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (done) return;
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");   // a block that has not started has no memory to write to
    __syncthreads();
    // part[k] = this block's rows of <V_k, w>, k < cols (k = nc: <w, w>)
    auto dots = [&](int cols) {
        for (int k0 = 4 * warp; k0 < cols; k0 += 4 * (CS_THREADS / 32)) {
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
            for (int r = lane; r < rows; r += 32) {
                const double wr = w[r];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (k0 + j < cols) acc[j] = fma(cs_tile[(size_t)(k0 + j) * R + r], wr, acc[j]);
            }
            warp_reduce_scatter<4>(acc, lane);
            if (lane % 8 == 0 && k0 + lane / 8 < cols) part[k0 + lane / 8] = acc[0];
        }
        __syncthreads();
    };
    // out[k] = the sum of every block's part[k], added in block order
    auto exchange = [&](int which, int cols, double *out) {
        for (int t = tid; t < cols * CS_CTAS; t += CS_THREADS) {
            const int q = t / cols, k = t - q * cols;
            unsigned dst;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(smem_addr(&ex[which][rank][k])), "r"(q));
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dst), "d"(part[k]) : "memory");
        }
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        for (int k = tid; k < cols; k += CS_THREADS) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < CS_CTAS; ++q) s += ex[which][q][k];
            out[k] = s;
        }
        __syncthreads();
    };
    // w -= V c; the block's rows of <w, w> if asked for
    auto update = [&](const double *c) -> double {
        double sq = 0.0;
        for (int r = tid; r < rows; r += CS_THREADS) {
            double s0 = 0.0, s1 = 0.0;
            int k = 0;
            for (; k + 1 < nc; k += 2) {
                s0 = fma(cs_tile[(size_t)k * R + r], c[k], s0);
                s1 = fma(cs_tile[(size_t)(k + 1) * R + r], c[k + 1], s1);
            }
            if (k < nc) s0 = fma(cs_tile[(size_t)k * R + r], c[k], s0);
            const double v = w[r] - (s0 + s1);
            w[r] = v;
            sq = fma(v, v, sq);
        }
        return sq;
    };
    // h1 = V^T w and ||w||^2; w -= V h1; h2 = V^T w; w -= V h2; ||w||
    dots(nc + 1);
    asm volatile("barrier.cluster.wait;" ::: "memory");
    exchange(0, nc + 1, h);
    const double w0sq = h[nc];
    update(h);
    __syncthreads();
    dots(nc);
    exchange(1, nc, h2);
    double sq = warp_sum(update(h2));
    __syncthreads();
    if (lane == 0) part[1 + warp] = sq;
    __syncthreads();
    if (tid == 0) {
        sq = 0.0;
        for (int q = 0; q < CS_THREADS / 32; ++q) sq += part[1 + q];
        part[0] = sq;
    }
    __syncthreads();
    __shared__ double total[1];
    exchange(2, 1, total);
    const double hnext = sqrt(total[0]), inv = 1.0 / hnext;
    for (int r = tid; r < rows; r += CS_THREADS) V[(size_t)nc * ld + r0 + r] = w[r] * inv;
    if (rank != 0) return;
    double *hcol = d->H + (size_t)(nc - 1) * (d->m + 1);
    for (int k = tid; k < nc; k += CS_THREADS) {
        h[k] += h2[k];
        cs[k] = d->cs[k];
        sn[k] = d->sn[k];
    }
    __syncthreads();
    if (warp == 0) givens_update(d, nc, h, cs, sn, hnext, w0sq, lane);
    __syncthreads();
    for (int k = tid; k <= nc; k += CS_THREADS) hcol[k] = h[k];
}

// x[r] (or u[r]) = sum_j B[j][r] y[j] for j < k; add = 1 accumulates into x
__global__ void k_basis_combine(int n, int ld, const double *__restrict__ B, const GmresDev *d,
                                double *__restrict__ x, int add)
{
    if (rs_pdl_wait()) return;
    if (*(volatile const int *)&d->noupd) return;
    __shared__ double ys[RS_MAX_RESTART];
    const int k = d->k;
    for (int j = threadIdx.x; j < k; j += blockDim.x) ys[j] = d->y[j];
    __syncthreads();
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int j = 0; j < k; ++j) s = fma(B[(size_t)j * ld + r], ys[j], s);
        x[r] = add ? __dadd_rn(x[r], s) : s;
    }
}

// v = s * r with s a device scalar (the reciprocal of the normalising norm)
__global__ void k_scale_dev(int n, const double *__restrict__ r, const double *__restrict__ s,
                            double *__restrict__ v, const int *skip)
{
    if (rs_pdl_wait()) return;
    if (skip && *(volatile const int *)skip) return;
    const double a = *s;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) v[i] = r[i] * a;
}

// y = x / sqrt(*n2) (0 when *n2 = 0): the normalised LGMRES correction
__global__ void k_scale_rsqrt(int n, const double *__restrict__ x, const double *__restrict__ n2,
                              double *__restrict__ y, const int *skip)
{
    if (rs_pdl_wait()) return;
    if (skip && *(volatile const int *)skip) return;
    const double s = *n2;
    const double a = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) y[i] = x[i] * a;
}

__global__ void k_axpy_skip(int n, const double *__restrict__ x, double *__restrict__ y, const int *skip)
{
    if (rs_pdl_wait()) return;
    if (skip && *(volatile const int *)skip) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) y[i] += x[i];
}

// cycle start: beta = ||r||, convergence test on the true residual
__global__ void k_gmres_start(GmresDev *d, const double *r2, double rtol, int first)
{
    if (rs_pdl_wait()) return;
    if (threadIdx.x != 0) return;
    const double beta = sqrt(*r2);
    if (first) {
        d->tol = rtol * d->bnorm;
    }
    d->beta = beta;
    d->implicit = beta;
    d->converged = beta <= d->tol;
    d->cycle_done = d->converged || d->iters >= d->maxit;
    d->g[0] = beta;
    for (int j = 1; j <= d->m; ++j) d->g[j] = 0.0;
    d->k = 0;
    d->noupd = 1;
    d->hdiv = 1.0 / beta;      // v_1 = r / beta
}

// y = H(0:k,0:k)^{-1} g(0:k) by back-substitution, row by row, one thread's
// chain of k^2/2 multiply-adds: from a copy of H in shared memory (from
// global memory it took 62 us at k = 30, now 33)
__global__ void __launch_bounds__(256) k_gmres_backsolve(GmresDev *d)
{
    if (rs_pdl_wait()) return;
    __shared__ double hs[(RS_MAX_RESTART * (RS_MAX_RESTART + 1)) / 2];   // column l: rows 0..l, from l (l + 1) / 2
    __shared__ double ys[RS_MAX_RESTART];
    const int k = d->k, m1 = d->m + 1;
    for (int l = threadIdx.x >> 5; l < k; l += blockDim.x >> 5)
        for (int j = threadIdx.x & 31; j <= l; j += 32) hs[l * (l + 1) / 2 + j] = d->H[(size_t)l * m1 + j];
    for (int j = threadIdx.x; j < k; j += blockDim.x) ys[j] = d->g[j];
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int j = k - 1; j >= 0; --j) {
            double s = ys[j];
            for (int l = j + 1; l < k; ++l) s = fma(-hs[l * (l + 1) / 2 + j], ys[l], s);
            ys[j] = __ddiv_rn(s, hs[j * (j + 1) / 2 + j]);
        }
        d->noupd = k == 0;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < k; j += blockDim.x) d->y[j] = ys[j];
}

// Blocks of a reduction over n rows, `rows` of them per block and round: at
// most red_blocks, and no block without rows, since the last block adds one
// partial per block (at 1920 rows the CGS2 passes took 9 to 25 us with 304
// blocks of which 15 had rows, and take 6 to 19 with those 15).
static int red_grid(rs_ctx *ctx, int n, int rows)
{
    return std::max(1, std::min(ctx->red_blocks, (n + rows - 1) / rows));
}

static int blas_grid(rs_ctx *ctx, int n)
{
    return std::max(1, std::min((n + 255) / 256, ctx->num_sms * 8));
}

template <int NC, int NCC, int MODE>
static int launch_cgs_pass(rs_ctx *ctx, int n, int ld, int nc, double *V, GmresDev *d)
{
    typedef CgsCfg<NC> C;
    static unsigned long long raised = 0;   // devices whose shared-memory limit was raised
    const unsigned long long bit = 1ull << (ctx->device & 63);
    if (C::SMEM > 48 * 1024 && !(raised & bit)) {
        RS_CUDA_TRY(cudaFuncSetAttribute(k_cgs_pass<NC, NCC, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)C::SMEM));
        raised |= bit;
    }
    RsProfScope prof(ctx, MODE == CGS_DOTS ? RS_PROF_CGS_DOTS
                          : MODE == CGS_UPDATE_DOTS ? RS_PROF_CGS_UPDATE_DOTS : RS_PROF_CGS_UPDATE_NORM);
    rs_pdl(k_cgs_pass<NC, NCC, MODE>, red_grid(ctx, n, C::TILE), C::THREADS, C::SMEM, ctx)(
        n, ld, nc, V, V + (size_t)nc * ld, ctx->red_partials, ctx->red_ticket, d, ctx->d_err, ctx->spin_limit);
    return rs_check_launch(ctx);
}

// NCC = nc rounded down to 4; the reduction and ring width NC (a power of
// two) holds the up to 3 columns past it
template <int NCC>
static int launch_cgs(rs_ctx *ctx, int n, int ld, int nc, double *V, GmresDev *d)
{
    constexpr int NC = NCC + 3 <= 8 ? 8 : NCC + 3 <= 16 ? 16 : NCC + 3 <= 32 ? 32 : 64;
    int st = launch_cgs_pass<NC, NCC, CGS_DOTS>(ctx, n, ld, nc, V, d);
    if (!st) st = launch_cgs_pass<NC, NCC, CGS_UPDATE_DOTS>(ctx, n, ld, nc, V, d);
    if (!st) st = launch_cgs_pass<NC, NCC, CGS_UPDATE_NORM>(ctx, n, ld, nc, V, d);
    return st;
}

// small systems: one launch, and V[:, nc] comes out scaled
static bool cgs_is_small(int n, int nc) { return n <= CS_MAX_ROWS && cgs_small_smem(n, nc) <= CS_SMEM; }

static int cgs_step(rs_ctx *ctx, int n, int ld, int nc, double *V, GmresDev *d)
{
    if (cgs_is_small(n, nc)) {
        static unsigned long long raised = 0;   // devices whose shared-memory limit was raised
        const unsigned long long bit = 1ull << (ctx->device & 63);
        if (!(raised & bit)) {
            RS_CUDA_TRY(cudaFuncSetAttribute(k_cgs_small, cudaFuncAttributeMaxDynamicSharedMemorySize, CS_SMEM));
            raised |= bit;
        }
        RsProfScope prof(ctx, RS_PROF_CGS_UPDATE_DOTS);
        rs_pdl(k_cgs_small, CS_CTAS, CS_THREADS, cgs_small_smem(n, nc), ctx)(n, ld, nc, V, d);
        return rs_check_launch(ctx);
    }
    switch (nc / 4) {
    case 0: return launch_cgs<0>(ctx, n, ld, nc, V, d);
    case 1: return launch_cgs<4>(ctx, n, ld, nc, V, d);
    case 2: return launch_cgs<8>(ctx, n, ld, nc, V, d);
    case 3: return launch_cgs<12>(ctx, n, ld, nc, V, d);
    case 4: return launch_cgs<16>(ctx, n, ld, nc, V, d);
    case 5: return launch_cgs<20>(ctx, n, ld, nc, V, d);
    case 6: return launch_cgs<24>(ctx, n, ld, nc, V, d);
    case 7: return launch_cgs<28>(ctx, n, ld, nc, V, d);
    case 8: return launch_cgs<32>(ctx, n, ld, nc, V, d);
    case 9: return launch_cgs<36>(ctx, n, ld, nc, V, d);
    case 10: return launch_cgs<40>(ctx, n, ld, nc, V, d);
    case 11: return launch_cgs<44>(ctx, n, ld, nc, V, d);
    case 12: return launch_cgs<48>(ctx, n, ld, nc, V, d);
    case 13: return launch_cgs<52>(ctx, n, ld, nc, V, d);
    case 14: return launch_cgs<56>(ctx, n, ld, nc, V, d);
    case 15: return launch_cgs<60>(ctx, n, ld, nc, V, d);
    default: return nc <= 64 ? launch_cgs<64 - 3>(ctx, n, ld, nc, V, d) : RS_ERR_INVALID_ARG;
    }
}

static int finish_info(rs_ctx *ctx, const rs_mat *A, const double *b, const double *x, double *r,
                       double bnorm, rs_solve_info *info)
{
    RS_TRY(rs_residual_launch(A, b, x, r, ctx->d_scalars + 1, nullptr));
    RS_CUDA_TRY(cudaMemcpyAsync(ctx->h_pinned + 1, ctx->d_scalars + 1, sizeof(double),
                                cudaMemcpyDeviceToHost, ctx->stream));
    RS_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    info->true_rel_res = bnorm > 0 ? sqrt(ctx->h_pinned[1]) / bnorm : 0.0;
    return RS_OK;
}

// GMRES(m) (Alg. 1 with right preconditioning and CGS2), FGMRES(m), and
// with aug_k > 0 (flexible only) LGMRES(m, aug_k): each cycle then adds one
// Arnoldi step per stored correction of the last aug_k cycles (newest
// first, held in a ring), and the cycle's correction Z y, normalised, joins
// the ring.
static int gmres_impl(const rs_mat *A, rs_pc *M, const rs_vec *bv, rs_vec *xv, int m, int aug_k, double rtol,
                      int maxit, int flexible, rs_solve_info *info)
{
    if (!A || !bv || !xv || !info) return RS_ERR_INVALID_ARG;
    if (m < 1 || aug_k < 0 || m + aug_k > RS_MAX_RESTART || (aug_k > 0 && !flexible) || maxit < 0 || !(rtol >= 0))
        return RS_ERR_INVALID_ARG;
    if (bv->n != A->n || xv->n != A->n) return RS_ERR_SIZE_MISMATCH;
    if (M && M->A->n != A->n) return RS_ERR_SIZE_MISMATCH;
    memset(info, 0, sizeof(*info));
    info->bad_row = -1;
    rs_ctx *ctx = A->ctx;
    const auto t0 = std::chrono::steady_clock::now();
    const int n = A->n;
    const int ld = (n + 31) / 32 * 32;
    double *V = nullptr, *Z = nullptr, *r = nullptr, *t = nullptr, *Aug = nullptr;
    GmresDev *d = nullptr;
    double *dhist = nullptr;
    int hlen = 0;
    int naug = 0, head = 0;      // stored corrections; the next ring slot
    // The host enqueues a cycle at most STEPS_AHEAD steps ahead of the device
    // and stops once the device has reported the cycle done: the kernels of
    // further steps would only return.
    constexpr int STEPS_AHEAD = 4;
    cudaEvent_t ev[STEPS_AHEAD] = {};
    volatile int *host_done = (volatile int *)(ctx->h_pinned + 32);
    int st = rs_alloc(ctx, (void **)&V, sizeof(double) * (size_t)ld * (m + aug_k + 1));
    if (!st && flexible) st = rs_alloc(ctx, (void **)&Z, sizeof(double) * (size_t)ld * (m + aug_k));
    if (!st && aug_k > 0) st = rs_alloc(ctx, (void **)&Aug, sizeof(double) * (size_t)ld * aug_k);
    if (!st) st = rs_alloc(ctx, (void **)&r, sizeof(double) * ld);
    if (!st) st = rs_alloc(ctx, (void **)&t, sizeof(double) * ld);
    if (!st) st = rs_alloc(ctx, (void **)&d, sizeof(GmresDev));
    if (!st) st = hist_begin(ctx, &dhist, &hlen);
    for (cudaEvent_t &e : ev)
        if (!st && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) st = RS_ERR_CUDA;
    int status = RS_NOT_CONVERGED;
    double bnorm = 0.0;
    const double *b = bv->d;
    double *x = xv->d;
    if (st) goto out;
    {
        GmresDev h0;
        memset(&h0, 0, sizeof(h0));
        h0.m = m;
        h0.maxit = maxit;
        h0.noupd = 1;
        h0.hist = dhist;
        h0.hist_len = hlen;
        h0.host_done = (int *)host_done;
        // ||b||
        st = rs_dot_launch(ctx, n, b, b, ctx->d_scalars);
        if (st) goto out;
        if (cudaMemcpyAsync(ctx->h_pinned, ctx->d_scalars, sizeof(double), cudaMemcpyDeviceToHost,
                            ctx->stream) != cudaSuccess ||
            cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
            st = RS_ERR_CUDA;
            goto out;
        }
        bnorm = sqrt(ctx->h_pinned[0]);
        if (bnorm == 0.0) {
            cudaMemsetAsync(x, 0, sizeof(double) * n, ctx->stream);
            status = RS_OK;
            goto done;
        }
        h0.bnorm = bnorm;
        cudaMemcpyAsync(d, &h0, sizeof(h0), cudaMemcpyHostToDevice, ctx->stream);
        const int gb = blas_grid(ctx, n);
        int *cycle_done = &d->cycle_done;
        int *noupd = &d->noupd;
        int first = 1;
        for (;;) {
            // this cycle's Arnoldi dimension: m, plus the stored corrections
            const int dim = m + naug;
            if (aug_k > 0 &&
                cudaMemcpyAsync(&d->m, &dim, sizeof(int), cudaMemcpyHostToDevice, ctx->stream) != cudaSuccess) {
                st = RS_ERR_CUDA;
                goto out;
            }
            // true residual and cycle start
            st = rs_residual_launch(A, b, x, r, &d->r2, nullptr);
            if (st) goto out;
            rs_pdl(k_gmres_start, 1, 32, 0, ctx)(d, &d->r2, rtol, first);
            first = 0;
            ctx->launches++;
            int hs[4];
            if (cudaMemcpyAsync(hs, &d->iters, sizeof(int) * 4, cudaMemcpyDeviceToHost, ctx->stream) != cudaSuccess ||
                cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
                st = RS_ERR_CUDA;
                goto out;
            }
            *host_done = 0;
            // hs: iters, k, cycle_done, converged
            info->iters = hs[0];
            if (hs[3]) { status = RS_OK; break; }
            if (hs[2]) { status = RS_NOT_CONVERGED; break; }
            rs_pdl(k_scale_dev, gb, 256, 0, ctx)(n, r, &d->hdiv, V, nullptr);
            ctx->launches++;
            for (int i = 0; i < dim; ++i) {
                if (i >= STEPS_AHEAD) {
                    if (cudaEventSynchronize(ev[i % STEPS_AHEAD]) != cudaSuccess) { st = RS_ERR_CUDA; goto out; }
                    if (*host_done) break;
                }
                double *vi = V + (size_t)i * ld;
                double *zi = flexible ? Z + (size_t)i * ld : t;
                double *w = V + (size_t)(i + 1) * ld;
                if (i >= m) {
                    // augmented step: the (i - m)-th newest stored correction
                    const int slot = ((head - 1 - (i - m)) % aug_k + aug_k) % aug_k;
                    if (cudaMemcpyAsync(zi, Aug + (size_t)slot * ld, sizeof(double) * n, cudaMemcpyDeviceToDevice,
                                        ctx->stream) != cudaSuccess)
                        st = RS_ERR_CUDA;
                } else if (M) {
                    st = rs_pc_apply_dev(M, vi, zi, cycle_done);
                } else if (flexible) {
                    if (cudaMemcpyAsync(zi, vi, sizeof(double) * n, cudaMemcpyDeviceToDevice, ctx->stream) !=
                        cudaSuccess)
                        st = RS_ERR_CUDA;
                } else {
                    zi = vi;
                }
                if (!st) st = rs_spmv_launch(A, zi, 1.0, 0.0, w, cycle_done);
                if (!st) st = cgs_step(ctx, n, ld, i + 1, V, d);
                if (!st && cudaEventRecord(ev[i % STEPS_AHEAD], ctx->stream) != cudaSuccess) st = RS_ERR_CUDA;
                if (st) goto out;
                if (i + 1 < dim && !cgs_is_small(n, i + 1)) {
                    rs_pdl(k_scale_dev, gb, 256, 0, ctx)(n, w, &d->hdiv, w, cycle_done);
                    ctx->launches++;
                }
            }
            rs_pdl(k_gmres_backsolve, 1, 256, 0, ctx)(d);
            ctx->launches++;
            if (flexible && aug_k > 0) {
                // the correction t = Z y; x += t; t / ||t|| joins the ring
                rs_pdl(k_basis_combine, gb, 256, 0, ctx)(n, ld, Z, d, t, 0);
                rs_pdl(k_axpy_skip, gb, 256, 0, ctx)(n, t, x, noupd);
                ctx->launches += 2;
                st = rs_dot_launch(ctx, n, t, t, &d->augn2);
                if (st) goto out;
                rs_pdl(k_scale_rsqrt, gb, 256, 0, ctx)(n, t, &d->augn2, Aug + (size_t)head * ld, noupd);
                ctx->launches++;
                head = (head + 1) % aug_k;
                naug = std::min(naug + 1, aug_k);
            } else if (flexible) {
                rs_pdl(k_basis_combine, gb, 256, 0, ctx)(n, ld, Z, d, x, 1);
                ctx->launches++;
            } else {
                rs_pdl(k_basis_combine, gb, 256, 0, ctx)(n, ld, V, d, r, 0);
                ctx->launches++;
                if (M) {
                    st = rs_pc_apply_dev(M, r, t, noupd);
                    if (st) goto out;
                    rs_pdl(k_axpy_skip, gb, 256, 0, ctx)(n, t, x, noupd);
                } else {
                    rs_pdl(k_axpy_skip, gb, 256, 0, ctx)(n, r, x, noupd);
                }
                ctx->launches++;
            }
            info->restarts++;
            if (cudaGetLastError() != cudaSuccess) { st = RS_ERR_CUDA; goto out; }
        }
        GmresDev hf;
        cudaMemcpyAsync(&hf, d, sizeof(hf), cudaMemcpyDeviceToHost, ctx->stream);
        cudaStreamSynchronize(ctx->stream);
        info->iters = hf.iters;
        info->implicit_rel_res = hf.implicit / bnorm;
    }
done:
    st = rs_collect_device_error(ctx, &info->bad_row);
    if (st) goto out;
    st = finish_info(ctx, A, b, x, r ? r : t, bnorm, info);
    if (st) goto out;
    if (status == RS_OK && info->true_rel_res > rtol && bnorm > 0) status = RS_NOT_CONVERGED;
out:
    {
        const int hs = hist_end(ctx, dhist, hlen, info->iters);
        if (!st) st = hs;
    }
    for (cudaEvent_t e : ev)
        if (e) cudaEventDestroy(e);
    rs_free(ctx, V);
    rs_free(ctx, Z);
    rs_free(ctx, Aug);
    rs_free(ctx, r);
    rs_free(ctx, t);
    rs_free(ctx, d);
    info->status = st ? st : status;
    info->solve_s = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    return info->status;
}

extern "C" int rs_solve_gmres(const rs_mat *A, rs_pc *M, const rs_vec *b, rs_vec *x, int32_t restart,
                              double rtol, int32_t maxit, rs_solve_info *info)
{
    return gmres_impl(A, M, b, x, restart, 0, rtol, maxit, 0, info);
}

extern "C" int rs_solve_fgmres(const rs_mat *A, rs_pc *M, const rs_vec *b, rs_vec *x, int32_t restart,
                               double rtol, int32_t maxit, rs_solve_info *info)
{
    return gmres_impl(A, M, b, x, restart, 0, rtol, maxit, 1, info);
}

extern "C" int rs_solve_lgmres(const rs_mat *A, rs_pc *M, const rs_vec *b, rs_vec *x, int32_t restart,
                               int32_t aug_k, double rtol, int32_t maxit, rs_solve_info *info)
{
    return gmres_impl(A, M, b, x, restart, aug_k, rtol, maxit, 1, info);
}

// ---------------------------------------------------------------------------
// BiCGSTAB
// ---------------------------------------------------------------------------
struct BicgDev {
    double red[8];          // reduction outputs
    double rho, rho0, alpha, omega, beta, tol, bnorm, implicit;
    int iters, done, half, fresh, breakdown, maxit, status, pad;
    double *hist;           // residual history (device), hist_len entries
    int hist_len, pad_;
};

// generic fused row kernel with up to 3 dot products and a scalar epilogue
//  op 0: p = r + beta (p - omega v)                             (no dots)
//  op 1: s = r - alpha v;  red = {||s||^2}                       -> half-step test
//  op 2: x += alpha ph + omega sh; r = s - omega t; red = {(rh,r), ||r||^2}
//  op 3: red = {(rh, v)}                                        -> alpha
//  op 4: red = {(t, s), (t, t)}                                 -> omega
//  op 5: x += alpha ph (half-step exit)
__global__ void __launch_bounds__(RS_RED_THREADS)
k_bicg(int op, int n, double *p, double *r, const double *__restrict__ v, double *s,
       const double *__restrict__ t, double *x, const double *__restrict__ ph,
       const double *__restrict__ sh, const double *__restrict__ rh, double *partials,
       unsigned *ticket, BicgDev *d)
{
    if (rs_pdl_wait()) return;
    if (op != 5 && (*(volatile int *)&d->done || *(volatile int *)&d->half)) return;
    if (op == 5 && !*(volatile int *)&d->half) return;
    const double alpha = d->alpha, omega = d->omega, beta = d->beta;
    double acc[2] = {0.0, 0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        switch (op) {
        case 0: p[i] = fma(beta, fma(-omega, v[i], p[i]), r[i]); break;
        case 1: {
            const double si = fma(-alpha, v[i], r[i]);
            s[i] = si;
            acc[0] = fma(si, si, acc[0]);
            break;
        }
        case 2: {
            x[i] = fma(omega, sh[i], fma(alpha, ph[i], x[i]));
            const double ri = fma(-omega, t[i], s[i]);
            r[i] = ri;
            acc[0] = fma(rh[i], ri, acc[0]);
            acc[1] = fma(ri, ri, acc[1]);
            break;
        }
        case 3: acc[0] = fma(rh[i], v[i], acc[0]); break;
        case 4:
            acc[0] = fma(t[i], s[i], acc[0]);
            acc[1] = fma(t[i], t[i], acc[1]);
            break;
        case 5: x[i] = fma(alpha, ph[i], x[i]); break;
        }
    }
    if (op == 0) return;
    if (op == 5) {
        // the half-step update runs once: the last block to finish clears the flag
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            if (atomicAdd(ticket, 1u) == gridDim.x - 1) {
                d->half = 0;
                *ticket = 0;
                __threadfence();
            }
        }
        return;
    }
    const int nv = (op == 2 || op == 4) ? 2 : 1;
    if (!reduce_partials<2>(acc, nv, partials, ticket, d->red)) return;
    if (threadIdx.x != 0) return;
    switch (op) {
    case 1: {
        d->iters += 1;
        const double sn = sqrt(d->red[0]);
        if (sn <= d->tol) {
            d->half = 1; d->implicit = sn; d->done = 1; d->fresh = 1;
            record_hist(d->hist, d->hist_len, d->iters, sn, d->bnorm);
        }
        break;
    }
    case 2: {
        const double rho = d->red[0];
        const double rn = sqrt(d->red[1]);
        d->implicit = rn;
        record_hist(d->hist, d->hist_len, d->iters, rn, d->bnorm);
        d->rho0 = d->rho;
        if (rn <= d->tol) { d->done = 1; d->fresh = 1; break; }
        if (!(d->omega != 0.0) || !isfinite(d->omega)) { d->breakdown = 1; d->done = 1; break; }
        if (!(fabs(rho) > 0.0) || !isfinite(rho)) { d->breakdown = 1; d->done = 1; break; }
        d->beta = (rho / d->rho0) * (d->alpha / d->omega);
        d->rho = rho;
        if (d->iters >= d->maxit) d->done = 1;
        break;
    }
    case 3: {
        const double rv = d->red[0];
        if (!(fabs(rv) > 0.0) || !isfinite(rv)) { d->breakdown = 1; d->done = 1; break; }
        d->alpha = d->rho / rv;
        break;
    }
    case 4: {
        const double ts = d->red[0], tt = d->red[1];
        d->omega = tt > 0.0 ? ts / tt : 0.0;
        break;
    }
    }
}

// restart from the true residual r = b - A x (already in r, ||r||^2 in red[1])
__global__ void k_bicg_restart(int n, const double *__restrict__ r, double *rh, double *p, double *v,
                               BicgDev *d)
{
    if (rs_pdl_wait()) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        rh[i] = r[i];
        p[i] = 0.0;
        v[i] = 0.0;
    }
}

__global__ void k_bicg_restart_scalars(BicgDev *d, const double *r2)
{
    if (rs_pdl_wait()) return;
    if (threadIdx.x) return;
    const double rn = sqrt(*r2);
    d->implicit = rn;
    d->fresh = 0;
    d->half = 0;
    d->done = 0;
    if (rn <= d->tol) { d->done = 1; d->status = 1; return; }   // status 1: converged
    if (d->iters >= d->maxit) { d->done = 1; return; }
    // rho = (rh, r) = ||r||^2 with rh = r; beta multiplies p = 0, so its value is irrelevant
    d->rho0 = 1.0;
    d->alpha = 1.0;
    d->omega = 1.0;
    d->rho = *r2;
    d->beta = 0.0;
    if (!(d->rho > 0.0) || !isfinite(d->rho)) { d->breakdown = 1; d->done = 1; }
}

extern "C" int rs_solve_bicgstab(const rs_mat *A, rs_pc *M, const rs_vec *bv, rs_vec *xv, double rtol,
                                 int32_t maxit, rs_solve_info *info)
{
    if (!A || !bv || !xv || !info) return RS_ERR_INVALID_ARG;
    if (maxit < 0 || !(rtol >= 0)) return RS_ERR_INVALID_ARG;
    if (bv->n != A->n || xv->n != A->n) return RS_ERR_SIZE_MISMATCH;
    memset(info, 0, sizeof(*info));
    info->bad_row = -1;
    rs_ctx *ctx = A->ctx;
    const auto t0 = std::chrono::steady_clock::now();
    const int n = A->n;
    const int ld = (n + 31) / 32 * 32;
    double *buf = nullptr;
    BicgDev *d = nullptr;
    double *dhist = nullptr;
    int hlen = 0;
    int st = rs_alloc(ctx, (void **)&buf, sizeof(double) * (size_t)ld * 8);
    if (!st) st = rs_alloc(ctx, (void **)&d, sizeof(BicgDev));
    if (!st) st = hist_begin(ctx, &dhist, &hlen);
    int status = RS_NOT_CONVERGED;
    double bnorm = 0.0;
    const double *b = bv->d;
    double *x = xv->d;
    double *r = buf, *rh = buf + ld, *p = buf + 2 * (size_t)ld, *v = buf + 3 * (size_t)ld;
    double *s = buf + 4 * (size_t)ld, *t = buf + 5 * (size_t)ld, *ph = buf + 6 * (size_t)ld;
    double *sh = buf + 7 * (size_t)ld;
    if (!M) {            // no preconditioner: M^{-1} p = p, M^{-1} s = s
        ph = p;
        sh = s;
    }
    if (st) goto out;
    {
        st = rs_dot_launch(ctx, n, b, b, ctx->d_scalars);
        if (st) goto out;
        cudaMemcpyAsync(ctx->h_pinned, ctx->d_scalars, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream);
        if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) { st = RS_ERR_CUDA; goto out; }
        bnorm = sqrt(ctx->h_pinned[0]);
        if (bnorm == 0.0) {
            cudaMemsetAsync(x, 0, sizeof(double) * n, ctx->stream);
            status = RS_OK;
            goto done;
        }
        BicgDev h0;
        memset(&h0, 0, sizeof(h0));
        h0.tol = rtol * bnorm;
        h0.bnorm = bnorm;
        h0.maxit = maxit;
        h0.hist = dhist;
        h0.hist_len = hlen;
        cudaMemcpyAsync(d, &h0, sizeof(h0), cudaMemcpyHostToDevice, ctx->stream);
        const int gr = red_grid(ctx, n, RS_RED_THREADS), gb = blas_grid(ctx, n);
        int *halt = &d->done;
        const int batch = 8;
        for (;;) {
            // (re)start from the true residual
            st = rs_residual_launch(A, b, x, r, &d->red[1], nullptr);
            if (st) goto out;
            rs_pdl(k_bicg_restart, gb, 256, 0, ctx)(n, r, rh, p, v, d);
            rs_pdl(k_bicg_restart_scalars, 1, 32, 0, ctx)(d, &d->red[1]);
            ctx->launches += 2;
            bool restart = false;
            while (!restart) {
                for (int it = 0; it < batch; ++it) {
                    {
                        RsProfScope prof(ctx, RS_PROF_BLAS1);
                        rs_pdl(k_bicg, gr, RS_RED_THREADS, 0, ctx)(0, n, p, r, v, s, t, x, ph, sh, rh,
                                                                       ctx->red_partials, ctx->red_ticket, d);
                    }
                    ctx->launches++;
                    if (M) st = rs_pc_apply_dev(M, p, ph, halt);
                    if (st) goto out;
                    st = rs_spmv_launch(A, ph, 1.0, 0.0, v, halt);
                    if (st) goto out;
                    {
                        RsProfScope prof(ctx, RS_PROF_BLAS1);
                        rs_pdl(k_bicg, gr, RS_RED_THREADS, 0, ctx)(3, n, p, r, v, s, t, x, ph, sh, rh,
                                                                       ctx->red_partials, ctx->red_ticket, d);
                    }
                    {
                        RsProfScope prof(ctx, RS_PROF_BLAS1);
                        rs_pdl(k_bicg, gr, RS_RED_THREADS, 0, ctx)(1, n, p, r, v, s, t, x, ph, sh, rh,
                                                                       ctx->red_partials, ctx->red_ticket, d);
                    }
                    {
                        RsProfScope prof(ctx, RS_PROF_BLAS1);
                        rs_pdl(k_bicg, gr, RS_RED_THREADS, 0, ctx)(5, n, p, r, v, s, t, x, ph, sh, rh,
                                                                       ctx->red_partials, ctx->red_ticket, d);
                    }
                    ctx->launches += 3;
                    if (M) st = rs_pc_apply_dev(M, s, sh, halt);
                    if (st) goto out;
                    st = rs_spmv_launch(A, sh, 1.0, 0.0, t, halt);
                    if (st) goto out;
                    {
                        RsProfScope prof(ctx, RS_PROF_BLAS1);
                        rs_pdl(k_bicg, gr, RS_RED_THREADS, 0, ctx)(4, n, p, r, v, s, t, x, ph, sh, rh,
                                                                       ctx->red_partials, ctx->red_ticket, d);
                    }
                    {
                        RsProfScope prof(ctx, RS_PROF_BLAS1);
                        rs_pdl(k_bicg, gr, RS_RED_THREADS, 0, ctx)(2, n, p, r, v, s, t, x, ph, sh, rh,
                                                                       ctx->red_partials, ctx->red_ticket, d);
                    }
                    ctx->launches += 2;
                }
                BicgDev hd;
                if (cudaMemcpyAsync(&hd, d, sizeof(hd), cudaMemcpyDeviceToHost, ctx->stream) != cudaSuccess ||
                    cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
                    st = RS_ERR_CUDA;
                    goto out;
                }
                info->iters = hd.iters;
                info->implicit_rel_res = hd.implicit / bnorm;
                if (hd.status == 1) { status = RS_OK; goto done; }
                if (hd.breakdown) { status = RS_ERR_BREAKDOWN; goto done; }
                if (hd.fresh) { restart = true; break; }       // confirm with the true residual
                if (hd.done || hd.iters >= maxit) { status = RS_NOT_CONVERGED; goto done; }
            }
        }
    }
done:
    st = rs_collect_device_error(ctx, &info->bad_row);
    if (st) goto out;
    st = finish_info(ctx, A, b, x, r, bnorm, info);
    if (st) goto out;
    if (status == RS_OK && info->true_rel_res > rtol && bnorm > 0) status = RS_NOT_CONVERGED;
    if (status == RS_NOT_CONVERGED && info->true_rel_res <= rtol && bnorm > 0) status = RS_OK;
out:
    {
        const int hs = hist_end(ctx, dhist, hlen, info->iters);
        if (!st) st = hs;
    }
    rs_free(ctx, buf);
    rs_free(ctx, d);
    info->status = st ? st : status;
    info->solve_s = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    return info->status;
}

// ---------------------------------------------------------------------------
// Preconditioned conjugate gradient (Alg. 2), device-resident like BiCGSTAB:
// the scalars live in device memory and the last block of each reduction
// forms beta or alpha; the host synchronises once per batch of iterations.
// ---------------------------------------------------------------------------
struct CgDev {
    double red[2];
    double rho, rho0, alpha, beta, tol, bnorm, implicit;
    int iters, done, fresh, breakdown, maxit, status, first, pad;
    double *hist;           // residual history (device), hist_len entries
    int hist_len, pad_;
};

//  op 0: red = {(r, z)}                 -> rho, beta = rho / rho_prev (0 on the first pass)
//  op 1: p = z + beta p
//  op 2: red = {(p, q)}                 -> alpha = rho / (p, q)
//  op 3: x += alpha p; r -= alpha q; red = {||r||^2} -> convergence test
__global__ void __launch_bounds__(RS_RED_THREADS)
k_cg(int op, int n, double *x, double *r, const double *__restrict__ z, double *p,
     const double *__restrict__ q, double *partials, unsigned *ticket, CgDev *d)
{
    if (rs_pdl_wait()) return;
    if (*(volatile int *)&d->done) return;
    const double alpha = d->alpha, beta = d->beta;
    double acc[1] = {0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        switch (op) {
        case 0: acc[0] = fma(r[i], z[i], acc[0]); break;
        case 1: p[i] = fma(beta, p[i], z[i]); break;
        case 2: acc[0] = fma(p[i], q[i], acc[0]); break;
        case 3: {
            x[i] = fma(alpha, p[i], x[i]);
            const double ri = fma(-alpha, q[i], r[i]);
            r[i] = ri;
            acc[0] = fma(ri, ri, acc[0]);
            break;
        }
        }
    }
    if (op == 1) return;
    if (!reduce_partials<1>(acc, 1, partials, ticket, d->red)) return;
    if (threadIdx.x != 0) return;
    switch (op) {
    case 0: {
        const double rho = d->red[0];
        if (!(rho != 0.0) || !isfinite(rho)) { d->breakdown = 1; d->done = 1; break; }
        d->beta = d->first ? 0.0 : rho / d->rho0;
        d->first = 0;
        d->rho = rho;
        break;
    }
    case 2: {
        const double pq = d->red[0];
        if (!(pq > 0.0) || !isfinite(pq)) { d->breakdown = 1; d->done = 1; break; }
        d->alpha = d->rho / pq;
        break;
    }
    case 3: {
        d->iters += 1;
        d->rho0 = d->rho;
        const double rn = sqrt(d->red[0]);
        d->implicit = rn;
        record_hist(d->hist, d->hist_len, d->iters, rn, d->bnorm);
        if (rn <= d->tol) { d->done = 1; d->fresh = 1; break; }
        if (d->iters >= d->maxit) d->done = 1;
        break;
    }
    }
}

// restart from the true residual (in r, ||r||^2 in *r2): p = 0, first pass
__global__ void k_cg_restart(int n, double *p, CgDev *d, const double *r2)
{
    if (rs_pdl_wait()) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) p[i] = 0.0;
    if (blockIdx.x || threadIdx.x) return;
    const double rn = sqrt(*r2);
    d->implicit = rn;
    d->fresh = 0;
    d->done = 0;
    d->first = 1;
    d->beta = 0.0;
    if (rn <= d->tol) { d->done = 1; d->status = 1; return; }   // status 1: converged
    if (d->iters >= d->maxit) d->done = 1;
}

extern "C" int rs_solve_cg(const rs_mat *A, rs_pc *M, const rs_vec *bv, rs_vec *xv, double rtol, int32_t maxit,
                           rs_solve_info *info)
{
    if (!A || !bv || !xv || !info) return RS_ERR_INVALID_ARG;
    if (maxit < 0 || !(rtol >= 0)) return RS_ERR_INVALID_ARG;
    if (bv->n != A->n || xv->n != A->n) return RS_ERR_SIZE_MISMATCH;
    memset(info, 0, sizeof(*info));
    info->bad_row = -1;
    rs_ctx *ctx = A->ctx;
    const auto t0 = std::chrono::steady_clock::now();
    const int n = A->n;
    const int ld = (n + 31) / 32 * 32;
    double *buf = nullptr;
    CgDev *d = nullptr;
    double *dhist = nullptr;
    int hlen = 0;
    int st = rs_alloc(ctx, (void **)&buf, sizeof(double) * (size_t)ld * 4);
    if (!st) st = rs_alloc(ctx, (void **)&d, sizeof(CgDev));
    if (!st) st = hist_begin(ctx, &dhist, &hlen);
    int status = RS_NOT_CONVERGED;
    double bnorm = 0.0;
    const double *b = bv->d;
    double *x = xv->d;
    double *r = buf, *z = buf + ld, *p = buf + 2 * (size_t)ld, *q = buf + 3 * (size_t)ld;
    if (!M) z = r;       // no preconditioner: z = r
    if (st) goto out;
    {
        st = rs_dot_launch(ctx, n, b, b, ctx->d_scalars);
        if (st) goto out;
        cudaMemcpyAsync(ctx->h_pinned, ctx->d_scalars, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream);
        if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) { st = RS_ERR_CUDA; goto out; }
        bnorm = sqrt(ctx->h_pinned[0]);
        if (bnorm == 0.0) {
            cudaMemsetAsync(x, 0, sizeof(double) * n, ctx->stream);
            status = RS_OK;
            goto done;
        }
        CgDev h0;
        memset(&h0, 0, sizeof(h0));
        h0.tol = rtol * bnorm;
        h0.bnorm = bnorm;
        h0.maxit = maxit;
        h0.hist = dhist;
        h0.hist_len = hlen;
        cudaMemcpyAsync(d, &h0, sizeof(h0), cudaMemcpyHostToDevice, ctx->stream);
        const int gr = red_grid(ctx, n, RS_RED_THREADS), gb = blas_grid(ctx, n);
        int *halt = &d->done;
        const int batch = 8;
        for (;;) {
            st = rs_residual_launch(A, b, x, r, &d->red[1], nullptr);
            if (st) goto out;
            rs_pdl(k_cg_restart, gb, 256, 0, ctx)(n, p, d, &d->red[1]);
            ctx->launches++;
            bool restart = false;
            while (!restart) {
                for (int it = 0; it < batch; ++it) {
                    if (M) st = rs_pc_apply_dev(M, r, z, halt);
                    if (st) goto out;
                    {
                        RsProfScope prof(ctx, RS_PROF_BLAS1);
                        rs_pdl(k_cg, gr, RS_RED_THREADS, 0, ctx)(0, n, x, r, z, p, q, ctx->red_partials,
                                                                     ctx->red_ticket, d);
                    }
                    {
                        RsProfScope prof(ctx, RS_PROF_BLAS1);
                        rs_pdl(k_cg, gb, RS_RED_THREADS, 0, ctx)(1, n, x, r, z, p, q, ctx->red_partials,
                                                                     ctx->red_ticket, d);
                    }
                    ctx->launches += 2;
                    st = rs_spmv_launch(A, p, 1.0, 0.0, q, halt);
                    if (st) goto out;
                    {
                        RsProfScope prof(ctx, RS_PROF_BLAS1);
                        rs_pdl(k_cg, gr, RS_RED_THREADS, 0, ctx)(2, n, x, r, z, p, q, ctx->red_partials,
                                                                     ctx->red_ticket, d);
                    }
                    {
                        RsProfScope prof(ctx, RS_PROF_BLAS1);
                        rs_pdl(k_cg, gr, RS_RED_THREADS, 0, ctx)(3, n, x, r, z, p, q, ctx->red_partials,
                                                                     ctx->red_ticket, d);
                    }
                    ctx->launches += 2;
                }
                CgDev hd;
                if (cudaMemcpyAsync(&hd, d, sizeof(hd), cudaMemcpyDeviceToHost, ctx->stream) != cudaSuccess ||
                    cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
                    st = RS_ERR_CUDA;
                    goto out;
                }
                info->iters = hd.iters;
                info->implicit_rel_res = hd.implicit / bnorm;
                if (hd.status == 1) { status = RS_OK; goto done; }
                if (hd.breakdown) { status = RS_ERR_BREAKDOWN; goto done; }
                if (hd.fresh) { restart = true; break; }       // confirm with the true residual
                if (hd.done || hd.iters >= maxit) { status = RS_NOT_CONVERGED; goto done; }
            }
        }
    }
done:
    st = rs_collect_device_error(ctx, &info->bad_row);
    if (st) goto out;
    st = finish_info(ctx, A, b, x, r, bnorm, info);
    if (st) goto out;
    if (status == RS_OK && info->true_rel_res > rtol && bnorm > 0) status = RS_NOT_CONVERGED;
    if (status == RS_NOT_CONVERGED && info->true_rel_res <= rtol && bnorm > 0) status = RS_OK;
out:
    {
        const int hs = hist_end(ctx, dhist, hlen, info->iters);
        if (!st) st = hs;
    }
    rs_free(ctx, buf);
    rs_free(ctx, d);
    info->status = st ? st : status;
    info->solve_s = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    return info->status;
}
