// Triangular sweeps of small structured grids in one block.
//
// On a small grid the wavefront sweeps of rs_wave.cu are all latency: four
// launches, units that hand values to each other through L2 (about 2 us a
// hop) and 500 cycles a step.  Here one block solves L y = r and U z = y
// (Eq. 3) in one launch.  The cells of a wavefront x + y + z = h do not read
// one another, so the block takes the wavefronts in turn with a barrier
// between them, a thread per scalar row, the values in shared memory.
//
// What bounds it is the length of a step (a thread's instructions, the
// shared-memory latency, the FP64 multiply-adds of one SM, the barrier), so
// everything that can be is out of it:
//   - the values lie on the grid padded by a zero cell per line, line per
//     plane and two planes, so a row reads its three neighbours at fixed
//     distances and none is tested for;
//   - the records (a row's place, its L or U entries) come in chunks of one
//     size for both sweeps, a wavefront each, idle threads marked by place -1; a thread reads
//     its next one into registers before the barrier;
//   - they stream through a ring of shared-memory slots, two or four
//     wavefronts a slot and copy.  A producer warp waits for the copies and
//     joins the barrier once per slot, which also tells it which one is free
//     (joining every step, its own 0.3 us set the pace).
//
// Arithmetic: that of the wavefront sweeps, operation for operation (L in
// ascending column order; U premultiplied by D_i, sum_j D y_j, then the z, x
// and y neighbours; cells outside the grid count as 0), so the results are
// the same bit for bit.
#include <algorithm>
#include <vector>

#include "rs_internal.cuh"

namespace {

constexpr int LV_MIN_SLOTS = 3, LV_MAX_SLOTS = 8;   // groups of wavefronts in the ring
constexpr int LV_MAX_LEVELS = 1024;
constexpr int LV_MAX_ROWS = 992;                    // compute threads; one more warp produces
constexpr int LV_IO_THREADS = 512;                  // threads that move r in and z out, at least
constexpr int LV_HDR = 128;                         // mbarriers
constexpr size_t LV_SMEM = 220 * 1024;
constexpr long long LV_DRAIN = 1LL << 30;           // cycles a late copy is still waited for

struct LevelArgs {
    int n, nx, nxy, nlev;                           // cells, strides, wavefronts
    int group, ngroup;                              // wavefronts a slot (2 or 4), slots a sweep
    int wc;                                         // cells per chunk (the widest wavefront, a multiple of 4)
    int nt;                                         // compute threads: the rows of a chunk, rounded up to 32
    int px, pxy, ncell;                             // strides and cells of the padded grid
    int nslots;
    const int *place;                               // [n] padded cell of each natural row
    int *err;
    long long limit;
    const int *skip;
};

// Bytes of a chunk: a place per cell, then the block rows of BS values per row,
// 4 of U, 3 of L (the fourth is left out).  One size for both, so that a ring slot
// has its places at the same offsets whatever it holds: a copy that has been
// given up on, or lands later than that, leaves there the -1 of the start or places of
// the grid, never a value's bits.  (A test of every place before its use took
// 0.4 to 1 us of an apply's 13 to 42, in the steps' chain; L's larger copies take none.)
template <int BS, typename T>
__host__ __device__ __forceinline__ int lv_plane(int wc) { return wc * BS * (int)sizeof(T); }
template <int BS, typename T>
__host__ __device__ __forceinline__ int lv_chunk(int wc) { return 4 * wc + 4 * BS * lv_plane<BS, T>(wc); }
// bytes of a value array on the padded grid; blocks keep y and z apart, since
// a cell's rows all read its y
template <int BS, typename T>
__host__ __device__ __forceinline__ int lv_values(int ncell) { return (ncell * BS * (int)sizeof(T) + 15) & ~15; }

// one sweep's wavefronts; q: this thread's record of the first one, already read
template <int BS, typename T, bool LOWER>
struct LevelRec {
    static constexpr int NV = (LOWER ? 3 : 4) * BS;
    int e;                                          // padded cell, or -1
    T v[NV];
    __device__ __forceinline__ void load(const unsigned char *slot, int cell, int row, int wc, int ps)
    {
        e = ((const int *)slot)[cell];
        const T *p = (const T *)(slot + 4 * wc) + row;
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] = *(const T *)((const unsigned char *)p + k * ps);
    }
    __device__ __forceinline__ void solve(T *yv, T *zv, int i, int px, int pxy) const
    {
        T *dst = (LOWER ? yv : zv) + e * BS;
        const T *nz = dst + (LOWER ? -pxy : pxy) * BS, *ny = dst + (LOWER ? -px : px) * BS, *nx = dst + (LOWER ? -BS : BS);
        T acc, a[BS], b[BS], c[BS];
#pragma unroll
        for (int j = 0; j < BS; ++j) {
            a[j] = nz[j];
            b[j] = LOWER ? ny[j] : nx[j];
            c[j] = LOWER ? nx[j] : ny[j];
        }
        if (LOWER) {
            acc = yv[e * BS + i];
        } else {
            acc = T(0);
#pragma unroll
            for (int j = 0; j < BS; ++j) acc = mad(v[3 * BS + j], yv[e * BS + j], acc);
        }
#pragma unroll
        for (int j = 0; j < BS; ++j) acc = msub(acc, v[j], a[j]);
#pragma unroll
        for (int j = 0; j < BS; ++j) acc = msub(acc, v[BS + j], b[j]);
#pragma unroll
        for (int j = 0; j < BS; ++j) acc = msub(acc, v[2 * BS + j], c[j]);
        dst[i] = acc;
    }
};

template <int BS, typename T>
__global__ void __launch_bounds__(LV_MAX_ROWS + 32)
k_level_solve(LevelArgs g, const unsigned char *__restrict__ lbuf, const unsigned char *__restrict__ ubuf,
              const double *__restrict__ r, const double *__restrict__ scale, double *__restrict__ z)
{
    extern __shared__ __align__(128) unsigned char lv_smem[];
    unsigned long long *full = (unsigned long long *)lv_smem;
    const int vbytes = lv_values<BS, T>(g.ncell);
    T *yv = (T *)(lv_smem + LV_HDR), *zv = BS > 1 ? (T *)(lv_smem + LV_HDR + vbytes) : yv;
    unsigned char *ring = lv_smem + LV_HDR + (BS > 1 ? 2 : 1) * vbytes;
    const int cb = lv_chunk<BS, T>(g.wc), sb = g.group * cb;      // bytes of a chunk and of a slot
    // threads: nt compute, then helpers that only move r and z (up to nio in
    // all), then the producer warp
    const int nt = g.nt, nio = blockDim.x - 32, tid = threadIdx.x;
    if (tid == 0) {
        for (int s = 0; s < g.nslots; ++s) mbar_init(&full[s], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the padding to 0, and the places of every slot's chunks to -1
    for (int k = tid; k < (BS > 1 ? 2 : 1) * vbytes / 16; k += blockDim.x) ((uint4 *)yv)[k] = make_uint4(0, 0, 0, 0);
    if (tid < g.wc)
        for (int sl = 0; sl < g.nslots; ++sl)
            for (int w = 0; w < g.group; ++w) ((int *)(ring + sl * sb + w * cb))[tid] = -1;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (rs_pdl_wait()) return;
    if (g.skip && *(volatile const int *)g.skip) return;
    __syncthreads();
    const int groups = 2 * g.ngroup;
    if (tid >= nio) {
        // producer: group j goes to slot j mod nslots
        const int lane = tid - nio;
        int ij = 0, isl = 0, wsl = 0;                // next group to copy, its slot; slot of the next one to wait for
        unsigned wph = 0;
        const unsigned char *src = lbuf;
        auto issue = [&]() {
            mbar_arrive_expect_tx(&full[isl], sb);
            bulk_g2s(ring + isl * sb, src, sb, &full[isl]);
            src += sb;
            if (++ij == g.ngroup) src = ubuf;
            if (++isl == g.nslots) isl = 0;
        };
        // bounded: a wait longer than the limit, however short the limit, is
        // recorded as a timeout; given up only much later
        bool dead = false;
        auto arrived = [&]() {
            unsigned long long *b = &full[wsl];
            const unsigned par = wph;
            if (++wsl == g.nslots) {
                wsl = 0;
                wph ^= 1;
            }
            if (dead) return;
            const long long t0 = clock64(), giveup = 4 * g.limit + LV_DRAIN;
            bool late = false;
            for (;;) {
                const bool in = mbar_try_wait(b, par);
                const long long dt = clock64() - t0;
                if (!late && dt > g.limit) {
                    late = true;
                    atomicOr(g.err, RS_DEVERR_TIMEOUT);
                }
                if (in) break;
                if (dt > giveup) {
                    dead = true;
                    break;
                }
            }
        };
        if (lane == 0) {
            for (int j = 0; j < min(g.nslots, groups); ++j) issue();
            arrived();
        }
        __syncthreads();
        // the barrier at the end of group j's first step: group j + 1 has
        // arrived, and group j - 1 has been read
        for (int j = 0; j < groups; ++j) {
            if (lane == 0 && j + 1 < groups) arrived();
            __syncwarp();
            asm volatile("bar.sync 1, %0;" ::"r"(nt + 32) : "memory");
            if (lane == 0 && j > 0 && ij < groups && !dead) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                issue();
            }
        }
        return;
    }
    {
        const double sc = scale ? *scale : 1.0;
        constexpr int U = BS == 1 ? 8 : 2;          // cells whose loads are in flight together
        for (int i0 = tid; i0 < g.n; i0 += U * nio) {
            int e[U];
            double v[U][BS];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = min(i0 + u * nio, g.n - 1);
                e[u] = __ldg(g.place + i);
#pragma unroll
                for (int j = 0; j < BS; ++j) v[u][j] = __ldg(r + (size_t)i * BS + j);
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + u * nio < g.n) {
#pragma unroll
                    for (int j = 0; j < BS; ++j) yv[e[u] * BS + j] = (T)(sc == 1.0 ? v[u][j] : v[u][j] * sc);
                }
        }
    }
    const int cell = tid / BS, i = tid - cell * BS, ps = lv_plane<BS, T>(g.wc);
    const bool in = cell < g.wc;
    const unsigned char *slot = ring, *end = ring + g.nslots * sb;
    __syncthreads();                                // r and the first group are in place
    if (tid < nt) {
        LevelRec<BS, T, true> ql;
        LevelRec<BS, T, false> qu;
        ql.e = qu.e = -1;
        auto barrier = [&](bool first) {                // with the producer at a group's first step
            if (first) asm volatile("bar.sync 1, %0;" ::"r"(nt + 32) : "memory");
            else asm volatile("bar.sync 2, %0;" ::"r"(nt) : "memory");
        };
        auto advance = [&]() {
            slot += sb;
            if (slot == end) slot = ring;
        };
        if (in) ql.load(slot, cell, tid, g.wc, ps);
        for (int j = 0; j < g.ngroup; ++j) {
            const unsigned char *c = slot;
            for (int k = 1; k < g.group; ++k) {
                if (ql.e >= 0) ql.solve(yv, zv, i, g.px, g.pxy);
                c += cb;
                if (in) ql.load(c, cell, tid, g.wc, ps);
                barrier(k == 1);
            }
            if (ql.e >= 0) ql.solve(yv, zv, i, g.px, g.pxy);
            advance();
            if (in) {
                if (j + 1 < g.ngroup) ql.load(slot, cell, tid, g.wc, ps);
                else qu.load(slot, cell, tid, g.wc, ps);
            }
            barrier(false);
        }
        for (int j = 0; j < g.ngroup; ++j) {
            const unsigned char *c = slot;
            for (int k = 1; k < g.group; ++k) {
                if (qu.e >= 0) qu.solve(yv, zv, i, g.px, g.pxy);
                c += cb;
                if (in) qu.load(c, cell, tid, g.wc, ps);
                barrier(k == 1);
            }
            if (qu.e >= 0) qu.solve(yv, zv, i, g.px, g.pxy);
            advance();
            if (in && j + 1 < g.ngroup) qu.load(slot, cell, tid, g.wc, ps);
            barrier(false);
        }
    }
    asm volatile("bar.sync 3, %0;" ::"r"(nio) : "memory");
    constexpr int U = 8;
    for (int k0 = tid; k0 < g.n; k0 += U * nio) {
        int e[U];
#pragma unroll
        for (int u = 0; u < U; ++u) e[u] = __ldg(g.place + min(k0 + u * nio, g.n - 1));
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (k0 + u * nio < g.n) {
#pragma unroll
                for (int j = 0; j < BS; ++j) z[(size_t)(k0 + u * nio) * BS + j] = (double)zv[e[u] * BS + j];
            }
    }
}

// The chunks of both triangles from the FP64 factor in the matrix pattern, as
// in k_wave_gather: L_z, L_y, L_x of each row; D_i U_ij for the z, x and y
// neighbours and D_i = inv(U_ii).  A thread per cell in wavefront order
// (slot: its place in its wavefront); U's chunks lie in its own order (last
// wavefront first).  Places outside a wavefront were set to -1, values to 0.
template <int BS, typename T>
__global__ void k_level_gather(LevelArgs g, int ny, const int2 *__restrict__ cells, const int *__restrict__ ptr,
                               const int *__restrict__ col, const int *__restrict__ diagpos,
                               const double *__restrict__ lu, const double *__restrict__ dinv,
                               unsigned char *__restrict__ lbuf, unsigned char *__restrict__ ubuf)
{
    constexpr int B2 = BS * BS;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.n) return;
    const int i = cells[t].x, p = cells[t].y;
    const int h = i % g.nx + (i / g.nx) % ny + i / g.nxy;
    unsigned char *lc = lbuf + (size_t)h * lv_chunk<BS, T>(g.wc);
    unsigned char *uc = ubuf + (size_t)(g.nlev - 1 - h) * lv_chunk<BS, T>(g.wc);
    ((int *)lc)[p] = ((int *)uc)[p] = g.place[i];
    const int ps = lv_plane<BS, T>(g.wc);
    auto put = [&](unsigned char *c, int blk, int a, int b, double v) {
        ((T *)(c + 4 * g.wc + (size_t)(blk * BS + b) * ps))[p * BS + a] = (T)v;
    };
    double D[B2];
    if (BS == 1) {
        D[0] = 1.0 / lu[diagpos[i]];
    } else {
#pragma unroll
        for (int k = 0; k < B2; ++k) D[k] = dinv[(size_t)i * B2 + k];
    }
    for (int blk = 0; blk < 3; ++blk)
#pragma unroll
        for (int a = 0; a < BS; ++a)
#pragma unroll
            for (int b = 0; b < BS; ++b) {
                put(lc, blk, a, b, 0.0);
                put(uc, blk, a, b, 0.0);
            }
#pragma unroll
    for (int a = 0; a < BS; ++a)
#pragma unroll
        for (int b = 0; b < BS; ++b) put(uc, 3, a, b, D[a * BS + b]);
    for (int q = ptr[i]; q < ptr[i + 1]; ++q) {
        const int d = col[q] - i;
        const double *av = lu + (size_t)q * B2;
        const int ls = d == -g.nxy ? 0 : d == -g.nx ? 1 : d == -1 ? 2 : -1;
        const int us = d == g.nxy ? 0 : d == 1 ? 1 : d == g.nx ? 2 : -1;
        if (ls >= 0) {
#pragma unroll
            for (int a = 0; a < BS; ++a)
#pragma unroll
                for (int b = 0; b < BS; ++b) put(lc, ls, a, b, av[a * BS + b]);
        } else if (us >= 0) {
#pragma unroll
            for (int a = 0; a < BS; ++a)
#pragma unroll
                for (int b = 0; b < BS; ++b) {
                    double s = 0.0;
#pragma unroll
                    for (int m = 0; m < BS; ++m) s = __dadd_rn(s, __dmul_rn(D[a * BS + m], av[m * BS + b]));
                    put(uc, us, a, b, s);
                }
        }
    }
}

// idle places: -1 in every chunk's places, 0 elsewhere
__global__ void k_level_clear(int64_t nwords, int chunk_words, int wc, int *__restrict__ buf)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nwords; k += (int64_t)gridDim.x * blockDim.x)
        buf[k] = k % chunk_words < wc ? -1 : 0;
}

LevelArgs level_args(const IluFactor *f, const int *skip)
{
    const WaveLayout &W = f->W;
    LevelArgs g;
    g.n = W.nx * W.ny * W.nz;
    g.nx = W.nx;
    g.nxy = W.nx * W.ny;
    g.nlev = W.nx + W.ny + W.nz - 2;
    g.wc = W.one_wc;
    g.nt = W.one_threads;
    g.px = W.nx + 1;
    g.pxy = g.px * (W.ny + 1);
    g.ncell = g.pxy * (W.nz + 2);
    g.nslots = W.one_nslots;
    g.group = W.one_group;
    g.ngroup = (g.nlev + g.group - 1) / g.group;
    g.place = W.one_place;
    g.err = f->ctx->d_err;
    g.limit = f->ctx->spin_limit;
    g.skip = skip;
    return g;
}

// cells on each wavefront
std::vector<int> level_sizes(int nx, int ny, int nz)
{
    std::vector<int> w(nx + ny + nz - 2, 0);
    for (int z = 0; z < nz; ++z)
        for (int y = 0; y < ny; ++y) {       // +1 on [y + z, y + z + nx): differences, summed below
            ++w[y + z];
            if (y + z + nx < (int)w.size()) --w[y + z + nx];
        }
    for (size_t h = 1; h < w.size(); ++h) w[h] += w[h - 1];
    return w;
}

int widest(const std::vector<int> &w) { return (*std::max_element(w.begin(), w.end()) + 3) & ~3; }

// wavefronts a slot and slots that fit beside the values; 0 slots: too few
template <int BS, typename T>
int lv_slots(int64_t ncell, int wc, int *group)
{
    if (ncell * BS * (int64_t)sizeof(T) > (int64_t)LV_SMEM) return 0;
    const size_t fixed = LV_HDR + (BS > 1 ? 2 : 1) * (size_t)lv_values<BS, T>((int)ncell);
    if (fixed >= LV_SMEM) return 0;
    for (*group = 4; *group >= 2; *group /= 2) {
        const size_t ns = (LV_SMEM - fixed) / (*group * lv_chunk<BS, T>(wc));
        if (ns >= LV_MIN_SLOTS) return (int)std::min<size_t>(ns, LV_MAX_SLOTS);
    }
    return 0;
}

template <int BS, typename T>
int level_create(IluFactor *f, const std::vector<int> &w)
{
    rs_ctx *ctx = f->ctx;
    WaveLayout &W = f->W;
    const int nx = W.nx, ny = W.ny, nz = W.nz, n = nx * ny * nz, nlev = (int)w.size();
    W.one_wc = widest(w);
    W.one_nslots = lv_slots<BS, T>((int64_t)(nx + 1) * (ny + 1) * (nz + 2), W.one_wc, &W.one_group);
    const LevelArgs g = level_args(f, nullptr);
    W.one_threads = (W.one_wc * BS + 31) / 32 * 32;
    std::vector<int> place(n), at(nlev, 0);
    std::vector<int2> cells(n);
    for (int z = 0, i = 0; z < nz; ++z)
        for (int y = 0; y < ny; ++y)
            for (int x = 0; x < nx; ++x, ++i) {
                place[i] = x + g.px * y + g.pxy * (z + 1);     // one zero plane before, one after
                cells[i] = make_int2(i, at[x + y + z]++);
            }
    const int64_t chunks = (int64_t)g.ngroup * g.group;    // the last group filled up with empty ones
    const int64_t words = chunks * lv_chunk<BS, T>(W.one_wc) / 4;
    int st = rs_alloc(ctx, (void **)&W.one_place, sizeof(int) * n);
    st = st ? st : rs_alloc(ctx, (void **)&W.one_cells, sizeof(int2) * n);
    st = st ? st : rs_alloc(ctx, &W.lrec, 4 * (size_t)words);
    st = st ? st : rs_alloc(ctx, &W.urec, 4 * (size_t)words);
    if (st) return st;
    RS_CUDA_TRY(cudaMemcpyAsync(W.one_place, place.data(), sizeof(int) * n, cudaMemcpyHostToDevice, ctx->stream));
    RS_CUDA_TRY(cudaMemcpyAsync(W.one_cells, cells.data(), sizeof(int2) * n, cudaMemcpyHostToDevice, ctx->stream));
    k_level_clear<<<256, 256, 0, ctx->stream>>>(words, lv_chunk<BS, T>(W.one_wc) / 4, W.one_wc, (int *)W.lrec);
    k_level_clear<<<256, 256, 0, ctx->stream>>>(words, lv_chunk<BS, T>(W.one_wc) / 4, W.one_wc, (int *)W.urec);
    ctx->launches += 1;
    RS_TRY(rs_check_launch(ctx));
    RS_CUDA_TRY(cudaStreamSynchronize(ctx->stream));        // the host arrays end here
    W.on = W.one = 1;
    return RS_OK;
}

template <int BS, typename T>
int level_gather(IluFactor *f)
{
    const WaveLayout &W = f->W;
    const LevelArgs g = level_args(f, nullptr);
    k_level_gather<BS, T><<<(g.n + 127) / 128, 128, 0, f->ctx->stream>>>(
        g, W.ny, W.one_cells, f->ptr, f->col, f->diagpos, f->lu, f->dinv, (unsigned char *)W.lrec,
        (unsigned char *)W.urec);
    return rs_check_launch(f->ctx);
}

template <int BS, typename T>
int level_apply(IluFactor *f, const double *r, double *z, const double *scale, const int *skip)
{
    rs_ctx *ctx = f->ctx;
    const WaveLayout &W = f->W;
    static unsigned long long raised = 0;      // one bit per device
    const unsigned long long bit = 1ull << (ctx->device & 63);
    if (!(raised & bit)) {
        RS_CUDA_TRY(cudaFuncSetAttribute(k_level_solve<BS, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LV_SMEM));
        raised |= bit;
    }
    const LevelArgs g = level_args(f, skip);
    const size_t smem = LV_HDR + (BS > 1 ? 2 : 1) * (size_t)lv_values<BS, T>(g.ncell) +
                        (size_t)g.nslots * g.group * lv_chunk<BS, T>(g.wc);
    // L and U are one kernel: the profiler counts it as the L sweep
    RsProfScope prof(ctx, BS == 1 ? RS_PROF_LSWEEP : RS_PROF_BLSWEEP);
    rs_pdl(k_level_solve<BS, T>, 1, std::max(W.one_threads, LV_IO_THREADS) + 32, smem, ctx)(
        g, (const unsigned char *)W.lrec, (const unsigned char *)W.urec, r, scale, z);
    return rs_check_launch(ctx);
}

// Estimated cycles of one sweep in one block and in the wavefront sweeps, from
// timings of both over 15 grids of 512 to 24,000 cells.  Where the line lies
// (both sweeps together, in us, one block / wavefronts): FP64 20^3 45 / 61,
// 24^3 72 / 69, 100 x 10 x 10 72 / 79, 160 x 10 x 8 109 / 98; FP32 16 x 12 x
// 10 16 / 33, 24^3 47 / 51, 160 x 10 x 8 74 / 51; 3 x 3 blocks in FP32 8^3
// 16 / 33, 16 x 12 x 10 31 / 45.  Larger grids do not fit in shared memory.
template <int BS, typename T>
bool level_fits(const std::vector<int> &w, int nx, int ny, int nz, int hops)
{
    if ((int)w.size() > LV_MAX_LEVELS || (int64_t)widest(w) * BS > LV_MAX_ROWS) return false;
    const int64_t ncell = (int64_t)(nx + 1) * (ny + 1) * (nz + 2);
    int group;
    if (!lv_slots<BS, T>(ncell, widest(w), &group)) return false;
    const bool dbl = sizeof(T) == 8;
    const double step = dbl ? 240 + 320.0 * BS : 375 + 15.0 * BS;       // a wavefront of up to 128 rows
    const double more = dbl ? 220 + 200.0 * BS : 180 + 20.0 * BS;       // each further 128 rows
    double one = 7000;
    for (int c : w) one += step + more * ((c * BS - 1) / 128);
    const double wave = w.size() * (dbl ? (BS == 1 ? 500.0 : 2500.0) : (BS == 1 ? 270.0 : 450.0)) + 4000.0 * hops + 9000;
    return one < 0.95 * wave;
}

#define RS_LEVEL_SWITCH(BSV, FP32, CALL)                                       \
    switch (BSV) {                                                             \
    case 1: return FP32 ? CALL(1, float) : CALL(1, double);                    \
    case 2: return FP32 ? CALL(2, float) : CALL(2, double);                    \
    case 3: return FP32 ? CALL(3, float) : CALL(3, double);                    \
    case 4: return FP32 ? CALL(4, float) : CALL(4, double);                    \
    }

}  // namespace

bool rs_level_fits(int bs, int fp32, int nx, int ny, int nz, int hops)
{
    const std::vector<int> w = level_sizes(nx, ny, nz);
#define FITS(B, T) level_fits<B, T>(w, nx, ny, nz, hops)
    RS_LEVEL_SWITCH(bs, fp32, FITS)
#undef FITS
    return false;
}

int rs_level_create(IluFactor *f)
{
    const std::vector<int> w = level_sizes(f->W.nx, f->W.ny, f->W.nz);
#define CREATE(B, T) level_create<B, T>(f, w)
    RS_LEVEL_SWITCH(f->bs, f->fp32, CREATE)
#undef CREATE
    return RS_ERR_INVALID_ARG;
}

int rs_level_gather(IluFactor *f)
{
#define GATHER(B, T) level_gather<B, T>(f)
    RS_LEVEL_SWITCH(f->bs, f->fp32, GATHER)
#undef GATHER
    return RS_ERR_INVALID_ARG;
}

int rs_level_apply(IluFactor *f, const double *r, double *z, const double *scale, const int *skip)
{
#define APPLY(B, T) level_apply<B, T>(f, r, z, scale, skip)
    RS_LEVEL_SWITCH(f->bs, f->fp32, APPLY)
#undef APPLY
    return RS_ERR_INVALID_ARG;
}
