// Triangular sweeps of independent parts, a block per part: the subdomains of
// restricted additive Schwarz (rs_ras.cu).
//
// The stacked matrix's subdomains do not read one another.  The segment
// sweeps hand every value from warp to warp through L2, 1.6 us (ILU(0)) to
// 3 us (ILU(1)) a segment level.  Where a subdomain's values fit in shared
// memory, one block now takes it through both sweeps in one launch, level by
// level of its row dependency graph: a level's rows do not read one another,
// a thread takes a row, and a level costs a barrier, the shared-memory
// gathers and the row's chain of multiply-adds.  The block reads the right-hand
// side through the subdomain's row list and writes only the rows it owns, so
// the gather and scatter passes of the apply go too.
//
// The rows' records come in chunks of at most PT_ROWS rows of a level (places;
// values by entry; columns by entry, 16-bit and local), streamed through a
// ring of shared-memory slots, two chunks a slot and copy, by a producer warp
// that joins the barrier once per slot (as in rs_level.cu).
// A row with fewer entries than its chunk's widest reads a zero at the end of
// the values.
//
// Arithmetic: L in ascending column order, U premultiplied by D_i = 1 / u_ii:
// z_i = D_i y_i - sum_j (D_i U_ij) z_j.
//
// What bounds it: a level's chain, 64 cycles per FP64 entry plus about 600
// cycles of gathers, barrier and instructions.  100 x 90 x 50 in 90 boxes,
// overlap 1, ILU(1) (107 levels of up to 120 rows and 6 entries a sweep):
// 243 us an apply with the segment sweeps, 159 here.
#include <string.h>

#include <algorithm>
#include <vector>

#include "rs_bounds.cuh"
#include "rs_internal.cuh"

namespace {

constexpr int PT_ROWS = 128;                        // rows of a chunk: the compute threads
constexpr int PT_REG = 8;                           // entries of a row read before the barrier
constexpr int PT_GROUP = 2;                         // chunks a slot
constexpr int PT_IO = 512;                          // threads that move the vectors in and out
constexpr int PT_MIN_SLOTS = 3, PT_MAX_SLOTS = 6;
constexpr int PT_MAX_GROUPS = 2048;                 // of both sweeps of a part (their table is in shared memory)
constexpr int PT_HDR = 128;                         // mbarriers; at PT_LOST the mark of a copy given up on
constexpr int PT_LOST = 64;
constexpr size_t PT_SMEM = 220 * 1024;
constexpr long long PT_DRAIN = 1LL << 30;           // cycles a late copy is still waited for
constexpr unsigned short PT_IDLE = 0xFFFF;

struct PartInfo {
    int row0, nrow;                                 // stacked rows
    int group0, nl, nu;                             // first group, groups of the L and of the U sweep
};
// offset and size of a group in 16 bytes; its chunks' rows (a multiple of 8)
// and entries of the widest, w | m << 16
struct PtGroup {
    int off, size, c0, c1;
};
struct PtChunk {
    int off, wm;                                    // offset in 16 bytes, w | m << 16
};

template <typename T, bool LOWER>
__host__ __device__ __forceinline__ int pt_bytes(int wm)
{
    const int w = wm & 0xFFFF, m = wm >> 16;
    return w * (2 + (LOWER ? 0 : (int)sizeof(T)) + m * ((int)sizeof(T) + 2));
}

struct PartArgs {
    const PartInfo *part;
    const PtGroup *group;
    const unsigned char *buf;
    const int *gidx, *own;
    int slot, nslots, vbytes, tbytes;               // ring; bytes of the values and of the group table
    int *err;
    long long limit;
    const int *skip;
};

// a thread's row of a chunk
template <typename T, bool LOWER>
struct PartRec {
    int e, m, w;
    T acc, v[PT_REG];                               // the right-hand side; entries
    unsigned short c[PT_REG];
    const unsigned char *vals;                      // of this thread's row
    const unsigned char *cols;
    __device__ __forceinline__ void load(const unsigned char *ch, int wm, int t, const T *y, int nrow, const volatile int *lost)
    {
        w = wm & 0xFFFF;
        m = wm >> 16;
        e = PT_IDLE;
        if (t < w) {
            e = ((const unsigned short *)ch)[t] | *lost;
            vals = ch + 2 * w + t * sizeof(T);
            cols = ch + 2 * w + (m + (LOWER ? 0 : 1)) * w * sizeof(T) + 2 * t;
            const unsigned char *pv = vals, *pc = cols;
#pragma unroll
            for (int k = 0; k < PT_REG; ++k)
                if (k < m) {
                    v[k] = *(const T *)pv;
                    c[k] = *(const unsigned short *)pc;
                    pv += w * sizeof(T);
                    pc += 2 * w;
                }
            // no other row writes y[e]: out of the step's chain
            acc = y[rs_part_place(e, nrow) ? e : nrow];
            if (!LOWER) acc = mad(*(const T *)(vals + m * w * sizeof(T)), acc, T(0));
        }
    }
    __device__ __forceinline__ void solve(T *y) const
    {
        T x[PT_REG], s = acc;
#pragma unroll
        for (int k = 0; k < PT_REG; ++k)
            if (k < m) x[k] = y[c[k]];
#pragma unroll
        for (int k = 0; k < PT_REG; ++k)
            if (k < m) s = msub(s, v[k], x[k]);
        for (int k = PT_REG; k < m; ++k)
            s = msub(s, *(const T *)(vals + k * w * sizeof(T)),
                     y[*(const unsigned short *)(cols + 2 * k * w)]);
        y[e] = s;
    }
};

template <typename T>
__global__ void __launch_bounds__(PT_IO + 32)
k_part_solve(PartArgs g, const double *__restrict__ r, double *__restrict__ z)
{
    extern __shared__ __align__(128) unsigned char pt_smem[];
    unsigned long long *full = (unsigned long long *)pt_smem;
    PtGroup *tab = (PtGroup *)(pt_smem + PT_HDR);
    T *y = (T *)(pt_smem + PT_HDR + g.tbytes);
    unsigned char *ring = pt_smem + PT_HDR + g.tbytes + g.vbytes;
    const int tid = threadIdx.x;
    volatile int *lost = (volatile int *)(pt_smem + PT_LOST);
    if (tid == 0) {
        *lost = 0;
        for (int s = 0; s < g.nslots; ++s) mbar_init(&full[s], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (rs_pdl_wait()) return;
    if (g.skip && *(volatile const int *)g.skip) return;
    const PartInfo P = g.part[blockIdx.x];
    const int groups = P.nl + P.nu;
    for (int k = tid; k < groups; k += blockDim.x) tab[k] = g.group[P.group0 + k];
    __syncthreads();
    if (tid >= PT_IO) {
        // producer: group j goes to slot j mod nslots
        const int lane = tid - PT_IO;
        int ij = 0, isl = 0, wsl = 0;
        unsigned wph = 0;
        bool dead = false;
        auto issue = [&]() {
            const PtGroup t = tab[ij++];
            mbar_arrive_expect_tx(&full[isl], 16u * t.size);
            bulk_g2s(ring + isl * g.slot, g.buf + 16 * (size_t)t.off, 16u * t.size, &full[isl]);
            if (++isl == g.nslots) isl = 0;
        };
        // bounded: a wait longer than the limit, however short the limit, is
        // recorded as a timeout; given up only much later
        auto arrived = [&]() {
            unsigned long long *b = &full[wsl];
            const unsigned par = wph;
            if (++wsl == g.nslots) {
                wsl = 0;
                wph ^= 1;
            }
            if (dead) return;
            const long long t0 = clock64(), giveup = 4 * g.limit + PT_DRAIN;
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
                    *lost = RS_PART_LOST;
                    break;
                }
            }
        };
        if (lane == 0) {
            for (int j = 0; j < min(g.nslots, groups); ++j) issue();
            arrived();
        }
        __syncthreads();
        // the barrier at the end of group j's first chunk: group j + 1 has
        // arrived (or is marked lost, and no record of it is used), and group
        // j - 1 has been read
        for (int j = 0; j < groups; ++j) {
            if (lane == 0 && j + 1 < groups) arrived();
            __syncwarp();
            asm volatile("bar.sync 1, %0;" ::"r"(PT_ROWS + 32) : "memory");
            if (lane == 0 && j > 0 && ij < groups && !dead) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                issue();
            }
        }
        return;
    }
    constexpr int U = 4;                             // rows whose loads are in flight together
    for (int l0 = tid; l0 < P.nrow; l0 += U * PT_IO) {
        int gi[U];
        double v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) gi[u] = __ldg(g.gidx + P.row0 + min(l0 + u * PT_IO, P.nrow - 1));
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = __ldg(r + gi[u]);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (l0 + u * PT_IO < P.nrow) y[l0 + u * PT_IO] = (T)v[u];
    }
    if (tid == 0) y[P.nrow] = T(0);
    __syncthreads();
    if (tid < PT_ROWS) {
        auto barrier = [&](bool first) {             // with the producer at a group's first chunk
            if (first) asm volatile("bar.sync 1, %0;" ::"r"(PT_ROWS + 32) : "memory");
            else asm volatile("bar.sync 2, %0;" ::"r"(PT_ROWS) : "memory");
        };
        const unsigned char *slot = ring, *end = ring + g.nslots * g.slot;
        auto advance = [&]() {
            slot += g.slot;
            if (slot == end) slot = ring;
        };
        static_assert(PT_GROUP == 2, "the chunks of a group are written out below");
        PartRec<T, true> ql;
        PartRec<T, false> qu;
        PtGroup t = tab[0], tn;                      // this group and the next one
        ql.load(slot, t.c0, tid, y, P.nrow, lost);
        for (int j = 0; j < P.nl; ++j) {
            tn = tab[min(j + 1, groups - 1)];
            if (rs_part_place(ql.e, P.nrow)) ql.solve(y);
            ql.load(slot + pt_bytes<T, true>(t.c0), t.c1, tid, y, P.nrow, lost);
            barrier(true);
            if (rs_part_place(ql.e, P.nrow)) ql.solve(y);
            advance();
            // U's first right-hand side may be a value of this step: after the barrier
            if (j + 1 < P.nl) ql.load(slot, tn.c0, tid, y, P.nrow, lost);
            t = tn;
            barrier(false);
        }
        qu.load(slot, t.c0, tid, y, P.nrow, lost);
        for (int j = 0; j < P.nu; ++j) {
            tn = tab[min(P.nl + j + 1, groups - 1)];
            if (rs_part_place(qu.e, P.nrow)) qu.solve(y);
            qu.load(slot + pt_bytes<T, false>(t.c0), t.c1, tid, y, P.nrow, lost);
            barrier(true);
            if (rs_part_place(qu.e, P.nrow)) qu.solve(y);
            advance();
            if (j + 1 < P.nu) qu.load(slot, tn.c0, tid, y, P.nrow, lost);
            t = tn;
            barrier(false);
        }
    }
    asm volatile("bar.sync 3, %0;" ::"r"(PT_IO) : "memory");
    for (int l0 = tid; l0 < P.nrow; l0 += U * PT_IO) {
        int gi[U], ow[U];
#pragma unroll
        for (int u = 0; u < U; ++u) gi[u] = __ldg(g.gidx + P.row0 + min(l0 + u * PT_IO, P.nrow - 1));
#pragma unroll
        for (int u = 0; u < U; ++u) ow[u] = __ldg(g.own + gi[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int l = l0 + u * PT_IO;
            if (l < P.nrow && ow[u] == P.row0 + l) z[gi[u]] = (double)y[l];
        }
    }
}

// Idle places of every chunk; a block per chunk.
__global__ void k_part_clear(const PtChunk *__restrict__ chunk, unsigned char *__restrict__ buf)
{
    const PtChunk c = chunk[blockIdx.x];
    unsigned short *p = (unsigned short *)(buf + 16 * (size_t)c.off);
    for (int k = threadIdx.x; k < (c.wm & 0xFFFF); k += blockDim.x) p[k] = PT_IDLE;
}

// The chunks from the FP64 factor in the stacked pattern: a thread per row and
// triangle; at: the row's chunk times PT_ROWS plus its place there.
template <typename T>
__global__ void k_part_gather(int n, const int *__restrict__ lat, const int *__restrict__ uat,
                              const int *__restrict__ prow, const PtChunk *__restrict__ chunk,
                              const int2 *__restrict__ prange, const int *__restrict__ ptr,
                              const int *__restrict__ col, const int *__restrict__ diagpos,
                              const double *__restrict__ lu, unsigned char *__restrict__ buf)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int2 pr = prange[prow[i]];                 // the part's first row and rows
    const int dp = diagpos[i];
    const double D = 1.0 / lu[dp];
    for (int tri = 0; tri < 2; ++tri) {
        const int a = tri ? uat[i] : lat[i], k0 = a % PT_ROWS;
        const PtChunk h = chunk[a / PT_ROWS];
        const int w = h.wm & 0xFFFF, m = h.wm >> 16;
        unsigned char *ch = buf + 16 * (size_t)h.off;
        ((unsigned short *)ch)[k0] = (unsigned short)(i - pr.x);
        T *v = (T *)(ch + 2 * w) + k0;
        unsigned short *c = (unsigned short *)(ch + 2 * w + (m + tri) * w * sizeof(T)) + k0;
        const int p0 = tri ? dp + 1 : ptr[i], p1 = tri ? ptr[i + 1] : dp;
        for (int k = 0; k < m; ++k) {
            const bool in = p0 + k < p1;
            v[k * w] = in ? (T)(tri ? __dmul_rn(D, lu[p0 + k]) : lu[p0 + k]) : T(0);
            c[k * w] = (unsigned short)(in ? col[p0 + k] - pr.x : pr.y);
        }
        if (tri) v[m * w] = (T)D;
    }
}

}  // namespace

struct PartSweep {
    rs_ctx *ctx;
    int fp32, nparts, n;
    PartInfo *part = nullptr;
    PtGroup *group = nullptr;
    unsigned char *buf = nullptr;
    int slot = 0, nslots = 0, vbytes = 0, tbytes = 0;
};

void rs_part_destroy(PartSweep *S)
{
    if (!S) return;
    rs_ctx *c = S->ctx;
    rs_free(c, S->part);
    rs_free(c, S->group);
    rs_free(c, S->buf);
    delete S;
}

// Chunks of one sweep of one part (stacked rows r0..r0 + ns): rows by level, at
// most PT_ROWS of one level a chunk, filled up to whole groups; end: the
// offset of the next chunk, in 16 bytes; dpos: the diagonals' entries.
struct PartPlan {
    std::vector<PartInfo> part;
    std::vector<PtGroup> group;
    std::vector<PtChunk> chunk;
    std::vector<int> lat, uat, prow, lev, order, start, fill;
    std::vector<int2> prange;
    int64_t end = 0;
    int slot = 1;                                    // largest group, in 16 bytes
};

template <typename T, bool LOWER>
static void part_chunks(PartPlan &S, int r0, int ns, const std::vector<int> &ptr, const std::vector<int> &col,
                        const std::vector<int> &dpos)
{
    std::vector<int> &at = LOWER ? S.lat : S.uat;
    S.lev.assign(ns, 0);
    int nlev = 0;
    for (int s = 0; s < ns; ++s) {
        const int l = LOWER ? s : ns - 1 - s, i = r0 + l;
        const int a = LOWER ? ptr[i] : dpos[i] + 1, b = LOWER ? dpos[i] : ptr[i + 1];
        int v = 0;
        for (int q = a; q < b; ++q) v = std::max(v, S.lev[col[q] - r0] + 1);
        S.lev[l] = v;
        nlev = std::max(nlev, v + 1);
    }
    S.start.assign(nlev + 1, 0);
    for (int l = 0; l < ns; ++l) ++S.start[S.lev[l] + 1];
    for (int h = 0; h < nlev; ++h) S.start[h + 1] += S.start[h];
    S.order.resize(ns);
    S.fill.assign(S.start.begin(), S.start.end() - 1);
    for (int l = 0; l < ns; ++l) S.order[S.fill[S.lev[l]]++] = l;
    int chunks = 0;
    auto add = [&](int k0, int k1) {
        int m = 0;
        for (int k = k0; k < k1; ++k) {
            const int i = r0 + S.order[k];
            m = std::max(m, LOWER ? dpos[i] - ptr[i] : ptr[i + 1] - 1 - dpos[i]);
            at[i] = (int)S.chunk.size() * PT_ROWS + k - k0;
        }
        const int wm = std::max(8, (k1 - k0 + 7) & ~7) | m << 16, size = pt_bytes<T, LOWER>(wm) / 16;
        S.chunk.push_back({(int)S.end, wm});
        if (chunks++ % PT_GROUP == 0) {
            S.group.push_back({(int)S.end, size, wm, 0});
        } else {
            S.group.back().size += size;
            S.group.back().c1 = wm;
        }
        S.slot = std::max(S.slot, S.group.back().size);
        S.end += size;
    };
    for (int h = 0; h < nlev; ++h)
        for (int k = S.start[h]; k < S.start[h + 1]; k += PT_ROWS) add(k, std::min(k + PT_ROWS, S.start[h + 1]));
    while (chunks % PT_GROUP) add(0, 0);
}

template <typename T>
static int part_create(rs_ctx *ctx, const std::vector<int> &sbase, const std::vector<int> &ptr,
                       const std::vector<int> &col, const IluFactor *f, int seg_levels, PartSweep **out)
{
    const int np = (int)sbase.size() - 1, n = sbase[np];
    int most = 0;
    for (int s = 0; s < np; ++s) most = std::max(most, sbase[s + 1] - sbase[s]);
    const int vbytes = ((most + 1) * (int)sizeof(T) + 15) & ~15;
    if (n < 1 || most >= PT_IDLE || (size_t)vbytes > PT_SMEM) return RS_OK;
    PartPlan S;
    std::vector<int> dpos(n);
    S.lat.resize(n);
    S.uat.resize(n);
    S.prow.resize(n);
    int groups = 0;
    for (int s = 0; s < np; ++s) {
        const int r0 = sbase[s], ns = sbase[s + 1] - r0;
        if (ns == 0) continue;
        for (int i = r0; i < r0 + ns; ++i) {
            int q = ptr[i];
            while (col[q] < i) ++q;
            if (ptr[i + 1] - ptr[i] > 0x7fff) return RS_OK;
            dpos[i] = q;
            S.prow[i] = (int)S.part.size();
        }
        PartInfo P = {r0, ns, (int)S.group.size(), 0, 0};
        part_chunks<T, true>(S, r0, ns, ptr, col, dpos);
        P.nl = (int)S.group.size() - P.group0;
        part_chunks<T, false>(S, r0, ns, ptr, col, dpos);
        P.nu = (int)S.group.size() - P.group0 - P.nl;
        groups = std::max(groups, P.nl + P.nu);
        S.part.push_back(P);
        S.prange.push_back(make_int2(r0, ns));
        if (S.end > 0x7fffffff || S.chunk.size() > 0x7fffffff / PT_ROWS) return RS_OK;
    }
    const int slot = 16 * S.slot, tbytes = groups * (int)sizeof(PtGroup);
    const size_t fixed = PT_HDR + (size_t)tbytes + vbytes;
    if (groups > PT_MAX_GROUPS || fixed + (size_t)PT_MIN_SLOTS * slot > PT_SMEM) return RS_OK;
    // a second block per SM when there are more parts than SMs
    int nslots = (int)std::min<size_t>((PT_SMEM - fixed) / slot, PT_MAX_SLOTS);
    const size_t half = PT_SMEM / 2 - 1024;
    if ((int)S.part.size() > ctx->num_sms && half >= fixed + (size_t)PT_MIN_SLOTS * slot)
        nslots = (int)std::min<size_t>((half - fixed) / slot, PT_MAX_SLOTS);
    // The rule: both times in us, fitted to 52 applies of 1,920 to 524,288 rows in 1 to
    // 450 boxes, ILU(0) to ILU(2) (within 10 % of nearly all).  Here a step costs
    // its FP64 or FP32 chain of m entries, and blocks on one SM take turns.  A segment
    // level costs the chain of a segment's rows or the hand-off between short
    // segments (`line` rows each).  One block / segments, us: 24 x 20 x 17 in 1 x 2 x 2 boxes,
    // ILU(1) 105 / 86 FP64, 47 / 52 FP32; in 2 x 2 x 2 87 / 92 and 39 / 59; 40 x 36 x 30 in
    // 6 x 6 x 6 103 / 75 and 48 / 50; 100 x 90 x 50 in 90 159 / 245 and 71 / 185, in 450
    // 271 / 254 and 119 / 196; one box of 24^3, ILU(0) 219 / 107 and 96 / 74.
    const bool dbl = sizeof(T) == 8;
    const int rounds = ((int)S.part.size() + ctx->num_sms - 1) / ctx->num_sms, steps = PT_GROUP * groups;
    int64_t ent = 0;
    for (const PtChunk &c : S.chunk) ent += c.wm >> 16;
    const double m = (double)ent / S.chunk.size(), line = 2.0 * n / (f->SL.nseg + f->SU.nseg);
    const double mine = rounds * (dbl ? 9.5 + 0.0046 * most + steps * (0.372 + 0.038 * m)
                                      : 8.1 + 0.0032 * most + steps * (0.064 + 0.027 * m));
    const double level = dbl ? std::max(0.2 + 0.21 * m, 1.5 - 0.02 * line) : std::max(0.3 + 0.085 * m, 0.95 - 0.01 * line);
    const double theirs = 8.0 + seg_levels * level + n * (dbl ? 0.21e-3 : 0.15e-3);
    if (mine > theirs) return RS_OK;
    PartSweep *R = new PartSweep();
    R->ctx = ctx;
    R->fp32 = !dbl;
    R->nparts = (int)S.part.size();
    R->n = n;
    R->slot = slot;
    R->nslots = nslots;
    R->vbytes = vbytes;
    R->tbytes = tbytes;
    int st = RS_OK;
    std::vector<void *> tmp;
    auto up = [&](auto **d, const auto &v, bool keep) {
        if (!st) st = rs_alloc(ctx, (void **)d, sizeof(v[0]) * v.size());
        if (!st && !keep) tmp.push_back(*d);
        if (!st && cudaMemcpyAsync(*d, v.data(), sizeof(v[0]) * v.size(), cudaMemcpyHostToDevice, ctx->stream) != cudaSuccess)
            st = RS_ERR_CUDA;
    };
    int *lat = nullptr, *uat = nullptr, *prow = nullptr;
    int2 *prange = nullptr;
    PtChunk *chunk = nullptr;
    up(&R->part, S.part, true);
    up(&R->group, S.group, true);
    up(&lat, S.lat, false);
    up(&uat, S.uat, false);
    up(&prow, S.prow, false);
    up(&prange, S.prange, false);
    up(&chunk, S.chunk, false);
    if (!st) st = rs_alloc(ctx, (void **)&R->buf, 16 * (size_t)S.end);
    if (!st) {
        k_part_clear<<<(int)S.chunk.size(), PT_ROWS, 0, ctx->stream>>>(chunk, R->buf);
        k_part_gather<T><<<(n + 127) / 128, 128, 0, ctx->stream>>>(n, lat, uat, prow, chunk, prange, f->ptr, f->col,
                                                                   f->diagpos, f->lu, R->buf);
        ctx->launches += 1;
        st = rs_check_launch(ctx);
    }
    if (!st && cudaStreamSynchronize(ctx->stream) != cudaSuccess) st = RS_ERR_CUDA;    // the host arrays end here
    for (void *p : tmp) rs_free(ctx, p);
    if (st) {
        rs_part_destroy(R);
        if (st == RS_ERR_OOM) {              // no room: the segment sweeps
            cudaGetLastError();
            st = RS_OK;
        }
        return st;
    }
    *out = R;
    return RS_OK;
}

int rs_part_create(rs_ctx *ctx, const std::vector<int> &sbase, const std::vector<int> &ptr, const std::vector<int> &col,
                   const IluFactor *f, int seg_levels, PartSweep **out)
{
    *out = nullptr;
    return f->fp32 ? part_create<float>(ctx, sbase, ptr, col, f, seg_levels, out)
                   : part_create<double>(ctx, sbase, ptr, col, f, seg_levels, out);
}

template <typename T>
static int part_apply(const PartSweep *S, const int *gidx, const int *own, const double *r, double *z, const int *skip)
{
    rs_ctx *ctx = S->ctx;
    static unsigned long long raised = 0;      // one bit per device
    const unsigned long long bit = 1ull << (ctx->device & 63);
    if (!(raised & bit)) {
        RS_CUDA_TRY(cudaFuncSetAttribute(k_part_solve<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PT_SMEM));
        raised |= bit;
    }
    PartArgs g;
    g.part = S->part;
    g.group = S->group;
    g.buf = S->buf;
    g.gidx = gidx;
    g.own = own;
    g.slot = S->slot;
    g.nslots = S->nslots;
    g.vbytes = S->vbytes;
    g.tbytes = S->tbytes;
    g.err = ctx->d_err;
    g.limit = ctx->spin_limit;
    g.skip = skip;
    // L, U, gather and scatter are one kernel: the profiler counts it as the L sweep
    RsProfScope prof(ctx, RS_PROF_LSWEEP);
    rs_pdl(k_part_solve<T>, S->nparts, PT_IO + 32, PT_HDR + S->tbytes + S->vbytes + (size_t)S->nslots * S->slot,
           ctx)(g, r, z);
    return rs_check_launch(ctx);
}

int rs_part_apply(const PartSweep *S, const int *gidx, const int *own, const double *r, double *z, const int *skip)
{
    return S->fp32 ? part_apply<float>(S, gidx, own, r, z, skip) : part_apply<double>(S, gidx, own, r, z, skip);
}
